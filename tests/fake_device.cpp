// fake_device.cpp -- a CUDA runtime and kernel launchers that run nothing, for
// CPU tests of libsl1m's host code (sl1m_host.cpp, sl1m_gridplan.cpp,
// sl1m_server.cpp, sl1m_refine.cpp).  Device memory is host memory; an
// allocation can be made to fail; every launcher checks, as the kernels would
// rely on it, that its plan belongs to the problems it is given and that what it
// reads and writes lies in live allocations, and notes what does not in
// fake_faults().  A captured graph keeps its launches' checks and runs them again
// at every launch.  Solves end after their first ticks (every phase reads DONE)
// unless they are held.
// A new problem takes the lowest free place of a few, so one made after another
// was destroyed has its address.
#include <cuda_runtime.h>
#include <dlfcn.h>

#include <atomic>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <functional>
#include <map>
#include <mutex>
#include <new>
#include <set>
#include <string>
#include <system_error>
#include <thread>
#include <vector>

#include "sl1m_host.h"
#include "sl1m_kernels.h"

using namespace sl1m;

namespace {

std::atomic<int> g_no_threads{0};                  // threads of the library's cannot be started
std::atomic<size_t> g_host_limit{SIZE_MAX};        // host allocations above this throw

std::recursive_mutex g_mu;
std::map<const char*, size_t> g_live;              // device allocations
size_t g_held = 0, g_total = (size_t)280 << 30, g_peak = 0;
size_t g_fail_min = 0;                             // allocations of this size and more ...
int g_fail_n = 0;                                  // ... fail this many times
std::string g_faults;
long long g_count[5];                              // launches: pairs fwd, adj, lattice fwd, adj; table fills
std::set<const void*> g_checked;                    // lattices whose lists were compared
bool g_hold = false;                                // solves run on
thread_local bool t_capturing = false;
using Check = std::function<void()>;
std::vector<Check> g_captured;

#define LOCK std::lock_guard<std::recursive_mutex> lk(g_mu)

void fault(const char* fmt, ...)
{
    char b[256];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(b, sizeof b, fmt, ap);
    va_end(ap);
    g_faults += std::string(b) + "\n";
}
bool need(const void* p, size_t bytes, const char* what)
{
    auto it = g_live.upper_bound((const char*)p);
    const bool ok = p && it != g_live.begin() && (--it, (const char*)p + bytes <= it->first + it->second);
    if (!ok) fault("%s: %zu bytes at %p are not in a live allocation", what, bytes, p);
    return ok;
}
void launch(Check c)
{
    LOCK;
    if (t_capturing) g_captured.push_back(c);
    c();
}

// The plan's share of problem p: `blocks` owned blocks by `units` streamed ones.
void check_plan(const char* what, const DevProblem* probs, const Plan* plp, bool mixed, bool gains, int op)
{
    if (!need(plp, sizeof *plp, what)) return;
    const Plan& pl = *plp;
    if (!need(probs, sizeof *probs * pl.n_probs, what) || !need(pl.prob_u0, 8 * (pl.n_probs + 1), what) ||
        !need(pl.prob_b0, 4 * (pl.n_probs + 1), what) || !need(pl.blk_poff, 4 * pl.n_blocks, what))
        return;
    for (int p = 0; p < pl.n_probs; ++p) {
        const DevProblem& P = probs[p];
        const long long units = pl.prob_u0[p + 1] - pl.prob_u0[p], blocks = pl.prob_b0[p + 1] - pl.prob_b0[p];
        if (units == 0) continue;
        const Side &own = op ? P.pix : P.vis, &str = op ? P.vis : P.pix;
        if (blocks != own_blocks(mixed, op, gains, own.n_gran) ||
            units != blocks * stream_units(mixed, str.n_gran) || (P.n_ant > 0) != gains)
            fault("%s: the plan is not that of problem %d", what, p);
    }
}
void check_grid(const char* what, const GridOp& g)
{
    const size_t rows = (size_t)g.np_pass * g.ny << g.lx, planes = (size_t)g.np_pass << (g.lx + g.ly);
    need(g.g1, 8 * rows, what);
    need(g.g2, 8 * planes, what);
    need(g.cell, (size_t)4 * g.nx * g.ny, what);
}

constexpr int N_PLACES = 8;
alignas(64) char g_place[N_PLACES][sizeof(sl1m_problem)];
bool g_used[N_PLACES];

// The lattice's lists, restated from its definition: positions as grid_setup_vis
// (below) made them, padding slots as in P.vis.orig.
void check_lists(const DevProblem& P, const GridOp& g)
{
    const int txn = (1 << g.lx) / GR_TILE, tyn = (1 << g.ly) / GR_TILE, tiles = txn * tyn, ni = g.np - GRW + 1;
    const int nv = P.vis.n_pad, mx = (1 << g.lx) - 1, my = (1 << g.ly) - 1;
    if (!need(g.pos, (size_t)nv * 16, "positions") || !need(P.vis.orig, (size_t)nv * 4, "slots")) return;
    std::vector<std::vector<int>> by((size_t)tiles * ni);
    std::vector<unsigned char> act((size_t)g.np * tiles, 0), colact((size_t)g.np * txn, 0);
    for (int k = 0; k < nv; ++k) {
        if (P.vis.orig[k] < 0) continue;
        bool seen[4] = {};
        const int4 q = g.pos[k];
        int at[4];
        for (int c = 0; c < 4; ++c) {
            const int x = (c & 1 ? (q.x + GRW - 1) & mx : q.x) / GR_TILE, y = (c & 2 ? (q.y + GRW - 1) & my : q.y) / GR_TILE;
            at[c] = y * txn + x;
            for (int d = 0; d < c; ++d) seen[c] |= at[d] == at[c];
            if (seen[c]) continue;
            by[(size_t)at[c] * ni + q.z].push_back(k);
            for (int z = q.z; z < q.z + GRW; ++z) act[((size_t)z * txn + x) * tyn + y] = colact[(size_t)z * txn + x] = 1;
        }
    }
    std::vector<int> start = {0}, list, order;
    for (int t = 0; t < tiles; ++t) {
        for (int z = 0; z < ni; ++z) {
            for (int k : by[(size_t)t * ni + z]) {
                list.push_back(k);
                if ((g.pos[k].y / GR_TILE) * txn + g.pos[k].x / GR_TILE == t) order.push_back(k);
            }
            start.push_back((int)list.size());
        }
        start.push_back((int)list.size());
    }
    for (int k = 0; k < nv; ++k)
        if (P.vis.orig[k] < 0) order.push_back(k);
    const auto same = [](const auto& v, const auto* p, const char* what) {
        if (!need(p, v.size() * sizeof v[0], what) || memcmp(p, v.data(), v.size() * sizeof v[0])) fault("lattice: %s differs", what);
    };
    same(start, g.start, "start");
    same(list, g.list, "list");
    same(order, g.order, "order");
    same(act, g.act, "act");
    same(colact, g.colact, "colact");
}

}  // namespace

// std::async and std::thread of the library come here (it is linked symbolically).
void std::thread::_M_start_thread(_State_ptr s, void (*dep)())
{
    if (g_no_threads) throw std::system_error(std::make_error_code(std::errc::resource_unavailable_try_again));
    using Start = void (*)(std::thread*, _State_ptr, void (*)());
    static const Start next = (Start)dlsym(RTLD_NEXT, "_ZNSt6thread15_M_start_threadESt10unique_ptrINS_6_StateESt14"
                                                      "default_deleteIS1_EEPFvvE");
    next(this, std::move(s), dep);
}

void* operator new(size_t n, const std::nothrow_t&) noexcept
{
    LOCK;
    for (int i = 0; n == sizeof(sl1m_problem) && i < N_PLACES; ++i)
        if (!g_used[i]) {
            g_used[i] = true;
            return g_place[i];
        }
    return malloc(n);
}
void* operator new(size_t n)
{
    void* p = n > g_host_limit ? nullptr : malloc(n);
    if (p) return p;
    throw std::bad_alloc();
}
void operator delete(void* p) noexcept
{
    const size_t at = (char*)p - g_place[0];
    if (p && at < sizeof g_place) {
        LOCK;
        g_used[at / sizeof(sl1m_problem)] = false;
    } else {
        free(p);
    }
}
void operator delete(void* p, size_t) noexcept { operator delete(p); }

extern "C" {

const char* fake_faults() { return g_faults.c_str(); }
void fake_reset()
{
    LOCK;
    g_faults.clear();
    g_fail_n = 0;
    g_hold = false;
    g_checked.clear();
    g_total = (size_t)280 << 30;
    g_peak = g_held;
    memset(g_count, 0, sizeof g_count);
}
void fake_fail(size_t min_bytes, int n) { LOCK; g_fail_min = min_bytes; g_fail_n = n; }
void fake_no_threads(int on) { g_no_threads = on; }
void fake_host_limit(size_t n) { g_host_limit = n; }
void fake_hold(int on) { LOCK; g_hold = on; }
void fake_total(size_t bytes) { LOCK; g_total = bytes; }
size_t fake_held() { return g_held; }
size_t fake_peak() { return g_peak; }
long long fake_count(int what) { return g_count[what]; }

// (kernels' files, not linked here)
int sl1m_forward_noalloc(sl1m_problem*, const double*, double*, int) { return SL1M_ERR_CUDA; }
int sl1m_measure_sfu(sl1m_ctx*, double*, double*) { return SL1M_ERR_CUDA; }

cudaError_t cudaMalloc(void** p, size_t n)
{
    LOCK;
    *p = nullptr;
    if ((g_fail_n > 0 && n >= g_fail_min && g_fail_n--) || g_held + n > g_total) return cudaErrorMemoryAllocation;
    *p = malloc(n);
    g_live[(const char*)*p] = n;
    g_held += n;
    g_peak = std::max(g_peak, g_held);
    return cudaSuccess;
}
cudaError_t cudaFree(void* p)
{
    LOCK;
    if (!p) return cudaSuccess;
    const auto it = g_live.find((const char*)p);
    if (it == g_live.end()) return fault("cudaFree: not an allocation"), cudaErrorInvalidValue;
    g_held -= it->second;
    g_live.erase(it);
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) { LOCK; *f = g_total - g_held; *t = g_total; return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t)
{
    LOCK;
    if (k != cudaMemcpyDeviceToHost && !need(d, n, "copy to the device")) return cudaErrorInvalidValue;
    if (k != cudaMemcpyHostToDevice && !need(s, n, "copy from the device")) return cudaErrorInvalidValue;
    memmove(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t)
{
    LOCK;
    if (!need(d, n, "memset")) return cudaErrorInvalidValue;
    memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int)
{
    memset(p, 0, sizeof *p);
    p->multiProcessorCount = 152;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)malloc(1); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { free(s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)malloc(1); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { free(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode)
{
    LOCK;
    t_capturing = true;
    g_captured.clear();
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g)
{
    LOCK;
    t_capturing = false;
    *g = (cudaGraph_t) new std::vector<Check>(g_captured);
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t g, unsigned long long)
{
    *x = (cudaGraphExec_t) new std::vector<Check>(*(std::vector<Check>*)g);
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t)
{
    LOCK;
    for (auto& c : *(std::vector<Check>*)x) c();
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { delete (std::vector<Check>*)g; return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { delete (std::vector<Check>*)x; return cudaSuccess; }

}  // extern "C"

namespace sl1m {

cudaError_t launch_forward(int precision, bool gains, int, const DevProblem* probs, const Plan* plp, int,
                           double2* partial, cudaStream_t, int)
{
    launch([=] {
        check_plan("forward", probs, plp, precision != 0, gains, 0);
        need(partial, (size_t)plp->n_slots * plp->blk_el * 16, "forward's partial sums");
        ++g_count[0];
    });
    return cudaSuccess;
}
cudaError_t launch_adjoint(int precision, bool gains, int, const DevProblem* probs, const Plan* plp, int,
                           double* partial, cudaStream_t, int)
{
    launch([=] {
        check_plan("adjoint", probs, plp, precision != 0, gains, 1);
        need(partial, (size_t)plp->n_slots * plp->blk_el * 8, "adjoint's partial sums");
        ++g_count[1];
    });
    return cudaSuccess;
}
cudaError_t grid_forward(const DevProblem* probs, int p, const GridOp& g, int n_vis_pad, double2* partial, cudaStream_t,
                         long long* n)
{
    launch([=] {
        check_grid("lattice forward", g);
        need(partial, (size_t)n_vis_pad * 16, "lattice forward's sums");
        if (need(probs, sizeof *probs * (p + 1), "lattice forward") &&
            (probs[p].vis.n_pad != n_vis_pad || !need(g.order, (size_t)n_vis_pad * 4, "lattice forward's order")))
            fault("lattice forward: another problem's tables");
        if (g_checked.insert(g.start).second) check_lists(probs[p], g);
        ++g_count[2];
    });
    *n += 3;
    return cudaSuccess;
}
cudaError_t grid_adjoint(const DevProblem* probs, int p, const GridOp& g, int n_pix, int n_pix_pad, double* partial,
                         cudaStream_t, long long* n)
{
    launch([=] {
        check_grid("lattice adjoint", g);
        need(partial, (size_t)n_pix_pad * 8 * g.n_chunk, "lattice adjoint's sums");
        if (g.n_chunk * GR_PCH > g.np_pass) fault("lattice adjoint: sums of more planes than a pass has");
        if (need(probs, sizeof *probs * (p + 1), "lattice adjoint") && probs[p].pix.n != n_pix)
            fault("lattice adjoint: another problem's tables");
        ++g_count[3];
    });
    *n += 3;
    return cudaSuccess;
}
cudaError_t grid_prepare_kernels(int, int) { return cudaSuccess; }
cudaError_t grid_setup_cells(const d4*, GridOp, const double*, const double*, double, double, float*, float2*, cudaStream_t)
{
    return cudaSuccess;
}
cudaError_t grid_setup_vis(const d4*, int n, GridOp g, double, double, double, double, double, double, double, int4* pos,
                           float*, float2*, cudaStream_t)
{
    unsigned r = 12345;                                // (any positions; half of them in a few tiles)
    const auto next = [&](int m) { return (int)((r = r * 1664525u + 1013904223u) >> 8) % m; };
    for (int k = 0; need(pos, (size_t)n * 16, "positions") && k < n; ++k)
        pos[k] = k % 2 ? make_int4(next(1 << g.lx), next(1 << g.ly), next(g.np - GRW + 1), 0)
                       : make_int4(next(40), (1 << g.ly) - 1 - next(9), next(g.np - GRW + 1) / 3, 1);
    return cudaSuccess;
}
cudaError_t fp64_init_tables(cudaStream_t) { LOCK; ++g_count[4]; return cudaSuccess; }
cudaError_t launch_fwd_finish(const DevProblem* probs, const Plan* plp, const Plan&, int, const double2* partial, int,
                              double2*, cudaStream_t)
{
    launch([=] {
        if (need(plp, sizeof *plp, "forward finish") && need(probs, sizeof *probs * plp->n_probs, "forward finish"))
            need(partial, (size_t)plp->n_slots * plp->blk_el * 16, "forward finish's partial sums");
    });
    return cudaSuccess;
}
cudaError_t launch_adj_finish(const DevProblem* probs, const Plan* plp, const Plan&, int, const double* partial, double*,
                              cudaStream_t)
{
    launch([=] {
        if (need(plp, sizeof *plp, "adjoint finish") && need(probs, sizeof *probs * plp->n_probs, "adjoint finish"))
            need(partial, (size_t)plp->n_slots * plp->blk_el * 8, "adjoint finish's partial sums");
    });
    return cudaSuccess;
}
cudaError_t launch_phases(const DevProblem* probs, const int* n, int, int* out, cudaStream_t)
{
    launch([=] {
        for (int i = 0; need(n, 4, "phases") && i < *n; ++i)
            if (need(probs[i].st, sizeof(SolveState), "phases")) out[i] = probs[i].st->phase = g_hold ? PH_SOLVE : PH_DONE;
    });
    return cudaSuccess;
}
cudaError_t wait_fault_read(unsigned* f, cudaStream_t) { *f = 0; return cudaSuccess; }
cudaError_t wait_fault_clear(cudaStream_t) { return cudaSuccess; }
cudaError_t launch_wait_selftest(unsigned long long*, int, cudaStream_t) { return cudaSuccess; }
unsigned long long wait_limit_ns() { return 1; }
int occupancy(int, bool, int, int) { return 4; }
cudaError_t launch_gather_real(const double*, double*, const int*, int, double, int*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_gather_resid(const double2*, const DevProblem*, int, int, double2*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_scatter_real(const double*, double*, const int*, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_scatter_cplx(const double2*, double2*, const int*, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_fill_valid(double*, const int*, int, double, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_weighted_vis(const DevProblem*, int, int, double2*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_gauss_class(const d4*, int, const double*, int, float4*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_mfista_mix(const DevProblem*, const Plan*, const Plan*, int, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_scalars(const DevProblem*, const int*, int, double*, cudaStream_t) { return cudaSuccess; }

}  // namespace sl1m
