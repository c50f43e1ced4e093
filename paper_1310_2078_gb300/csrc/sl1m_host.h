// sl1m_host.h -- host-side structures of libsl1m (internal).
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <future>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <thread>
#include <vector>

#include "sl1m.h"
#include "sl1m_dev.h"
#include "sl1m_grid.h"

// Device buffer owned by the library (cudaMalloc / cudaFree).
template <class T>
struct DBuf {
    T* p = nullptr;
    size_t n = 0;
    DBuf() = default;
    DBuf(const DBuf&) = delete;
    DBuf& operator=(const DBuf&) = delete;
    ~DBuf() { free(); }
    void free()
    {
        if (p) cudaFree(p);
        p = nullptr;
        n = 0;
    }
    cudaError_t alloc(size_t count)
    {
        free();
        if (count == 0) return cudaSuccess;
        cudaError_t e = cudaMalloc((void**)&p, count * sizeof(T));
        if (e != cudaSuccess) {
            p = nullptr;
            return e;
        }
        n = count;
        return cudaSuccess;
    }
    // Grow to at least `count` elements (contents are not preserved).  What
    // cannot grow stays as large as it was (beside the old memory first, then in
    // its place): others may count on it.
    cudaError_t reserve(size_t count, cudaStream_t st)
    {
        if (count <= n && p) return cudaSuccess;
        cudaStreamSynchronize(st);
        T* q = nullptr;
        cudaError_t e = cudaMalloc((void**)&q, count * sizeof(T));
        if (e == cudaSuccess) {
            free();
            p = q;
            n = count;
        } else if (const size_t had = n) {
            cudaGetLastError();
            e = alloc(count);
            if (e != cudaSuccess && alloc(had) != cudaSuccess) cudaGetLastError();   // (n = 0: nothing left)
        }
        return e;
    }
    // Allocate exactly `count` and copy from host (zero-fill when `zero`);
    // returns after the copy (the host source may be a temporary).
    cudaError_t upload(const T* src, size_t count, cudaStream_t st, bool zero = false)
    {
        cudaError_t e = alloc(count);
        if (e != cudaSuccess || count == 0) return e;
        if (zero) e = cudaMemsetAsync(p, 0, count * sizeof(T), st);
        else e = cudaMemcpyAsync(p, src, count * sizeof(T), cudaMemcpyHostToDevice, st);
        if (e != cudaSuccess) return e;
        return cudaStreamSynchronize(st);
    }
    size_t bytes() const { return n * sizeof(T); }
};

// Run fn(lo, hi) over [0, n) cut into contiguous chunks, one per host thread
// (at most 16), when n is large enough to pay for the threads.  For loops whose
// iterations write only their own outputs: the result is the one a single
// thread gives.
template <class F>
static inline void parallel_chunks(size_t n, size_t min_per_chunk, const F& fn)
{
    const size_t t = std::min<size_t>(16, std::max(1u, std::thread::hardware_concurrency()));
    const size_t nc = std::max<size_t>(1, std::min(t, n / std::max<size_t>(1, min_per_chunk)));
    if (nc <= 1) {
        fn((size_t)0, n);
        return;
    }
    std::vector<std::future<void>> fs;
    size_t done = 0;                       // chunks [0, done) run on threads
    try {
        for (size_t c = 1; c < nc; ++c) {
            fs.push_back(std::async(std::launch::async, [&fn, n, nc, c] { fn(n * c / nc, n * (c + 1) / nc); }));
            done = c;
        }
    } catch (...) {                        // no thread to be had: the rest runs here
    }
    fn(0, n / nc);
    for (size_t c = done + 1; c < nc; ++c) fn(n * c / nc, n * (c + 1) / nc);
    for (auto& f : fs) f.get();
}

struct HostPlan {
    std::vector<long long> u0;
    std::vector<int> b0, poff, clo, ncon;
    std::vector<long long> cta_u0;   // empty: uniform split
    long long U = 0;
    int C = 1, n_blocks = 0, n_slots = 0;
};

// Relative cost of the units of one problem in a plan: a constant per unit,
// or one value per `sub` units (block-major, streamed granule minor).
struct UnitCost {
    double uniform = 1.0;
    int sub = 1;
    std::vector<float> unit;
};

// costs == null: every unit costs the same; otherwise the CTA boundaries cut
// the summed cost into C equal parts.
void plan_host(const std::vector<int>& nb, const std::vector<int>& ns, int Cmax, HostPlan& H,
               const std::vector<const UnitCost*>* costs = nullptr);

// A plan whose tables and header live on the device (kernels take Plan*).
struct DevPlan {
    sl1m::Plan pl{};          // host copy of the header
    DBuf<long long> u0;
    DBuf<int> b0, poff, clo, ncon;
    DBuf<long long> cta;
    DBuf<sl1m::Plan> dpl;     // device header
};
cudaError_t build_plan(const std::vector<int>& nb, const std::vector<int>& ns, int Cmax, int own_gran, DevPlan& D,
                       cudaStream_t st, const std::vector<const UnitCost*>* costs = nullptr);

// Uploads a host plan's tables and header.
cudaError_t upload_plan(const HostPlan& H, int n_probs, int blk_el, DevPlan& D, cudaStream_t st);

// A problem's lattice operator: its tables, and the workspace it needs (the
// context's, shared by every problem of its stream).
struct GridTables {
    sl1m::GridOp op{};
    size_t ws_elems = 0;                 // float2 of workspace
    DBuf<int> cell, list, start, order, huge;
    DBuf<float> amp, wts;
    DBuf<float2> nu, wp, twx, twy, rot;
    DBuf<int4> pos;
    DBuf<unsigned char> act, colact;
    size_t bytes() const
    {
        return cell.bytes() + order.bytes() + list.bytes() + start.bytes() + amp.bytes() + wts.bytes() + nu.bytes() + wp.bytes() +
               twx.bytes() + twy.bytes() + rot.bytes() + pos.bytes() + act.bytes() + colact.bytes();
    }
};
constexpr size_t GR_WS_MAX = (size_t)4 << 30;      // bytes of workspace at most
// Operator classes of a batch: each problem's launches are of one of them.
constexpr int CLS_PAIRS = 0, CLS_GAINS = 1, CLS_GRID = 2, N_CLS = 3;

constexpr int NPROF = 7;

struct ProfRec {
    int kid;
    cudaEvent_t ev0, ev1;
    double pairs, bytes;
};

struct ProfTok {
    bool active = false;
    int kid = 0;
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
};

struct sl1m_problem;
struct Server;

// Device tables of a set of problems run together (one precision).
struct Batch {
    bool ready = false;                 // batch_set has succeeded
    int precision = 1;
    bool solver = false;
    std::vector<sl1m_problem*> probs;
    std::vector<sl1m::DevProblem> hdesc;
    DBuf<sl1m::DevProblem> desc;
    DBuf<int> n_probs_dev;
    DBuf<int> phases_dev;
    DevPlan plan[2][N_CLS];    // [0 forward / 1 adjoint][class]
    bool has_class[N_CLS] = {false, false, false};
    std::vector<int> cls;               // class of every problem
    std::vector<uint64_t> gens;         // layout of every problem when the plans were made
    std::vector<int> grid_slot[2];      // [op] first partial slot of every lattice problem
    size_t need_f[N_CLS] = {0, 0, 0}, need_a[N_CLS] = {0, 0, 0}, need_ws = 0;   // of the context's scratch
    int nst[2][2] = {{4, 4}, {4, 4}};   // tile shape per [op][class] (autotuned or default)
    int n_ant_max = 0;
    int sc_grid = 1;
    double pairs_class[N_CLS] = {0, 0, 0};
    double fin_bytes[2] = {0, 0};   // [forward finish, adjoint finish] per tick
    bool has_mfista = false;         // a tick ends with the MFISTA mix kernel
    // captured tick
    cudaGraphExec_t gexec = nullptr;
    bool graph_ok = false;
    long long tick_launches = 0;
    std::vector<const void*> cap_scratch;   // the context's scratch the capture baked in
    ~Batch();
};

// What the host reads back from the device, in pinned memory: copies into it are
// asynchronous, so a call waits for the stream once and not at each of them.
struct Mailbox {
    unsigned fault;                      // the bounded waits' flag
    sl1m::SolveState state;
    int phases[sl1m::MAX_PROBS];
    unsigned char result[256 * 1024];    // an operator call's result, when it fits
};

struct sl1m_ctx {
    int device = 0;
    cudaStream_t stream = nullptr;
    cudaStream_t upstream = nullptr;     // uploads of problems joining a running server
    bool own_stream = false;
    bool has_tables = false;             // counts among the users of the device's FP64 tables
    int num_sms = 1;
    std::string err;                     // last error message, guarded by err_mu: a running
    mutable std::mutex err_mu;           // server thread reports failures here too
    DBuf<double2> partial_f[N_CLS];      // partial sums per class: classes of a tick overlap
    DBuf<double> partial_a[N_CLS];
    cudaStream_t side[N_CLS - 1] = {};   // classes of a captured tick beside the stream's own
    cudaEvent_t ev_fork = nullptr, ev_join[N_CLS - 1] = {};
    // the scratch a captured tick bakes in
    std::vector<const void*> scratch() const
    {
        std::vector<const void*> v = {grid_ws.p};
        for (int c = 0; c < N_CLS; ++c) {
            v.push_back(partial_f[c].p);
            v.push_back(partial_a[c].p);
        }
        return v;
    }
    DBuf<float2> grid_ws;                // workspace of the lattice operators
    Mailbox* mail = nullptr;             // used by one call (or the server's loop) at a time
    std::vector<sl1m_problem*> problems;
    // autotuned (streamed granules per stage, CTAs per SM), keyed by
    // (precision, op, gains, Gaussian pixels, log2 of the units)
    std::map<long long, std::pair<int, int>> tune;
    Server* server = nullptr;            // running request loop
    Server* server_done = nullptr;       // stopped loop whose results are still collectable
    bool use_graphs = true;
    // profiling and counters
    bool prof = false;
    std::vector<ProfRec> pending;
    std::vector<cudaEvent_t> ev_pool;
    double prof_ms[NPROF] = {0}, prof_pairs[NPROF] = {0}, prof_bytes[NPROF] = {0};
    // pairs evaluated by the operator kernels of solver ticks, counted on the
    // device by the scalars kernel while profiling: [precision][0 fwd, 1 adj]
    DBuf<double> evals_dev;
    long long prof_n[NPROF] = {0};
    long long n_launch = 0, h2d = 0, d2h = 0;
    cudaEvent_t get_event();
    void drain_profile();
    ~sl1m_ctx();
};

void prof_begin(sl1m_ctx* ctx, int kid, ProfTok& tok);
void prof_end(sl1m_ctx* ctx, ProfTok& tok, double pairs, double bytes);
int sl1m_fail(sl1m_ctx* ctx, int code, const char* fmt, ...);

struct ProblemDev;

struct sl1m_problem {
    sl1m_ctx* ctx = nullptr;
    // caller data (host copies, caller order)
    int64_t n_vis = 0, n_pix = 0;
    int n_ant = 0;
    std::vector<double> uvw, vis, weights, lm, sigma, gains;
    std::vector<int> ant, kind;
    bool any_gauss = false;                    // a pixel of a Gaussian kind
    // device layout
    bool dirty = true;
    bool has_gauss = false;
    bool solver_ready = false;
    bool in_server = false;
    std::unique_ptr<ProblemDev> dev;
    sl1m::DevProblem hp{};          // layout part of the descriptor
    sl1m::SolveBufs hbufs{};
    std::vector<int> vis_orig, pix_orig;
    std::vector<double> last_img;             // image of the last refinement (caller's order)
    int algo = 0;                              // solver of the last init_solve (0 FISTA, 1 MFISTA)
    std::vector<float4> gext_vis, gext_pix;   // granule extents (host copies)
    std::vector<int> gkind_pix;               // pixel granule kinds
    std::vector<double> gsig_pix;             // and scales
    std::vector<int> gpairs_vis;              // gains: runs of equal antenna pairs per visibility granule
    std::vector<char> gown_vis;               // gains: whether its pairs have centres of their own
    UnitCost ucost[2][2];                      // [precision][0 forward / 1 adjoint]
    bool ucost_ok[2][2] = {{false, false}, {false, false}};
    std::unique_ptr<Batch> op_batch[2], solve_batch[2];
    std::unique_ptr<GridTables> grid;         // lattice operator of the mixed path, or null
    // what the lattice operator was last built or refused with: the budget, the
    // bytes it takes at least when memory was what it lacked, and whether it got
    // fewer planes at a time than it could use
    size_t grid_tried = 0, grid_least = 0;
    bool grid_cut = false;
    uint64_t gen = 0;                         // number of the layout: no two of a process share one
    const UnitCost& unit_cost(int precision, int op);

    // grid_budget: device bytes the lattice operator may take, tables, sums and
    // workspace (a laid-out problem that had less tries again)
    int rebuild(cudaStream_t st, size_t grid_budget = SIZE_MAX);
    void set_grid(cudaStream_t st, size_t grid_budget);    // 0: none
    size_t grid_own_bytes() const;                         // its tables and sums, without the workspace
    int ensure_r64(cudaStream_t st);
    int ensure_solver(cudaStream_t st);
    int init_solve(const sl1m_solve_opts* o, double L, bool power_only, cudaStream_t st);
    int read_state(sl1m::SolveState& s, cudaStream_t st);
    int fetch_image(double* host_out, cudaStream_t st);
    sl1m::DevProblem solver_desc() const;
    double pairs() const;
    size_t dev_bytes() const;
    size_t estimate_bytes(int precision) const;
    ~sl1m_problem();
};

// Builds P.grid when the laid-out problem's pixels are a lattice and the
// lattice operator is the faster one for it; false (P.grid null) otherwise.
bool grid_build(sl1m_problem& P, cudaStream_t st, size_t budget);

long long tune_key(int precision, int op, bool gains, bool gauss, long long units);

// batches (sl1m_host.cpp)
int batch_set(sl1m_ctx* ctx, Batch& B, const std::vector<sl1m_problem*>& probs,
              const std::vector<sl1m::DevProblem>& descs, int precision, bool solver);
int batch_op(sl1m_ctx* ctx, Batch& B, int op, double* user_out);
int batch_ticks(sl1m_ctx* ctx, Batch& B, int n);
int batch_phases(sl1m_ctx* ctx, Batch& B, std::vector<int>& out);

// server (sl1m_server.cpp)
void server_destroy(sl1m_ctx* ctx);
