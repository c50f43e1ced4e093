// sl1m_gridplan.cpp -- host side of the lattice operator (sl1m_grid.cu): is the
// pixel set a regular lattice, is the lattice operator the cheaper one for this
// problem, and its tables.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

#include "sl1m_host.h"

using namespace sl1m;

namespace {

// Gauss-Legendre nodes and weights of order 2 n on [0, 1]'s half of [-1, 1]
// (the rule is symmetric): Newton's iteration on the Legendre recurrence.
void gauss_legendre_half(int n, double* x, double* w)
{
    const int m = 2 * n;
    for (int i = 0; i < n; ++i) {
        double t = std::cos(M_PI * (i + 0.75) / (m + 0.5)), dp = 1.0;
        for (int it = 0; it < 60; ++it) {
            double p0 = 1.0, p1 = t;
            for (int k = 2; k <= m; ++k) {
                const double p2 = ((2 * k - 1) * t * p1 - (k - 1) * p0) / k;
                p0 = p1;
                p1 = p2;
            }
            dp = m * (t * p1 - p0) / (t * t - 1.0);
            const double d = p1 / dp;
            t -= d;
            if (std::fabs(d) < 1e-15) break;
        }
        x[i] = t;
        w[i] = 2.0 / ((1.0 - t * t) * dp * dp);
    }
}

// One axis of the pixels: the offset and spacing of a lattice they all lie on.
struct Axis {
    bool ok = false;
    double x0 = 0.0, step = 1.0;     // coordinate = x0 + k step
    int kmin = 0, n = 1;
};

// The spacing is the smallest distance from the first pixel, refined over the
// whole span; every pixel then has to sit on its lattice point to within
// `tol` (a phase error of 1e-8 turn at the longest baseline).  A lattice whose
// first pixel has no neighbour one step away is not recognised.
Axis find_axis(const double* c, int64_t n, double tol)
{
    Axis A;
    A.x0 = c[0];
    const size_t nt = 64;                               // chunks of the reductions
    std::vector<double> near(nt, 1e300), lo(nt, 1e300), hi(nt, -1e300);
    const auto chunk = [&](size_t t) { return std::make_pair((size_t)n * t / nt, (size_t)n * (t + 1) / nt); };
    parallel_chunks(nt, (size_t)std::max<int64_t>(1, 65536 / std::max<int64_t>(1, n / (int64_t)nt)),
                    [&](size_t t0, size_t t1) {
        for (size_t t = t0; t < t1; ++t) {
            const auto r = chunk(t);
            for (size_t i = r.first; i < r.second; ++i) {
                const double v = c[2 * i], d = std::fabs(v - A.x0);
                if (d > tol) near[t] = std::min(near[t], d);
                lo[t] = std::min(lo[t], v);
                hi[t] = std::max(hi[t], v);
            }
        }
    });
    const double dmin = *std::min_element(near.begin(), near.end());
    const double xl = *std::min_element(lo.begin(), lo.end()), xh = *std::max_element(hi.begin(), hi.end());
    if (dmin > 1e299) {                                 // one value
        A.ok = true;
        return A;
    }
    const double span = xh - A.x0 > A.x0 - xl ? xh - A.x0 : A.x0 - xl;
    const double steps = std::rint(span / dmin);
    if (!(steps >= 1.0) || steps > 8192.0) return A;
    A.step = span / steps;
    A.kmin = (int)std::rint((xl - A.x0) / A.step);
    A.n = (int)std::rint((xh - A.x0) / A.step) - A.kmin + 1;
    std::vector<char> bad(nt, 0);
    parallel_chunks(nt, (size_t)std::max<int64_t>(1, 65536 / std::max<int64_t>(1, n / (int64_t)nt)),
                    [&](size_t t0, size_t t1) {
        for (size_t t = t0; t < t1; ++t) {
            const auto r = chunk(t);
            for (size_t i = r.first; i < r.second; ++i) {
                const double d = c[2 * i] - A.x0;
                if (std::fabs(d - std::rint(d / A.step) * A.step) > tol) bad[t] = 1;
            }
        }
    });
    A.ok = std::count(bad.begin(), bad.end(), 1) == 0;
    return A;
}

int log2_at_least(int n)
{
    int l = GR_LOG_MIN;
    while ((1 << l) < n) ++l;
    return l;
}

std::vector<float2> twiddles(int lg)
{
    std::vector<float2> t;
    t.reserve(grid_tw_elems(lg));
    const int radix = grid_radix(lg);
    for (int ns = grid_radix0(lg); ns < (1 << lg); ns *= radix)
        for (int m = 1; m < radix; m *= 2)
            for (int k = 0; k < ns; ++k) {
                const double a = 2.0 * M_PI * m * k / ((double)radix * ns);
                t.push_back(make_float2((float)std::cos(a), (float)-std::sin(a)));
            }
    return t;
}

}  // namespace

// Seconds of a pass (forward and adjoint averaged) by either operator, fitted to
// both on GB300 over 64^2 .. 1024^2 pixels x 1,500 .. 100,000 visibilities, fields
// of +/-0.02 .. +/-0.5 (us, forward / adjoint; pairs and then lattice):
//   64^2 x 4,000      41 / 38       43 / 87       256^2 +/-0.5 x 5,000   275 / 266    191 / 292
//   64^2 x 40,000    110 / 87       66 / 230      500^2 x 3,000          427 / 293     75 / 94
//   128^2 x 5,000     88 / 68       45 / 54       1024^2 +/-0.3 x 3,000 1609 / 1110   439 / 584
//   200^2 x 60,000  1185 / 853      98 / 120      1024^2 +/-0.3 x 1,000  629 / 415    291 / 395
// (64^2 and 256^2 +/-0.5: the rule takes the pairs; lattice measured with a slower
// spreading kernel.)
// Lattice: launches, the planes' cells, the visibilities, and the points that a
// tile's CTA spreads one after the other where there are few tiles.  The lattice
// is taken where it promises a tenth or more.
static double grid_seconds(const GridOp& g, double n_vis)
{
    return 4.2e-5 + 2.8e-12 * (double)g.np * grid_plane_elems(g) + 1.05e-9 * n_vis + 2.7e-7 * n_vis / grid_tiles(g);
}
static double pair_seconds(double pairs) { return 2.8e-5 + pairs / 2.4e12; }

bool grid_build(sl1m_problem& P, cudaStream_t st, size_t budget)
{
    P.grid.reset();
    P.grid_least = 0;
    P.grid_cut = false;
    if (P.n_ant > 0 || P.has_gauss) return false;
    const double pairs = P.pairs();
    if (0.9 * pair_seconds(pairs) < 4.2e-5) return false;   // launches, not pairs, decide
    // extents of the visibilities and of n - 1
    double um = 0, vm = 0, w0 = 1e300, w1 = -1e300, n0 = 1e300, n1 = -1e300;
    for (int64_t k = 0; k < P.n_vis; ++k) {
        um = std::max(um, std::fabs(P.uvw[3 * k]));
        vm = std::max(vm, std::fabs(P.uvw[3 * k + 1]));
        const double w = std::fabs(P.uvw[3 * k + 2]);      // w < 0: taken at the mirrored point
        w0 = std::min(w0, w);
        w1 = std::max(w1, w);
    }
    const Axis ax = find_axis(P.lm.data(), P.n_pix, 1e-8 / std::max(1.0, um));
    if (!ax.ok) return false;
    const Axis ay = find_axis(P.lm.data() + 1, P.n_pix, 1e-8 / std::max(1.0, vm));
    if (!ay.ok) return false;
    for (int64_t j = 0; j < P.n_pix; ++j) {
        const double l = P.lm[2 * j], m = P.lm[2 * j + 1], r2 = l * l + m * m;
        const double v = -r2 / (1.0 + std::sqrt(1.0 - r2));
        n0 = std::min(n0, v);
        n1 = std::max(n1, v);
    }
    auto T = std::make_unique<GridTables>();
    GridOp& g = T->op;
    g.nx = ax.n;
    g.ny = ay.n;
    g.lx = log2_at_least(2 * g.nx);
    g.ly = log2_at_least(2 * g.ny);
    if (g.lx > GR_LOG_MAX || g.ly > GR_LOG_MAX) return false;
    const double nc = 0.5 * (n0 + n1), B = std::max(0.5 * (n1 - n0), 1e-15);
    const double dw = 0.25 / B, span = (w1 - w0) / dw;
    if (!(span < 1e5)) return false;
    g.np = (int)std::ceil(span) + GRW;
    if (grid_seconds(g, (double)P.n_vis) > 0.9 * pair_seconds(pairs)) return false;
    g.cx = g.nx / 2;
    g.cy = g.ny / 2;
    // the workspace holds as many planes as fit GR_WS_MAX bytes and a quarter
    // of what is free
    size_t free_b = 0, total_b = 0;
    if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) return false;
    const size_t plane = grid_plane_elems(g) * sizeof(float2);
    const size_t ws_max = std::min({GR_WS_MAX, free_b / 4, budget / 2});
    const size_t nv = P.hp.vis.n_pad, cells = (size_t)g.nx * g.ny;
    const int tiles = grid_tiles(g), ni = g.np - GRW + 1;
    const size_t tab = cells * 16 + nv * (16 + 12 * GRW + 8 + 20) + (size_t)tiles * (ni * 5 + 44);
    const size_t want = (size_t)(g.np + GR_PCH - 1) / GR_PCH, got = ws_max / (plane * GR_PCH);
    g.np_pass = (int)std::min(want, got) * GR_PCH;
    g.n_chunk = 1;                                        // (with the fewest planes)
    P.grid_least = std::max(2 * plane * GR_PCH, tab + grid_sum_bytes(g, P.hp.vis.n_blk, P.hp.pix.n_blk) + plane * GR_PCH);
    if (g.np_pass < GR_PCH) return false;
    P.grid_cut = got < std::min(want, GR_WS_MAX / (plane * GR_PCH));
    g.n_chunk = g.np_pass / GR_PCH;
    T->ws_elems = grid_plane_elems(g) * g.np_pass;
    const size_t sums = grid_sum_bytes(g, P.hp.vis.n_blk, P.hp.pix.n_blk);
    if (tab + sums + T->ws_elems * sizeof(float2) > std::min(budget, free_b / 2)) return false;
    // powers of two that keep a coherent sum of the largest inputs in range
    const auto p2 = [](double n) { return (float)std::exp2(-std::ceil(std::log2(std::max(1.0, n)))); };
    g.fscale = p2((double)P.n_pix);
    g.ascale = p2((double)P.n_vis);
    // the cell of every pixel, by its sorted slot (each cell once)
    std::vector<int> cell(cells, -1);
    for (int t = 0; t < (int)P.pix_orig.size(); ++t) {
        const int o = P.pix_orig[t];
        if (o < 0) continue;
        const int ix = (int)std::rint((P.lm[2 * (size_t)o] - ax.x0) / ax.step) - ax.kmin;
        const int iy = (int)std::rint((P.lm[2 * (size_t)o + 1] - ay.x0) / ay.step) - ay.kmin;
        int& c = cell[(size_t)iy * g.nx + ix];
        if (c >= 0) return false;                        // two pixels at one place
        c = t;
    }
    // transforms of the kernel: its Fourier integral by Gauss-Legendre
    std::vector<double> quad(2 * GR_NQ), cxy((size_t)g.nx + g.ny);
    gauss_legendre_half(GR_NQ, quad.data(), quad.data() + GR_NQ);
    for (int q = 0; q < GR_NQ; ++q) {
        const double t = quad[q];
        quad[GR_NQ + q] *= 0.5 * GRW * std::exp(GR_BETA * (std::sqrt(1.0 - t * t) - 1.0));
        quad[q] = 0.5 * GRW * t;
    }
    const auto inv_hat = [&](double xi) {
        double s = 0.0;
        for (int q = 0; q < GR_NQ; ++q) s += quad[GR_NQ + q] * std::cos(2.0 * M_PI * xi * quad[q]);
        return 0.5 / s;
    };
    for (int i = 0; i < g.nx; ++i) cxy[i] = inv_hat((double)(i - g.cx) / (1 << g.lx));
    for (int i = 0; i < g.ny; ++i) cxy[g.nx + i] = inv_hat((double)(i - g.cy) / (1 << g.ly));
    const double wp0 = w0 - (0.5 * GRW - 0.5) * dw;
    std::vector<float2> wp(g.np);
    for (int p = 0; p < g.np; ++p) {
        const double w = wp0 + p * dw;
        wp[p] = make_float2((float)w, (float)(w - (double)(float)w));
    }
    const std::vector<float2> tx = twiddles(g.lx), ty = twiddles(g.ly);
    // any failure below (memory, above all) leaves the pair operator in place
    bool ok = T->cell.upload(cell.data(), cells, st) == cudaSuccess && T->wp.upload(wp.data(), wp.size(), st) == cudaSuccess &&
              T->twx.upload(tx.data(), tx.size(), st) == cudaSuccess && T->twy.upload(ty.data(), ty.size(), st) == cudaSuccess &&
              T->amp.alloc(cells) == cudaSuccess && T->nu.alloc(cells) == cudaSuccess && T->pos.alloc(nv) == cudaSuccess &&
              T->wts.alloc(nv * 3 * GRW) == cudaSuccess && T->rot.alloc(nv) == cudaSuccess;
    DBuf<double> dq, dc;
    ok = ok && dq.upload(quad.data(), quad.size(), st) == cudaSuccess && dc.upload(cxy.data(), cxy.size(), st) == cudaSuccess;
    std::vector<int4> pos(nv);
    if (ok) {
        g.cell = T->cell.p;
        g.wp = T->wp.p;
        g.twx = T->twx.p;
        g.twy = T->twy.p;
        ok = grid_setup_cells(P.hp.pix.d, g, dc.p, dq.p, nc, dw, T->amp.p, T->nu.p, st) == cudaSuccess &&
             grid_setup_vis(P.hp.vis.d, (int)nv, g, ax.step, ay.step, ax.x0 + (ax.kmin + g.cx) * ax.step,
                            ay.x0 + (ay.kmin + g.cy) * ay.step, nc, wp0, dw, T->pos.p, T->wts.p, T->rot.p,
                            st) == cudaSuccess &&
             cudaMemcpyAsync(pos.data(), T->pos.p, nv * sizeof(int4), cudaMemcpyDeviceToHost, st) == cudaSuccess &&
             cudaStreamSynchronize(st) == cudaSuccess;
    }
    // visibilities per tile (at most two tiles per axis), by first plane, in the
    // library's order: a counting sort
    std::vector<int> start, list, order;
    if (ok) {
        const int txn = (1 << g.lx) / GR_TILE, mx = (1 << g.lx) - 1, my = (1 << g.ly) - 1;
        start.assign((size_t)tiles * (ni + 1) + 1, 0);
        const auto each = [&](const auto& f) {
            for (size_t k = 0; k < nv; ++k) {
                if (P.vis_orig[k] < 0) continue;
                const int xa = pos[k].x / GR_TILE, xb = ((pos[k].x + GRW - 1) & mx) / GR_TILE;
                const int ya = pos[k].y / GR_TILE, yb = ((pos[k].y + GRW - 1) & my) / GR_TILE;
                for (int y = 0; y < (ya == yb ? 1 : 2); ++y)
                    for (int x = 0; x < (xa == xb ? 1 : 2); ++x)
                        f(k, ((size_t)(y ? yb : ya) * txn + (x ? xb : xa)) * (ni + 1) + pos[k].z);
            }
        };
        each([&](size_t, size_t at) { ++start[at + 1]; });
        for (size_t i = 1; i < start.size(); ++i) start[i] += start[i - 1];
        list.resize(std::max(1, start.back()));
        std::vector<int> fill(start.begin(), start.end() - 1);
        each([&](size_t k, size_t at) { list[fill[at]++] = (int)k; });
        // each visibility once, at its first tile; then the padding slots
        order.reserve(nv);
        for (int t = 0; t < tiles; ++t)
            for (int i = start[(size_t)t * (ni + 1)]; i < start[(size_t)(t + 1) * (ni + 1)]; ++i) {
                const int4 q = pos[list[i]];
                if ((q.y / GR_TILE) * txn + q.x / GR_TILE == t) order.push_back(list[i]);
            }
        for (size_t k = 0; k < nv; ++k)
            if (P.vis_orig[k] < 0) order.push_back((int)k);
        // which tiles of each plane have a visibility
        const int tyn = (1 << g.ly) / GR_TILE;
        std::vector<unsigned char> act((size_t)g.np * tiles, 0), colact((size_t)g.np * txn, 0);
        for (int t = 0; t < tiles; ++t)
            for (int i = 0, done = 0; i < ni; ++i) {     // planes below `done` are marked
                const size_t at = (size_t)t * (ni + 1) + i;
                if (start[at] == start[at + 1]) continue;
                for (int p = std::max(i, done); p < i + GRW; ++p) {
                    act[((size_t)p * txn + t % txn) * tyn + t / txn] = 1;
                    colact[(size_t)p * txn + t % txn] = 1;
                }
                done = i + GRW;
            }
        ok = T->start.upload(start.data(), start.size(), st) == cudaSuccess &&
             T->list.upload(list.data(), list.size(), st) == cudaSuccess &&
             T->order.upload(order.data(), order.size(), st) == cudaSuccess &&
             T->act.upload(act.data(), act.size(), st) == cudaSuccess &&
             T->colact.upload(colact.data(), colact.size(), st) == cudaSuccess;
    }
    if (!ok) {
        cudaGetLastError();
        return false;
    }
    g.amp = T->amp.p;
    g.nu = T->nu.p;
    g.pos = T->pos.p;
    g.wts = T->wts.p;
    g.rot = T->rot.p;
    g.order = T->order.p;
    g.list = T->list.p;
    g.start = T->start.p;
    g.act = T->act.p;
    g.colact = T->colact.p;
    static std::mutex mu;
    {
        std::lock_guard<std::mutex> lk(mu);
        if (grid_prepare_kernels(g.lx, g.ly) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
    }
    P.grid = std::move(T);
    return true;
}
