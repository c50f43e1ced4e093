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

// Loops over the pixels, cut into NT chunks, on as many threads as pay (one takes
// tens of us to start).
constexpr size_t NT = 16;
template <class F>
void pixel_chunks(int64_t n, const F& fn)
{
    parallel_chunks(NT, (size_t)std::max<int64_t>(1, 65536 * (int64_t)NT / std::max<int64_t>(1, n)), [&](size_t t0, size_t t1) {
        for (size_t t = t0; t < t1; ++t) fn(t, (size_t)n * t / NT, (size_t)n * (t + 1) / NT);
    });
}

// Both axes, and the range of n - 1.  The spacing is the smallest distance from
// the first pixel, refined over the whole span; every pixel then has to sit on its
// lattice point to within `tol` (a phase error of 1e-8 turn at the longest
// baseline).  A lattice whose first pixel has no neighbour one step away is not
// recognised.
void find_axes(const double* lm, int64_t n, const double (&tol)[2], Axis (&A)[2], double& n0, double& n1)
{
    struct Part {
        double near[2] = {1e300, 1e300}, lo[2] = {1e300, 1e300}, hi[2] = {-1e300, -1e300}, n0 = 1e300, n1 = -1e300;
        bool off[2] = {false, false};
    };
    std::vector<Part> part(NT);
    for (int a = 0; a < 2; ++a) A[a].x0 = lm[a];
    pixel_chunks(n, [&](size_t t, size_t i0, size_t i1) {
        Part p;
        for (size_t i = i0; i < i1; ++i) {
            for (int a = 0; a < 2; ++a) {
                const double v = lm[2 * i + a], d = std::fabs(v - A[a].x0);
                if (d > tol[a]) p.near[a] = std::min(p.near[a], d);
                p.lo[a] = std::min(p.lo[a], v);
                p.hi[a] = std::max(p.hi[a], v);
            }
            const double r2 = lm[2 * i] * lm[2 * i] + lm[2 * i + 1] * lm[2 * i + 1];
            const double v = -r2 / (1.0 + std::sqrt(1.0 - r2));
            p.n0 = std::min(p.n0, v);
            p.n1 = std::max(p.n1, v);
        }
        part[t] = p;
    });
    Part all;
    for (const Part& p : part) {
        for (int a = 0; a < 2; ++a) {
            all.near[a] = std::min(all.near[a], p.near[a]);
            all.lo[a] = std::min(all.lo[a], p.lo[a]);
            all.hi[a] = std::max(all.hi[a], p.hi[a]);
        }
        all.n0 = std::min(all.n0, p.n0);
        all.n1 = std::max(all.n1, p.n1);
    }
    n0 = all.n0;
    n1 = all.n1;
    for (int a = 0; a < 2; ++a) {
        if (all.near[a] > 1e299) continue;              // one value
        const double up = all.hi[a] - A[a].x0, down = A[a].x0 - all.lo[a], span = up > down ? up : down;
        const double steps = std::rint(span / all.near[a]);
        if (!(steps >= 1.0) || steps > 8192.0) return;
        A[a].step = span / steps;
        A[a].kmin = (int)std::rint((all.lo[a] - A[a].x0) / A[a].step);
        A[a].n = (int)std::rint((all.hi[a] - A[a].x0) / A[a].step) - A[a].kmin + 1;
    }
    pixel_chunks(n, [&](size_t t, size_t i0, size_t i1) {
        bool off[2] = {false, false};
        for (int a = 0; a < 2; ++a) {
            if (A[a].n == 1) continue;
            for (size_t i = i0; i < i1; ++i) {
                const double d = lm[2 * i + a] - A[a].x0;
                off[a] |= std::fabs(d - std::rint(d / A[a].step) * A[a].step) > tol[a];
            }
        }
        std::copy(off, off + 2, part[t].off);
    });
    for (int a = 0; a < 2; ++a)
        A[a].ok = std::none_of(part.begin(), part.end(), [a](const Part& p) { return p.off[a]; });
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
// The fit is older than the ring-buffer spreading and the radix-16 transforms and puts
// the lattice about a third too high (256^2 +/-0.5 x 40,320: 400 us, measured 300;
// 1024^2 x 406,400: 1,444, measured 1,055); pairs on the exact path, three times as dear,
// are not in pair_seconds (256^2 +/-0.5 x 5,000: 165 us, measured 270).  Both err
// towards the pairs, and both directions take one operator: 64^2 x 40,000 would want
// the lattice forward and the pair adjoint.
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
    Axis axes[2];
    find_axes(P.lm.data(), P.n_pix, {1e-8 / std::max(1.0, um), 1e-8 / std::max(1.0, vm)}, axes, n0, n1);
    const Axis &ax = axes[0], &ay = axes[1];
    if (!ax.ok || !ay.ok) return false;
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
    const double wp0 = w0 - (0.5 * GRW - 0.5) * dw;
    // any failure below (memory, above all) leaves the pair operator in place.  The
    // set-up kernels run while the host makes the tables and the lists.
    bool ok = T->pos.alloc(nv) == cudaSuccess && T->wts.alloc(nv * 3 * GRW) == cudaSuccess && T->rot.alloc(nv) == cudaSuccess &&
              grid_setup_vis(P.hp.vis.d, (int)nv, g, ax.step, ay.step, ax.x0 + (ax.kmin + g.nx / 2) * ax.step,
                             ay.x0 + (ay.kmin + g.ny / 2) * ay.step, nc, wp0, dw, T->pos.p, T->wts.p, T->rot.p,
                             st) == cudaSuccess;
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
    const auto hats = [&](int n, int c, int lg, double* out) {        // (even in i - c)
        for (int i = 0; i <= c; ++i) out[i] = inv_hat((double)(i - c) / (1 << lg));
        for (int i = c + 1; i < n; ++i) out[i] = 2 * c - i >= 0 ? out[2 * c - i] : inv_hat((double)(i - c) / (1 << lg));
    };
    hats(g.nx, g.cx, g.lx, cxy.data());
    if (g.ny == g.nx && g.ly == g.lx) std::copy(cxy.begin(), cxy.begin() + g.nx, cxy.begin() + g.nx);
    else hats(g.ny, g.cy, g.ly, cxy.data() + g.nx);
    std::vector<float2> wp(g.np);
    for (int p = 0; p < g.np; ++p) {
        const double w = wp0 + p * dw;
        wp[p] = make_float2((float)w, (float)(w - (double)(float)w));
    }
    const std::vector<float2> tx = twiddles(g.lx), ty = twiddles(g.ly);
    ok = ok && T->cell.upload(cell.data(), cells, st) == cudaSuccess && T->wp.upload(wp.data(), wp.size(), st) == cudaSuccess &&
         T->twx.upload(tx.data(), tx.size(), st) == cudaSuccess && T->twy.upload(ty.data(), ty.size(), st) == cudaSuccess &&
         T->amp.alloc(cells) == cudaSuccess && T->nu.alloc(cells) == cudaSuccess &&
         T->huge.upload(nullptr, 3, st, true) == cudaSuccess;
    DBuf<double> dq, dc;
    ok = ok && dq.upload(quad.data(), quad.size(), st) == cudaSuccess && dc.upload(cxy.data(), cxy.size(), st) == cudaSuccess;
    std::vector<int4> pos(nv);
    if (ok) {
        g.cell = T->cell.p;
        g.wp = T->wp.p;
        g.twx = T->twx.p;
        g.twy = T->twy.p;
        ok = cudaMemcpyAsync(pos.data(), T->pos.p, nv * sizeof(int4), cudaMemcpyDeviceToHost, st) == cudaSuccess &&
             cudaStreamSynchronize(st) == cudaSuccess &&
             grid_setup_cells(P.hp.pix.d, g, dc.p, dq.p, nc, dw, T->amp.p, T->nu.p, st) == cudaSuccess;
    }
    // visibilities per tile (at most two tiles per axis), by first plane, in the
    // library's order: counting sorts by tile and then, within each, by plane;
    // on threads of their own by rows of tiles where there are many
    std::vector<int> start, list, order;
    if (ok) {
        const int txn = (1 << g.lx) / GR_TILE, tyn = (1 << g.ly) / GR_TILE, mx = (1 << g.lx) - 1, my = (1 << g.ly) - 1;
        struct Part {
            int y0, y1, n_list = 0, n_order = 0;
            std::vector<int> at, by_tile;                    // tile's first in by_tile; visibilities by tile
        };
        std::vector<Part> part(nv + (size_t)tiles * ni < ((size_t)1 << 20) ? 1 : std::min<size_t>(8, (size_t)tyn));
        for (size_t t = 0; t < part.size(); ++t) {
            part[t].y0 = (int)(tyn * t / part.size());
            part[t].y1 = (int)(tyn * (t + 1) / part.size());
        }
        const auto parts = [&](const auto& fn) {
            parallel_chunks(part.size(), 1, [&](size_t t0, size_t t1) {
                for (size_t t = t0; t < t1; ++t) fn(t, part[t]);
            });
        };
        parts([&](size_t, Part& p) {
            // f(visibility, tile, whether it counts) over a visibility's four tiles: a
            // test per tile would be guessed wrong half the time, so they all run
            const auto each = [&](const auto& f) {
                const int y0 = p.y0, rows = p.y1 - p.y0;
                for (size_t k = 0; k < nv; ++k) {
                    const int4 q = pos[k];
                    const unsigned xa = (unsigned)q.x / GR_TILE, xb = (unsigned)((q.x + GRW - 1) & mx) / GR_TILE;
                    const unsigned ya = (unsigned)q.y / GR_TILE - y0, yb = (unsigned)((q.y + GRW - 1) & my) / GR_TILE - y0;
                    const bool in = P.vis_orig[k] >= 0, a = in & (ya < (unsigned)rows), b = in & (yb < (unsigned)rows) & (yb != ya);
                    if (rows < tyn && !a && !b) continue;
                    const unsigned ra = a ? ya * txn : 0, rb = b ? yb * txn : 0;
                    f((int)k, ra + xa, a);
                    f((int)k, ra + xb, a & (xb != xa));
                    f((int)k, rb + xa, b);
                    f((int)k, rb + xb, b & (xb != xa));
                    p.n_order += a;
                }
            };
            // (a place more per tile: what does not count is written there, too)
            const int n = (p.y1 - p.y0) * txn;
            p.at.assign((size_t)n + 1, 0);
            each([&](int, unsigned t, bool in) { p.at[t + 1] += in; });
            for (int t = 0; t < n; ++t) {
                p.n_list += p.at[t + 1];
                p.at[t + 1] += p.at[t] + 1;
            }
            p.by_tile.resize(p.at.back());
            std::vector<int> fill(p.at.begin(), p.at.end() - 1);
            p.n_order = 0;
            each([&](int k, unsigned t, bool in) {
                p.by_tile[fill[t]] = k;
                fill[t] += in;
            });
        });
        std::vector<int> list0(part.size() + 1, 0), order0(part.size() + 1, 0);
        for (size_t t = 0; t < part.size(); ++t) {
            list0[t + 1] = list0[t] + part[t].n_list;
            order0[t + 1] = order0[t] + part[t].n_order;
        }
        start.resize((size_t)tiles * (ni + 1) + 1);
        start[0] = 0;
        list.resize(std::max(1, list0.back()));
        order.resize(nv);
        std::vector<unsigned char> act((size_t)g.np * tiles, 0), colact((size_t)g.np * txn, 0);
        parts([&](size_t n, Part& p) {
            std::vector<int> mine(p.n_order + 1);                    // (a place more: written before it is known to count)
            int* out = mine.data();
            std::vector<int> fill(ni);
            int sum = list0[n];
            for (int t = 0; t < (p.y1 - p.y0) * txn; ++t) {
                const int* k0 = p.by_tile.data() + p.at[t];
                const int* k1 = p.by_tile.data() + p.at[t + 1] - 1;
                const int tile = p.y0 * txn + t, first = sum;
                int* st = start.data() + (size_t)tile * (ni + 1) + 1;       // ends of the planes; st[-1]: the tile before
                std::fill(fill.begin(), fill.end(), 0);
                for (const int* k = k0; k < k1; ++k) ++fill[pos[*k].z];
                for (int z = 0; z < ni; ++z) {
                    st[z] = sum + fill[z];
                    fill[z] = sum;
                    sum = st[z];
                }
                st[ni] = sum;
                for (const int* k = k0; k < k1; ++k) list[fill[pos[*k].z]++] = *k;
                // each visibility once, at its first tile
                for (int i = first; i < sum; ++i) {
                    const int4 q = pos[list[i]];
                    *out = list[i];
                    out += (q.y / GR_TILE) * txn + q.x / GR_TILE == tile;
                }
            }
            std::copy(mine.data(), out, order.data() + order0[n]);
        });
        // which planes of a tile have a visibility (a column of tiles after the other: its
        // planes' bytes are neighbours); those below `done` are marked
        parts([&](size_t n, Part& p) {
            for (int x = 0; x < txn; ++x)
                for (int y = p.y0; y < p.y1; ++y) {
                    const int* st = start.data() + ((size_t)y * txn + x) * (ni + 1) + 1;
                    int from = y == p.y0 && x == 0 ? list0[n] : st[-1];
                    for (int z = 0, done = 0; z < ni; from = st[z], ++z) {
                        if (st[z] == from) continue;
                        for (int d = std::max(z, done); d < z + GRW; ++d) act[((size_t)d * txn + x) * tyn + y] = 1;
                        done = z + GRW;
                    }
                }
        });
        for (size_t c = 0; c < colact.size(); ++c) colact[c] = std::memchr(act.data() + c * tyn, 1, tyn) != nullptr;
        size_t at = order0.back();                           // then the padding slots
        for (size_t k = 0; k < nv; ++k)
            if (P.vis_orig[k] < 0) order[at++] = (int)k;
        ok = T->start.upload(start.data(), start.size(), st) == cudaSuccess &&
             T->list.upload(list.data(), list.size(), st) == cudaSuccess &&
             T->order.upload(order.data(), nv, st) == cudaSuccess &&
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
