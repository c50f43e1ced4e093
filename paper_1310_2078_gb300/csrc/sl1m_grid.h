// sl1m_grid.h -- the lattice operator of libsl1m (internal): forward and
// adjoint of Dirac pixels on a regular (l, m) lattice by gridding and FFT.
#pragma once
#include <cstddef>

#include "sl1m_dev.h"

namespace sl1m {

constexpr int GRW = 8;          // gridding kernel width: cells per axis, and planes in w
constexpr int GR_TILE = 16;     // the adjoint spreads onto tiles of GR_TILE^2 cells
constexpr int GR_PCH = 8;       // planes a CTA of the row kernels takes
constexpr int GR_LOG_MIN = 6, GR_LOG_MAX = 12;   // FFT lengths 64 .. 4096
// The exponential-of-semicircle kernel phi(z) = exp(GR_BETA (sqrt(1 - (2z/GRW)^2) - 1)).
constexpr double GR_BETA = 2.30 * GRW;
// Inputs are scaled by GR_SCALE, so that small ones stay clear of FP32's
// denormals, unless one is GR_HUGE or more (DevProblem::huge): then by 1 / the
// number of them, so that a coherent sum of the largest stays in range.  Powers of
// two: in between the results are the same.
constexpr double GR_HUGE = 1099511627776.0;            // 2^40
constexpr float GR_SCALE = 1099511627776.0f;
constexpr int GR_NQ = 32;       // Gauss-Legendre nodes on half the kernel's support

// One problem's lattice operator (pointers into device memory).
struct GridOp {
    int nx, ny;                 // lattice cells
    int cx, cy;                 // the cell at the origin of the transforms
    int lx, ly;                 // log2 of the FFT lengths (2^lx >= 2 nx, 2^ly >= 2 ny)
    int np;                     // planes in w
    int np_pass;                // planes the workspace holds at a time
    int n_chunk;                // adjoint partial slots: chunks of GR_PCH planes of one pass
    float fscale, ascale;       // powers of two that keep the transforms' sums of huge inputs in range
    const int* cell;            // [ny][nx] sorted pixel index, -1 where the lattice has no pixel
    const float* amp;           // [ny][nx] (1/n) / (kernel transforms), 0 without a pixel
    const float2* nu;           // [ny][nx] n - 1 - nc, FP32 hi and lo
    const float2* wp;           // [np] w of each plane, FP32 hi and lo
    const float2* twx;          // twiddles of the row and the column transforms
    const float2* twy;
    const int4* pos;            // [vis.n_pad] first cell x, y (wrapped), first plane, 1 if mirrored
    const float* wts;           // [vis.n_pad][3 GRW] kernel weights in x, y, w
    const float2* rot;          // [vis.n_pad] exp(-2 pi i (u lc + v mc + w nc))
    const int* order;           // [vis.n_pad] the visibilities by tile and first plane
    const int* list;            // visibilities touching each tile, by first plane
    const int* start;           // [tiles][np - GRW + 2] list offsets
    const unsigned char* act;   // [np][tiles in x][tiles in y] 1 where a visibility touches the plane's tile
    const unsigned char* colact;  // [np][tiles in x] any of them
    float2* g1;                 // workspace [np_pass][ny][2^lx]
    float2* g2;                 // workspace [np_pass][2^ly][2^lx]
};

inline size_t grid_plane_elems(const GridOp& g) { return ((size_t)g.ny + ((size_t)1 << g.ly)) << g.lx; }
inline int grid_tiles(const GridOp& g) { return ((1 << g.lx) / GR_TILE) * ((1 << g.ly) / GR_TILE); }
// Bytes of its partial sums, forward and adjoint.
inline size_t grid_sum_bytes(const GridOp& g, int vis_blk, int pix_blk)
{
    return ((size_t)vis_blk * 16 + (size_t)pix_blk * 8 * g.n_chunk) * BLK;
}
// Radix of a transform of length 2^lg, and of its first pass: 16 where that saves
// an exchange over radix 8.
constexpr int grid_radix(int lg) { return lg == 6 || lg == 9 ? 8 : 16; }
constexpr int grid_radix0(int lg) { return grid_radix(lg) == 8 ? 8 : lg % 4 ? 1 << (lg % 4) : 16; }
// float2 entries of its twiddle table.
inline int grid_tw_elems(int lg)
{
    const int radix = grid_radix(lg);
    int n = 0;
    for (int ns = grid_radix0(lg); ns < (1 << lg); ns *= radix) n += (radix == 16 ? 4 : 3) * ns;
    return n;
}

// set-up (once per layout)
cudaError_t grid_setup_vis(const d4* vd, int n_pad, GridOp g, double dl, double dm, double lc, double mc, double nc,
                           double w0, double dw, int4* pos, float* wts, float2* rot, cudaStream_t st);
cudaError_t grid_setup_cells(const d4* pd, GridOp g, const double* cxy, const double* quad, double nc, double dw,
                             float* amp, float2* nu, cudaStream_t st);

// operator launches for problem p of probs (nothing runs when the problem has
// no role in this step); *n_launch counts the kernels.
// Forward: sums into partial [vis.n_pad]; adjoint: into partial[slot], slot =
// block n_chunk + chunk, BLK elements each.
cudaError_t grid_forward(const DevProblem* probs, int p, const GridOp& g, int n_vis_pad, double2* partial,
                         cudaStream_t st, long long* n_launch);
cudaError_t grid_adjoint(const DevProblem* probs, int p, const GridOp& g, int n_pix, int n_pix_pad, double* partial,
                         cudaStream_t st, long long* n_launch);
// raises the dynamic shared-memory limits of the transforms of these lengths (not under capture)
cudaError_t grid_prepare_kernels(int lx, int ly);

}  // namespace sl1m
