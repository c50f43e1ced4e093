// sl1m_solver.cu -- the vector side of SL1M's FISTA (Hardy 2013, Sect. 3):
// finishing the stream-K partial sums of the operator kernels, the residual
// r = W (A y - V) and its norm, the positive soft threshold (Eq. threshp) and
// the momentum step of the algorithm box, the power iteration for L, and the
// per-problem FP64 scalars.  All reductions use a fixed order (deterministic,
// no atomics).  These kernels are bound by HBM bandwidth on large problems and
// by the latency of dependent loads on small ones.
#include <math.h>

#include "sl1m_dev.h"
#include "sl1m_grid.h"
#include "sl1m_kernels.h"

namespace sl1m {

// Marks an input of a lattice operator that needs the other scale (sl1m_grid.h).
__device__ __forceinline__ void mark_huge(int* flag, double v)
{
    if (flag && !(fabs(v) < GR_HUGE)) *flag = 1;
}
__device__ __forceinline__ void mark_huge(int* flag, double2 v)
{
    mark_huge(flag, v.x);
    mark_huge(flag, v.y);
}

// ---------------------------------------------------------- permutations

__global__ void gather_real_kernel(const double* __restrict__ src, double* __restrict__ dst,
                                   const int* __restrict__ orig, int n_pad, double scale, int* huge)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_pad; i += gridDim.x * blockDim.x) {
        const int o = orig[i];
        const double v = o >= 0 ? src[o] * scale : 0.0;
        dst[i] = v;
        mark_huge(huge, v);
    }
}

// r in the library's visibility order, and in polar form (write_polar).
__device__ __forceinline__ void write_polar(const DevProblem& P, int polar, int e, double2 v);
__global__ void gather_resid_kernel(const double2* __restrict__ src, const DevProblem* __restrict__ P, int polar,
                                    double2* __restrict__ dst)
{
    const int n_pad = P->vis.n_pad;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_pad; i += gridDim.x * blockDim.x) {
        const int o = P->vis.orig[i];
        const double2 v = o >= 0 ? src[o] : make_double2(0.0, 0.0);
        dst[i] = v;
        write_polar(*P, polar, i, v);
        mark_huge(P->huge ? P->huge + 1 : nullptr, v);
    }
}

__global__ void scatter_real_kernel(const double* __restrict__ src, double* __restrict__ dst,
                                    const int* __restrict__ orig, int n_pad)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_pad; i += gridDim.x * blockDim.x) {
        const int o = orig[i];
        if (o >= 0) dst[o] = src[i];
    }
}

__global__ void scatter_cplx_kernel(const double2* __restrict__ src, double2* __restrict__ dst,
                                    const int* __restrict__ orig, int n_pad)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_pad; i += gridDim.x * blockDim.x) {
        const int o = orig[i];
        if (o >= 0) dst[o] = src[i];
    }
}

__global__ void fill_valid_kernel(double* __restrict__ dst, const int* __restrict__ orig, int n_pad,
                                  double val)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_pad; i += gridDim.x * blockDim.x)
        dst[i] = orig[i] >= 0 ? val : 0.0;
}

// r = W V in the library's visibility order (input of the dirty image).
__global__ void weighted_vis_kernel(const DevProblem* __restrict__ P, int polar, double2* __restrict__ r)
{
    const int n_pad = P->vis.n_pad;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_pad; i += gridDim.x * blockDim.x) {
        const double w = P->vis.d[i].w;
        const double2 v = make_double2(w * P->V[i].x, w * P->V[i].y);
        r[i] = v;
        write_polar(*P, polar, i, v);
        mark_huge(P->huge ? P->huge + 1 : nullptr, v);
    }
}

static int grid_for(int n) { return n <= 0 ? 1 : (n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096; }

cudaError_t launch_gather_real(const double* src, double* dst, const int* orig, int n_pad,
                               double scale, int* huge, cudaStream_t st)
{
    gather_real_kernel<<<grid_for(n_pad), 256, 0, st>>>(src, dst, orig, n_pad, scale, huge);
    return cudaGetLastError();
}
cudaError_t launch_gather_resid(const double2* src, const DevProblem* P, int n_pad, int polar, double2* dst,
                                cudaStream_t st)
{
    gather_resid_kernel<<<grid_for(n_pad), 256, 0, st>>>(src, P, polar, dst);
    return cudaGetLastError();
}
cudaError_t launch_scatter_real(const double* src, double* dst, const int* orig, int n_pad,
                                cudaStream_t st)
{
    scatter_real_kernel<<<grid_for(n_pad), 256, 0, st>>>(src, dst, orig, n_pad);
    return cudaGetLastError();
}
cudaError_t launch_scatter_cplx(const double2* src, double2* dst, const int* orig, int n_pad,
                                cudaStream_t st)
{
    scatter_cplx_kernel<<<grid_for(n_pad), 256, 0, st>>>(src, dst, orig, n_pad);
    return cudaGetLastError();
}
cudaError_t launch_weighted_vis(const DevProblem* P, int n_pad, int polar, double2* r, cudaStream_t st)
{
    weighted_vis_kernel<<<grid_for(n_pad), 256, 0, st>>>(P, polar, r);
    return cudaGetLastError();
}

cudaError_t launch_fill_valid(double* dst, const int* orig, int n_pad, double val, cudaStream_t st)
{
    fill_valid_kernel<<<grid_for(n_pad), 256, 0, st>>>(dst, orig, n_pad, val);
    return cudaGetLastError();
}

// --------------------------------------------------------------- helpers

// t_{k+1} = (1 + sqrt(1 + 4 t_k^2)) / 2 and beta_k = (t_k - 1) / t_{k+1}
// (the momentum step of the FISTA box).
__device__ __forceinline__ void fista_beta(double t, double& t_next, double& beta)
{
    t_next = 0.5 * (1.0 + sqrt(1.0 + 4.0 * t * t));
    beta = (t - 1.0) / t_next;
}

__device__ __forceinline__ int find_blk_prob(const Plan& pl, int gb)
{
    int lo = 0, hi = pl.n_probs - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (pl.prob_b0[mid] <= gb) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Fixed-order sums over a warp (xor tree) and over a CTA of 256 threads (warps
// in order; every thread calls it, thread 0 has the result).
template <class T>
__device__ __forceinline__ T warp_sum(T v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
template <class T>
__device__ __forceinline__ T cta_sum(T v, T* sh)
{
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    T r = 0;
    if (threadIdx.x == 0)
        for (int w = 0; w < 8; ++w) r += sh[w];
    __syncthreads();
    return r;
}

// Mode of problem P in a finish kernel: FIN_OP (operator call), FIN_POWER,
// FIN_INIT, FIN_SOLVE, or -1 (P takes no part in this step).
__device__ __forceinline__ int fwd_finish_mode(const DevProblem& P)
{
    if (!P.st) return FIN_OP;
    switch (P.st->phase) {
    case PH_PINIT:
    case PH_POWER: return FIN_POWER;
    case PH_SINIT: return FIN_INIT;
    case PH_SOLVE: return FIN_SOLVE;
    default: return -1;
    }
}

__device__ __forceinline__ int adj_finish_mode(const DevProblem& P)
{
    if (!P.st) return FIN_OP;
    switch (P.st->phase) {
    case PH_POWER: return FIN_POWER;
    case PH_SOLVE: return FIN_SOLVE;
    default: return -1;
    }
}

template <class T>
__device__ __forceinline__ void add_in(T& s, const T& q);
template <>
__device__ __forceinline__ void add_in<double>(double& s, const double& q) { s += q; }
template <>
__device__ __forceinline__ void add_in<double2>(double2& s, const double2& q)
{
    s.x += q.x;
    s.y += q.y;
}
__device__ __forceinline__ double zero_of(double) { return 0.0; }
__device__ __forceinline__ double2 zero_of(double2) { return make_double2(0.0, 0.0); }

// The finish kernels sum an element's partial slots over SL threads (slots sl,
// sl + SL, ...; 8 loads in flight at a time), then the SL sums in order: the
// same order every time.  A CTA takes FIN_EL<SL> elements, whole granules of one
// block.  With one thread per element, a small problem -- few blocks, each
// with a partial slot of nearly every CTA of its operator -- was a chain of
// dependent loads in a handful of CTAs: 1024 pixels x 2208 visibilities in
// FP64, 2 CTAs summing 228 slots, took 108 us of a 280 us step.
template <int SL>
struct FinShape {
    static constexpr int THREADS = SL >= 8 ? 512 : 256;
    static constexpr int EL = THREADS / SL;             // elements per CTA: 64 or 256
    static constexpr int NG = EL / G;                   // granules per CTA
};

template <int SL, class T>
__device__ __forceinline__ T sum_slots(const T* __restrict__ partial, int blk_el, int poff, int ncon, int i,
                                       T* __restrict__ sh)
{
    constexpr int EL = FinShape<SL>::EL;
    const int sl = threadIdx.x / EL;
    T s = zero_of(T());
    int c = sl;
    for (; c + 7 * SL < ncon; c += 8 * SL) {
        T q[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) q[t] = partial[(size_t)(poff + c + t * SL) * blk_el + i];
#pragma unroll
        for (int t = 0; t < 8; ++t) add_in(s, q[t]);
    }
    for (; c < ncon; c += SL) add_in(s, partial[(size_t)(poff + c) * blk_el + i]);
    if (SL > 1) {
        sh[threadIdx.x] = s;
        __syncthreads();
        if (sl == 0)
            for (int t = 1; t < SL; ++t) add_in(s, sh[t * EL + threadIdx.x]);
        __syncthreads();
    }
    return s;
}

// Where a finish CTA works: granule group q of the plan.  False: nothing there.
template <int SL>
__device__ __forceinline__ bool fin_place(const Plan& pl, const DevProblem* probs, int q, bool vis, int& p, int& gb,
                                          int& i0, int& e0)
{
    const int per = max(1, pl.blk_el / FinShape<SL>::EL);       // groups per block
    gb = q / per;
    i0 = (q % per) * FinShape<SL>::EL;                          // first element within the block
    p = find_blk_prob(pl, gb);
    e0 = (gb - pl.prob_b0[p]) * pl.blk_el + i0;                 // ... and of the side
    return e0 < (vis ? probs[p].vis.n_pad : probs[p].pix.n_pad);
}

// r of the next adjoint in polar form, as its kernels read it: POLAR 1 r32
// (mixed), 2 r64 (FP64); modulus and argument are taken in FP64.
constexpr double INV_TWO_PI = 0.15915494309189533577;
__device__ __forceinline__ void write_polar(const DevProblem& P, int polar, int e, double2 v)
{
    if (polar == 0) return;
    const double m = hypot(v.x, v.y), a = atan2(v.y, v.x) * INV_TWO_PI;
    if (polar == 1) P.r32[e] = make_float2((float)m, (float)a);
    else if (P.r64) P.r64[e] = make_double2(a * R64_TURN, m);
}

// ---------------------------------------------------------- forward finish
// Grid-stride over the plan's owned blocks: sums the block's partial slots,
// then per problem
//   FIN_OP    : A x, into user_out in the caller's order
//   FIN_POWER : r = W (A x)                      (input of the next adjoint)
//   FIN_INIT  : AI_0 = A I_0, r = W (A I_0 - V), sums of W|A I_0 - V|^2
//   FIN_SOLVE : AI_k = A I_k, sums of W|A I_k - V|^2,
//               A y_{k+1} = AI_k + beta_k (AI_k - AI_{k-1})  (linearity),
//               r = W (A y_{k+1} - V)
//               (MFISTA: A z_k and its sums only)
// Sums are per granule of 64; r is also written in polar form (polar).
template <int SL>
__global__ void __launch_bounds__(FinShape<SL>::THREADS)
fwd_finish_kernel(const DevProblem* __restrict__ probs, const Plan* __restrict__ plp,
                  const double2* __restrict__ partial, int polar, double2* __restrict__ user_out)
{
    using S = FinShape<SL>;
    __shared__ double2 sh2[SL > 1 ? S::THREADS : 1];
    __shared__ double sh_r2[S::EL / 32];
    __shared__ int sh_bad[S::EL / 32];
    const Plan pl = *plp;
    const int nq = pl.n_blocks * max(1, pl.blk_el / S::EL);
    for (int q = blockIdx.x; q < nq; q += gridDim.x) {
        int p, gb, i0, e0;
        if (!fin_place<SL>(pl, probs, q, true, p, gb, i0, e0)) continue;
        const DevProblem& P = probs[p];
        const int mode = fwd_finish_mode(P);
        if (mode < 0) continue;
        if (P.huge && e0 == 0 && threadIdx.x == 0) P.huge[0] = 0;      // (the operator is done with it)
        const int t = threadIdx.x % S::EL, e = e0 + t;
        const bool in = e < P.vis.n_pad;
        const int poff = pl.blk_poff[gb], ncon = in ? pl.blk_ncon[gb] : 0;
        const double2 s = sum_slots<SL>(partial, pl.blk_el, poff, ncon, i0 + t, sh2);
        double bn = 0.0;
        int bad = 0;
        if (threadIdx.x < S::EL && in) {
            if (!isfinite(s.x) || !isfinite(s.y)) bad = 1;
            const SolveBufs& B = P.b;
            if (mode == FIN_OP) {
                const int o = user_out ? P.vis.orig[e] : e;
                if (o >= 0) (user_out ? user_out : P.fwd_out)[o] = s;
            } else if (mode == FIN_POWER) {
                const double W = P.vis.d[e].w;
                const double2 r = make_double2(W * s.x, W * s.y);
                B.r[e] = r;
                write_polar(P, polar, e, r);
                mark_huge(P.huge ? P.huge + 1 : nullptr, r);
            } else {
                const double W = P.vis.d[e].w;
                const double2 V = P.V[e];
                const double dr = s.x - V.x, di = s.y - V.y;
                bn = W * (dr * dr + di * di);
                double2 r = make_double2(W * dr, W * di);
                const SolveState& S2 = *P.st;
                if (mode == FIN_INIT) {
                    B.AI[0][e] = s;
                } else if (S2.algo) {
                    B.AI[1][e] = s;                 // A z_k; r is formed by the mix kernel
                } else {
                    double tn, beta;
                    fista_beta(S2.t, tn, beta);
                    const int par = (S2.k + 1) & 1;
                    const double2 old = B.AI[par ^ 1][e];
                    B.AI[par][e] = s;
                    const double ayr = s.x + beta * (s.x - old.x);
                    const double ayi = s.y + beta * (s.y - old.y);
                    r = make_double2(W * (ayr - V.x), W * (ayi - V.y));
                }
                if (mode == FIN_INIT || !S2.algo) {
                    B.r[e] = r;
                    write_polar(P, polar, e, r);
                    mark_huge(P.huge ? P.huge + 1 : nullptr, r);
                }
            }
        }
        if (mode == FIN_OP) continue;
        if (threadIdx.x < S::EL) {
            const double tot = warp_sum(bn);
            const int nb = warp_sum(bad);
            if ((threadIdx.x & 31) == 0) {
                sh_r2[threadIdx.x >> 5] = tot;
                sh_bad[threadIdx.x >> 5] = nb;
            }
        }
        __syncthreads();
        if (threadIdx.x < S::NG && e0 + (int)threadIdx.x * G < P.vis.n_pad) {
            const int g = e0 / G + threadIdx.x, w = 2 * threadIdx.x;
            P.b.blk_badv[g] = sh_bad[w] + sh_bad[w + 1];
            if (mode != FIN_POWER) P.b.blk_r2[g] = sh_r2[w] + sh_r2[w + 1];
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------- adjoint finish
//   FIN_OP    : Re A^H r, into user_out in the caller's order
//   FIN_POWER : z = (Re A^H W A x) * inv_mu into xv (= B x_unit), sums of z^2
//   FIN_SOLVE : I_k = T^{lambda/L}(y_k - g/L)                 (Eq. threshp)
//               y_{k+1} = I_k + beta_k (I_k - I_{k-1})        (FISTA box)
//               sums of I_k and of nnz
//               (MFISTA: z_k = T^{lambda/L}(y_k - g/L) and its sums only)
template <int SL>
__global__ void __launch_bounds__(FinShape<SL>::THREADS)
adj_finish_kernel(const DevProblem* __restrict__ probs, const Plan* __restrict__ plp,
                  const double* __restrict__ partial, double* __restrict__ user_out)
{
    using S = FinShape<SL>;
    __shared__ double sh1[SL > 1 ? S::THREADS : 1];
    __shared__ double sh_acc[S::EL / 32];
    __shared__ int sh_cnt[S::EL / 32], sh_bad[S::EL / 32];
    const Plan pl = *plp;
    const int nq = pl.n_blocks * max(1, pl.blk_el / S::EL);
    for (int q = blockIdx.x; q < nq; q += gridDim.x) {
        int p, gb, i0, e0;
        if (!fin_place<SL>(pl, probs, q, false, p, gb, i0, e0)) continue;
        const DevProblem& P = probs[p];
        const int mode = adj_finish_mode(P);
        if (mode < 0) continue;
        if (P.huge && e0 == 0 && threadIdx.x == 0) P.huge[1] = 0;      // (the operator is done with it)
        const int t = threadIdx.x % S::EL, e = e0 + t;
        const bool in = e < P.pix.n_pad;
        const int poff = pl.blk_poff[gb], ncon = in ? pl.blk_ncon[gb] : 0;
        // the step's other loads are issued before the partial sums
        const int par = mode == FIN_SOLVE && !P.st->algo ? (P.st->k + 1) & 1 : 0;
        double y0 = 0.0, Io = 0.0;
        int orig = 0;
        if (mode == FIN_SOLVE && threadIdx.x < S::EL && in) {
            y0 = P.b.y[e];
            Io = P.b.I[par ^ 1][e];
            orig = P.pix.orig[e];
        }
        const double s = sum_slots<SL>(partial, pl.blk_el, poff, ncon, i0 + t, sh1);
        double acc = 0.0;
        int cnt = 0, bad = 0;
        if (threadIdx.x < S::EL && in) {
            if (!isfinite(s)) bad = 1;
            const SolveBufs& B = P.b;
            if (mode == FIN_OP) {
                const int o = user_out ? P.pix.orig[e] : e;
                if (o >= 0) (user_out ? user_out : P.adj_out)[o] = s;
            } else if (mode == FIN_POWER) {
                const double z = s * P.st->inv_mu;
                B.xv[e] = z;
                mark_huge(P.huge, z);
                acc = z * z;
            } else {
                const SolveState& S2 = *P.st;
                const double inv_L = 1.0 / S2.L, thr = S2.lambda / S2.L;
                const double v = y0 - s * inv_L;
                double In = v > thr ? v - thr : 0.0;
                if (orig < 0) In = 0.0;
                mark_huge(P.huge, In);
                if (S2.algo) {
                    B.I[1][e] = In;                 // z_k; y is formed by the mix kernel
                } else {
                    double tn, beta;
                    fista_beta(S2.t, tn, beta);
                    B.I[par][e] = In;
                    B.y[e] = In + beta * (In - Io);
                }
                acc = In;
                cnt = In > 0.0;
            }
        }
        if (mode == FIN_OP) continue;
        if (threadIdx.x < S::EL) {
            const double tot = warp_sum(acc);
            const int nb = warp_sum(bad), nz = warp_sum(cnt);
            if ((threadIdx.x & 31) == 0) {
                sh_acc[threadIdx.x >> 5] = tot;
                sh_bad[threadIdx.x >> 5] = nb;
                sh_cnt[threadIdx.x >> 5] = nz;
            }
        }
        __syncthreads();
        if (threadIdx.x < S::NG && e0 + (int)threadIdx.x * G < P.pix.n_pad) {
            const SolveBufs& B = P.b;
            const int g = e0 / G + threadIdx.x, w = 2 * threadIdx.x;
            const double tot = sh_acc[w] + sh_acc[w + 1];
            if (mode == FIN_POWER) B.blk_z2[g] = tot;
            else {
                B.blk_l1[g] = tot;
                B.blk_nnz[g] = sh_cnt[w] + sh_cnt[w + 1];
            }
            B.blk_badp[g] = sh_bad[w] + sh_bad[w + 1];
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------ scalars
// One CTA of 256 threads per problem; fixed-order sums of the finish kernels'
// per-granule sums (thread-strided, then cta_sum).
template <class R, class T>
__device__ __forceinline__ R strided(const T* a, int n)
{
    R s = 0;
    for (int i = threadIdx.x; i < n; i += 256) s += a[i];
    return s;
}

// The phase machine of every solve in the batch (end of a tick).
__global__ void __launch_bounds__(256)
scalars_kernel(const DevProblem* __restrict__ probs, const int* __restrict__ n_probs, double* __restrict__ evals)
{
    __shared__ double shd[8];
    __shared__ long long shi[8];
    const int np = *n_probs;
    for (int p = blockIdx.x; p < np; p += gridDim.x) {
        const DevProblem& P = probs[p];
        if (!P.st) continue;
        SolveState& S = *P.st;
        const SolveBufs& B = P.b;
        const int nvb = P.vis.n_gran, npb = P.pix.n_gran;
        const int ph = S.phase;
        __syncthreads();                       // every thread has read the phase
        // pairs the operator kernels of this tick evaluated for this problem
        // (the roles of fwd_role / adj_role in the tick's phase)
        if (evals && threadIdx.x == 0) {
            const double pairs = (double)P.vis.n * (double)P.pix.n;
            if (ph == PH_PINIT || ph == PH_POWER || ph == PH_SINIT || ph == PH_SOLVE) atomicAdd(&evals[0], pairs);
            if (ph == PH_POWER || ph == PH_SOLVE) atomicAdd(&evals[1], pairs);
        }
        // the mix kernel of the previous tick has run (stream order)
        if (threadIdx.x == 0) S.mix_pending = 0;
        if (ph == PH_PINIT) {
            if (threadIdx.x == 0) S.phase = PH_POWER;
        } else if (ph == PH_POWER) {
            const double z2 = cta_sum(strided<double>(B.blk_z2, npb), shd);
            const long long bad =
                cta_sum(strided<long long>(B.blk_badv, nvb) + strided<long long>(B.blk_badp, npb), shi);
            if (threadIdx.x == 0) {
                const double mu = sqrt(z2);
                S.pit += 1;
                if (bad || !isfinite(mu) || mu == 0.0) {
                    S.nonfinite = (bad || !isfinite(mu)) ? 1 : 0;
                    S.mu = mu;
                    S.phase = PH_DONE;
                } else {
                    const bool conv = (S.pit > 1 && fabs(mu - S.mu_prev) <= S.ptol * mu) || S.pit >= S.pmax;
                    S.mu = mu;
                    S.mu_prev = mu;
                    S.inv_mu = 1.0 / mu;
                    if (conv) {
                        S.L = mu;
                        S.phase = S.power_only ? PH_DONE : PH_SINIT;
                    }
                }
            }
        } else if (ph == PH_SINIT) {
            const double r2 = cta_sum(strided<double>(B.blk_r2, nvb), shd);
            const long long bad = cta_sum(strided<long long>(B.blk_badv, nvb), shi);
            if (threadIdx.x == 0) {
                S.resid2 = r2;
                S.E_prev = 0.5 * r2 + S.lambda * S.l1;
                S.E = S.E_prev;
                S.k = 0;
                S.t = 1.0;
                S.converged = 0;
                S.nonfinite = bad ? 1 : 0;
                S.phase = (S.max_iter <= 0 || bad) ? PH_DONE : PH_SOLVE;
            }
        } else if (ph == PH_SOLVE) {
            const double r2 = cta_sum(strided<double>(B.blk_r2, nvb), shd);
            const double l1 = cta_sum(strided<double>(B.blk_l1, npb), shd);
            const long long nnz = cta_sum(strided<long long>(B.blk_nnz, npb), shi);
            const long long bad =
                cta_sum(strided<long long>(B.blk_badv, nvb) + strided<long long>(B.blk_badp, npb), shi);
            if (threadIdx.x == 0 && S.algo) {
                // MFISTA: keep the better of z_k and x_{k-1}; then
                // y_{k+1} = x_k + (t_k/t_{k+1})(z_k - x_k) + ((t_k-1)/t_{k+1})(x_k - x_{k-1})
                //         = x_{k-1} + c (z_k - x_{k-1}), c = 1 + (t_k-1)/t_{k+1} when z_k
                // is kept, t_k/t_{k+1} when it is not (formed by the mix kernel).
                double tn, beta;
                fista_beta(S.t, tn, beta);
                const double Fz = 0.5 * r2 + S.lambda * l1;
                const double Fx = S.E_prev;
                const int take = Fz <= Fx;
                S.take = take;
                S.cmix = take ? 1.0 + beta : S.t / tn;
                S.mix_pending = 1;
                S.k += 1;
                S.t = tn;
                S.beta = beta;
                if (take) {
                    S.resid2 = r2;
                    S.l1 = l1;
                    S.nnz = nnz;
                    S.E = Fz;
                }
                bool done = false;
                if (bad || !isfinite(Fz)) {
                    S.nonfinite = 1;
                    done = true;
                }
                if (S.tol > 0.0 && fabs(Fz - Fx) <= S.tol * Fx) {
                    S.converged = 1;
                    done = true;
                }
                if (S.k >= S.max_iter) done = true;
                S.E_prev = S.E;
                if (done) S.phase = PH_DONE;
            } else if (threadIdx.x == 0) {
                double tn, beta;
                fista_beta(S.t, tn, beta);
                const double E = 0.5 * r2 + S.lambda * l1;
                S.k += 1;
                S.t = tn;
                S.beta = beta;
                S.resid2 = r2;
                S.l1 = l1;
                S.nnz = nnz;
                S.E = E;
                bool done = false;
                if (bad || !isfinite(E)) {
                    S.nonfinite = 1;
                    done = true;
                }
                if (S.tol > 0.0 && fabs(E - S.E_prev) <= S.tol * S.E_prev) {
                    S.converged = 1;
                    done = true;
                }
                if (S.k >= S.max_iter) done = true;
                S.E_prev = E;
                if (done) S.phase = PH_DONE;
            }
        }
    }
}

// ------------------------------------------------------------ MFISTA mix
// Finishes an MFISTA step once the scalars kernel has compared F(z_k) with
// F(x_{k-1}): grid-stride over the visibility blocks of the forward plan and
// then the pixel blocks of the adjoint plan,
//   visibilities: A y_{k+1} = A x_{k-1} + c (A z_k - A x_{k-1})   (linearity)
//                 r = W (A y_{k+1} - V);  A x_k = A z_k if z_k was kept
//   pixels:       y_{k+1} = x_{k-1} + c (z_k - x_{k-1});  x_k = z_k if kept
__global__ void __launch_bounds__(256)
mfista_mix_kernel(const DevProblem* __restrict__ probs, const Plan* __restrict__ fplp,
                  const Plan* __restrict__ aplp, int polar)
{
    const Plan fp = *fplp, ap = *aplp;
    for (int gb = blockIdx.x; gb < fp.n_blocks + ap.n_blocks; gb += gridDim.x) {
        const bool vis = gb < fp.n_blocks;
        const Plan& pl = vis ? fp : ap;
        const int g = vis ? gb : gb - fp.n_blocks;
        const int p = find_blk_prob(pl, g);
        const DevProblem& P = probs[p];
        if (!P.st || !P.st->algo || !P.st->mix_pending) continue;
        const double c = P.st->cmix;
        const int take = P.st->take;
        const int blk = g - pl.prob_b0[p];
        const SolveBufs& B = P.b;
        for (int i = threadIdx.x; i < pl.blk_el; i += 256) {
            const int e = blk * pl.blk_el + i;
            if (vis) {
                if (e >= P.vis.n_pad) continue;
                const double2 ax = B.AI[0][e], az = B.AI[1][e], V = P.V[e];
                const double W = P.vis.d[e].w;
                const double ayr = ax.x + c * (az.x - ax.x), ayi = ax.y + c * (az.y - ax.y);
                const double2 r = make_double2(W * (ayr - V.x), W * (ayi - V.y));
                B.r[e] = r;
                write_polar(P, polar, e, r);
                mark_huge(P.huge ? P.huge + 1 : nullptr, r);
                if (take) B.AI[0][e] = az;
            } else {
                if (e >= P.pix.n_pad) continue;
                const double x = B.I[0][e], z = B.I[1][e];
                B.y[e] = x + c * (z - x);
                if (take) B.I[0][e] = z;
            }
        }
    }
}

// Phase of every problem of a batch, for the host (one int per problem).
__global__ void phases_kernel(const DevProblem* __restrict__ probs, const int* __restrict__ n_probs,
                              int* __restrict__ out)
{
    const int np = *n_probs;
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < np; p += gridDim.x * blockDim.x)
        out[p] = probs[p].st ? probs[p].st->phase : PH_IDLE;
}

// Threads per element by the mean number of slots of a block (the kernels'
// loads are 8 deep): up to 2 slots one thread has them in flight anyway; above
// 96, 8 threads take a few rounds each.  (Between 48 and 96 slots CTAs of 256 threads start
// sooner behind another stream's operator: 3,001 Dirac pixels x 129,891 visibilities
// adjoint, 76 slots, three streams in turn: 135.9 us a call with 8 threads, 132.4
// with 4.)  16 of them made CTAs of 1,024 threads and 64 registers, which start
// only on an empty SM: behind another stream's operator they waited for whole SMs
// and kept its CTAs off them meanwhile (35,344 multiscale pixels x 2,702
// visibilities forward, three streams in turn: 163 us a call; 151 with 8, and a
// 30-tick FP64 solve 5.71 -> 5.69 ms).
static int slot_threads(const Plan& pl)
{
    const double mean = (double)pl.n_slots / (pl.n_blocks > 0 ? pl.n_blocks : 1);
    return mean <= 2.0 && pl.blk_el >= 256 ? 1 : mean <= 96.0 ? 4 : 8;
}
template <int SL>
static int fin_grid(const Plan& pl, int num_sms)
{
    const long long nq = (long long)pl.n_blocks * (pl.blk_el > FinShape<SL>::EL ? pl.blk_el / FinShape<SL>::EL : 1);
    const long long most = (long long)num_sms * (2048 / FinShape<SL>::THREADS);
    return (int)(nq < 1 ? 1 : nq < most ? nq : most);
}

cudaError_t launch_fwd_finish(const DevProblem* probs, const Plan* plp, const Plan& pl, int num_sms,
                              const double2* partial, int polar, double2* user_out, cudaStream_t st)
{
    switch (slot_threads(pl)) {
    case 1: fwd_finish_kernel<1><<<fin_grid<1>(pl, num_sms), 256, 0, st>>>(probs, plp, partial, polar, user_out); break;
    case 4: fwd_finish_kernel<4><<<fin_grid<4>(pl, num_sms), 256, 0, st>>>(probs, plp, partial, polar, user_out); break;
    default: fwd_finish_kernel<8><<<fin_grid<8>(pl, num_sms), 512, 0, st>>>(probs, plp, partial, polar, user_out);
    }
    return cudaGetLastError();
}

cudaError_t launch_adj_finish(const DevProblem* probs, const Plan* plp, const Plan& pl, int num_sms,
                              const double* partial, double* user_out, cudaStream_t st)
{
    switch (slot_threads(pl)) {
    case 1: adj_finish_kernel<1><<<fin_grid<1>(pl, num_sms), 256, 0, st>>>(probs, plp, partial, user_out); break;
    case 4: adj_finish_kernel<4><<<fin_grid<4>(pl, num_sms), 256, 0, st>>>(probs, plp, partial, user_out); break;
    default: adj_finish_kernel<8><<<fin_grid<8>(pl, num_sms), 512, 0, st>>>(probs, plp, partial, user_out);
    }
    return cudaGetLastError();
}

cudaError_t launch_mfista_mix(const DevProblem* probs, const Plan* fplp, const Plan* aplp, int grid, int polar,
                              cudaStream_t st)
{
    mfista_mix_kernel<<<grid, 256, 0, st>>>(probs, fplp, aplp, polar);
    return cudaGetLastError();
}

cudaError_t launch_scalars(const DevProblem* probs, const int* n_probs, int grid, double* evals, cudaStream_t st)
{
    scalars_kernel<<<grid, 256, 0, st>>>(probs, n_probs, evals);
    return cudaGetLastError();
}

cudaError_t launch_phases(const DevProblem* probs, const int* n_probs, int grid, int* out, cudaStream_t st)
{
    phases_kernel<<<grid, 128, 0, st>>>(probs, n_probs, out);
    return cudaGetLastError();
}

}  // namespace sl1m
