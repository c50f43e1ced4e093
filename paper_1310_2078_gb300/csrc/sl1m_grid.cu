// sl1m_grid.cu -- the operator of Dirac pixels on a regular (l, m) lattice by
// gridding and FFT (Hardy 2013, Eq. sme with the entries of Eq. deltam).
//
//   V_k = sum_j (x_j / n_j) exp(-2 pi i (u_k l_j + v_k m_j + w_k (n_j - 1)))
//
// With l_j = lc + s dl and m_j = mc + t dm for integers s, t, the dependence on
// u and v is a Fourier series in s and t sampled off its grid, and that on w
// is a Fourier integral over nu = n - 1 - nc, |nu| <= B.  Both are evaluated
// by the same device (Dutt & Rokhlin 1993; the kernel is the "exponential of
// semicircle" of Barnett, Magland & af Klinteberg 2019): a function of bounded
// support sampled at twice its band is interpolated by a kernel phi of 8
// samples, once the other side has been divided by phi's transform.  So
//
//   forward   for every plane w_p: z_st = x amp exp(-2 pi i w_p nu), rows then
//             columns transformed (zero-padded to 2^lx, 2^ly), and each V_k
//             gathered from 8 x 8 cells of 8 planes;
//   adjoint   the transpose: r spread onto the planes, columns and rows
//             transformed back, Re(exp(+2 pi i w_p nu) z) summed over the planes.
//
// x is real, so V at (-u, -v, -w) is the conjugate of V at (u, v, w): the
// visibilities with w < 0 are taken at the mirrored point, and the planes cover
// only 0 .. max |w|.  Tiles of a plane that no visibility touches are neither
// written nor read, and columns without such a tile are not transformed.
//
// The interpolation error is 1e-7 of the result's norm and the whole operator
// in FP32 is 1.6e-7 to 2.8e-7 off FP64 (2-norm, sizes below and others),
// where evaluating every pair with the SFU's sine and cosine (sl1m_mixed.cu) is
// 3.6e-7 to 4.9e-7 off.  The work no longer grows with N_v N_p but with the
// planes' cells: per plane the kernels move up to (3 2^ly + 2 ny) 2^lx complex
// numbers.  Measured on GB300 against the pair kernels: 1024^2 pixels x 406,400
// visibilities (55 planes of 2048^2) forward 202.9 -> 0.99 ms, adjoint 141.7 ->
// 1.13 ms; 256^2 over +/-0.5 x 40,320 (273 planes of 512^2) 1.19 -> 0.25 ms and
// 0.85 -> 0.32 ms.  The planes' traffic alone would take 0.35 ms at paper scale
// (2.3 GB at the 6.7 TB/s of a copy) and 0.14 ms on the wide field.
#include <algorithm>

#include "sl1m_devfn.cuh"
#include "sl1m_grid.h"

namespace sl1m {

// ---------------------------------------------------------------- transforms

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b)
{
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
// SGN i a
template <int SGN>
__device__ __forceinline__ float2 crot(float2 a)
{
    return SGN < 0 ? make_float2(a.y, -a.x) : make_float2(-a.y, a.x);
}

template <int SGN>
__device__ __forceinline__ void dft4(float2& a0, float2& a1, float2& a2, float2& a3)
{
    const float2 s0 = cadd(a0, a2), s1 = csub(a0, a2), s2 = cadd(a1, a3), s3 = crot<SGN>(csub(a1, a3));
    a0 = cadd(s0, s2);
    a1 = cadd(s1, s3);
    a2 = csub(s0, s2);
    a3 = csub(s1, s3);
}

// Half-zero inputs: with the cells at elements [0, L/4) and [3L/4, L) of a
// transform (2^lx >= 2 nx, the origin in the middle), the middle half of the P
// elements that a thread holds are zero, and of its outputs only the outer
// quarters are cells.  PIN: the inputs are such; POUT: only those outputs are wanted.

// dft4 with the middle inputs zero.
template <int SGN>
__device__ __forceinline__ void dft4_outer(float2& a0, float2& a1, float2& a2, float2& a3)
{
    const float2 p = a0, q = a3, r = crot<SGN>(q);
    a0 = cadd(p, q);
    a1 = csub(p, r);
    a2 = csub(p, q);
    a3 = cadd(p, r);
}
// a e^{SGN 2 pi i M / 16}
template <int SGN, int M>
__device__ __forceinline__ float2 rot16(float2 a)
{
    constexpr float H = 0.70710678118654752f, C = 0.92387953251128676f, S = 0.38268343236508977f;
    if constexpr (M >= 8) {
        const float2 b = rot16<SGN, M - 8>(a);
        return make_float2(-b.x, -b.y);
    } else if constexpr (M >= 4) {
        return crot<SGN>(rot16<SGN, M - 4>(a));
    } else if constexpr (M == 0) {
        return a;
    } else if constexpr (M == 2) {
        const float2 b = crot<SGN>(a);
        return make_float2((a.x + b.x) * H, (a.y + b.y) * H);
    } else {
        return cmul(a, make_float2(M == 1 ? C : S, SGN * (M == 1 ? S : C)));
    }
}

// Transforms of 8 and 16 elements in place, as 2 x 4 and 4 x 4.
template <int SGN, bool PIN, bool POUT>
__device__ __forceinline__ void dft8(float2& v0, float2& v1, float2& v2, float2& v3, float2& v4, float2& v5,
                                     float2& v6, float2& v7)
{
    if (PIN) {
        dft4_outer<SGN>(v0, v2, v4, v6);
        dft4_outer<SGN>(v1, v3, v5, v7);
    } else {
        dft4<SGN>(v0, v2, v4, v6);            // even inputs: e0..e3 in v0, v2, v4, v6
        dft4<SGN>(v1, v3, v5, v7);            // odd inputs
    }
    const float2 o0 = v1, o1 = rot16<SGN, 2>(v3), o2 = rot16<SGN, 4>(v5), o3 = rot16<SGN, 6>(v7);
    const float2 e0 = v0, e1 = v2, e2 = v4, e3 = v6;
    v0 = cadd(e0, o0);
    v1 = cadd(e1, o1);
    if (!POUT) {
        v2 = cadd(e2, o2);
        v3 = cadd(e3, o3);
        v4 = csub(e0, o0);
        v5 = csub(e1, o1);
    }
    v6 = csub(e2, o2);
    v7 = csub(e3, o3);
}
// One second-stage transform of dft16: outputs K, K + 4, K + 8, K + 12.
template <int SGN, int K, bool POUT>
__device__ __forceinline__ void dft16_tail(const float2 (&t)[16], float2 (&v)[16])
{
    const float2 a0 = t[4 * K], a1 = rot16<SGN, K>(t[4 * K + 1]), a2 = rot16<SGN, 2 * K>(t[4 * K + 2]),
                 a3 = rot16<SGN, 3 * K>(t[4 * K + 3]);
    const float2 s0 = cadd(a0, a2), s1 = csub(a0, a2), s2 = cadd(a1, a3), s3 = crot<SGN>(csub(a1, a3));
    v[K] = cadd(s0, s2);
    if (!POUT) {
        v[K + 4] = cadd(s1, s3);
        v[K + 8] = csub(s0, s2);
    }
    v[K + 12] = csub(s1, s3);
}
template <int SGN, bool PIN, bool POUT>
__device__ __forceinline__ void dft16(float2 (&v)[16])
{
    float2 t[16];                             // t[4 k + a]: output k of the transform of v[a], v[a + 4], ..
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        float2 x0 = v[a], x1 = v[a + 4], x2 = v[a + 8], x3 = v[a + 12];
        if (PIN) dft4_outer<SGN>(x0, x1, x2, x3);
        else dft4<SGN>(x0, x1, x2, x3);
        t[a] = x0;
        t[4 + a] = x1;
        t[8 + a] = x2;
        t[12 + a] = x3;
    }
    dft16_tail<SGN, 0, POUT>(t, v);
    dft16_tail<SGN, 1, POUT>(t, v);
    dft16_tail<SGN, 2, POUT>(t, v);
    dft16_tail<SGN, 3, POUT>(t, v);
}

template <int SGN, bool PIN, bool POUT>
__device__ __forceinline__ void dft_all(float2 (&v)[16])
{
    dft16<SGN, PIN, POUT>(v);
}
template <int SGN, bool PIN, bool POUT>
__device__ __forceinline__ void dft_all(float2 (&v)[8])
{
    dft8<SGN, PIN, POUT>(v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7]);
}

// Shared-memory place of element i = e CB + c (element e of transform c of CB
// interleaved ones): its low four bits (the 16 float2 that one wavefront of
// shared memory holds) are XORed with its next four, or with sums of them, so
// that the 16 lanes of a half warp hit 16 different places in every access
// pattern of the passes below: unit stride, strides of 2, 4, 8 and 16 elements,
// and runs of 2, 4 or 8 elements 32, 64 or 128 (radix 8: 64) apart.  (A pad of one element
// per 8 instead cost the unit-stride reads a second wavefront.)  The map is
// linear over GF(2): place(e | d) = place(e) ^ place(d) for e and d without
// common bits, and d is always a constant.
template <int CB>
__host__ __device__ __forceinline__ constexpr int place(int i)
{
    return i ^ (CB == 1   ? ((i >> 4) ^ ((i >> 3) & 8)) & 15
                : CB == 4 ? ((i >> 4) ^ (i >> 6)) << 2 & 12
                          : ((i >> 4) ^ (i >> 5) ^ (i >> 6) ^ (i >> 7)) << 3 & 8);
}
template <int CB>
__device__ __forceinline__ float2& elem(float2* sm, int at, int d)     // at = place(e CB + c)
{
    const int pd = place<CB>(d * CB);
    return sm[(at ^ (pd & 15)) + (pd & ~15)];
}

template <int LOG>
struct FftShape {
    static constexpr int P = grid_radix(LOG), R0 = grid_radix0(LOG);
};

// Transform of length 2^LOG, radix P = 8 or 16 (grid_radix) after a first pass
// of radix 2, 4, 8 or 16 (Stockham order: no bit reversal).  A thread holds NB
// groups of P elements: on entry and on exit vs[n][q] is element gs[n] + q 2^LOG/P
// of its transform.  Every thread of the CTA calls it; sm holds the CTA's CB
// interleaved transforms, c is this thread's.  PP: sm is two buffers of PP
// elements used in turn (one barrier per exchange instead of two); sm is left at
// the next one to write.  Twiddles: per pass of stride ns, e^{-2 pi i k/(P ns)}
// and its 2nd, 4th (and 8th) powers for k < ns, rounded from FP64; the others are
// products of these.
//
// The transforms are bound by their exchanges (issue slots and barriers of passes
// that each move every element through shared memory and back; the memory they
// stream is a third of the time), so the radix is the one with fewer of them:
// 2^11 takes 2 with radix 16 and 3 with radix 8.  Radix 16 against 8 at the same
// threads' load, 55 planes of 2048^2: forward 1.017 -> 0.985 ms, adjoint 1.203 ->
// 1.129 ms, and a 31-operator solve of 15 planes 10.4 -> 9.8 ms.  2^6 and 2^9 take
// as many with radix 8 and are faster with it: 273 planes of 512^2 forward 0.25
// against 0.28 ms, adjoint 0.31 against 0.33 ms.  Also slower: two planes or two
// columns to a thread as float4 (twice the registers, half the warps: 1.18 -> 1.41
// ms), and leaving out the forward's writes of columns nobody reads (a test per
// element; 1.02 against 0.985 ms, although a third less is written).
template <int LOG, int SGN, int CB, int NB, bool PIN, bool POUT, int PP>
__device__ __forceinline__ void fft_pass_all(float2 (&vs)[NB][FftShape<LOG>::P], const int (&gs)[NB], int c,
                                             float2*& sm, int& par, const float2* __restrict__ tw)
{
    constexpr int P = FftShape<LOG>::P, R0 = FftShape<LOG>::R0, L = 1 << LOG, E = L / P;
#pragma unroll
    for (int n = 0; n < NB; ++n) {
        float2 (&v)[P] = vs[n];
        if constexpr (R0 == P) {
            dft_all<SGN, PIN, false>(v);
        } else if constexpr (R0 == 8) {
#pragma unroll
            for (int i = 0; i < 2; ++i)
                dft8<SGN, PIN, false>(v[i], v[i + 2], v[i + 4], v[i + 6], v[i + 8], v[i + 10], v[i + 12], v[i + 14]);
        } else if constexpr (R0 == 4) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (PIN) dft4_outer<SGN>(v[i], v[i + 4], v[i + 8], v[i + 12]);
                else dft4<SGN>(v[i], v[i + 4], v[i + 8], v[i + 12]);
            }
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float2 a = v[i], b = v[i + 8];
                v[i] = !PIN ? cadd(a, b) : i < 4 ? a : b;
                v[i + 8] = !PIN ? csub(a, b) : i < 4 ? a : make_float2(-b.x, -b.y);
            }
        }
        const int at = place<CB>(gs[n] * R0 * CB + c);        // output r of the i-th transform is v[i + r P/R0]
#pragma unroll
        for (int i = 0; i < P / R0; ++i)
#pragma unroll
            for (int r = 0; r < R0; ++r) elem<CB>(sm, at, i * E * R0 + r) = v[i + r * (P / R0)];
    }
#pragma unroll
    for (int ns = R0; ns < L; ns *= P) {
        __syncthreads();
#pragma unroll
        for (int n = 0; n < NB; ++n) {
            const int at = place<CB>(gs[n] * CB + c);
#pragma unroll
            for (int r = 0; r < P; ++r) vs[n][r] = elem<CB>(sm, at, r * E);
        }
        if (PP) {
            sm += par ? -PP : PP;
            par ^= 1;
        } else {
            __syncthreads();
        }
#pragma unroll
        for (int n = 0; n < NB; ++n) {
            float2 (&v)[P] = vs[n];
            const int k = gs[n] & (ns - 1);
            float2 w1 = __ldg(tw + k), w2 = __ldg(tw + ns + k), w4 = __ldg(tw + 2 * ns + k);
            if (SGN > 0) {
                w1.y = -w1.y;
                w2.y = -w2.y;
                w4.y = -w4.y;
            }
            const float2 w3 = cmul(w1, w2);
            if constexpr (P == 16) {
                float2 w8 = __ldg(tw + 3 * ns + k);
                if (SGN > 0) w8.y = -w8.y;
                const float2 w12 = cmul(w8, w4);
                v[8] = cmul(v[8], w8);
                v[9] = cmul(v[9], cmul(w8, w1));
                v[10] = cmul(v[10], cmul(w8, w2));
                v[11] = cmul(v[11], cmul(w8, w3));
                v[12] = cmul(v[12], w12);
                v[13] = cmul(v[13], cmul(w12, w1));
                v[14] = cmul(v[14], cmul(w12, w2));
                v[15] = cmul(v[15], cmul(w12, w3));
            }
            v[1] = cmul(v[1], w1);
            v[2] = cmul(v[2], w2);
            v[3] = cmul(v[3], w3);
            v[4] = cmul(v[4], w4);
            v[5] = cmul(v[5], cmul(w4, w1));
            v[6] = cmul(v[6], cmul(w4, w2));
            v[7] = cmul(v[7], cmul(w4, w3));
            if (ns * P < L) {
                dft_all<SGN, false, false>(v);
                const int at = place<CB>(((gs[n] - k) * P + k) * CB + c);
#pragma unroll
                for (int r = 0; r < P; ++r) elem<CB>(sm, at, r * ns) = v[r];
            } else {
                dft_all<SGN, false, POUT>(v);
            }
        }
        tw += (P == 16 ? 4 : 3) * ns;
    }
}

// The elements q of a thread's P that are cells.
template <int P>
__device__ __forceinline__ constexpr int cell_q(int i)
{
    return i < P / 4 ? i : i + P / 2;
}

// Cell index of element e (0 <= e < 2^lg) of a zero-padded axis whose cell c0
// sits at element 0; outside [0, n) where the padding is.
__device__ __forceinline__ int cell_of(int e, int lg, int c0)
{
    return (e < (1 << (lg - 1)) ? e : e - (1 << lg)) + c0;
}

// The scale of an operator's input (which: 0 forward, 1 adjoint; both marks are
// read at once, a chain of loads less).
__device__ __forceinline__ float in_scale(const DevProblem& P, int which, float huge_scale)
{
    const int now = P.huge[which], first = which == 0 ? P.huge[2] : 0;
    const bool init = which == 0 && P.st && P.st->phase == PH_SINIT;
    return (init ? first : now) ? huge_scale : GR_SCALE;
}

// exp(-2 pi i w nu) with both factors split in FP32 halves.
__device__ __forceinline__ float2 plane_phase(float2 w, float2 nu)
{
    const float f = frac_turns(tp_frac(w.x, w.y, nu.x, nu.y));
    float s, c;
    sincospif(2.0f * f, &s, &c);
    return make_float2(c, -s);
}

template <int LOG>
struct RowShape {
    static constexpr int P = grid_radix(LOG);                 // elements per thread
    static constexpr int T = (1 << LOG) / P;                  // threads per row
    static constexpr int WIDE = P == 16 ? 128 : 256;
    static constexpr int ROWS = T >= WIDE ? 1 : WIDE / T;     // rows per CTA
    static constexpr int CTAS = LOG == 12 ? 2 : P == 16 ? 5 : 3;
    static constexpr int THREADS = T * ROWS;
    static constexpr int BUF = ROWS << LOG;                   // shared elements of one buffer
    static constexpr int SMEM = 2 * BUF * (int)sizeof(float2);
};

// Forward, rows: z = x amp exp(-2 pi i w_p nu) along x, transformed, into g1.
// A CTA takes ROWS lattice rows of GR_PCH planes: x, amp and nu are read once
// for them.
template <int LOG>
__global__ void __launch_bounds__(RowShape<LOG>::THREADS, RowShape<LOG>::CTAS)
grid_rows_fwd_kernel(const DevProblem* __restrict__ probs, int prob, const GridOp g, int p0, int np)
{
    using S = RowShape<LOG>;
    constexpr int L = 1 << LOG;
    extern __shared__ __align__(16) float2 sm_rows[];         // two buffers of BUF
    const double* X;
    if (!fwd_role(probs[prob], X)) return;
    const int rb = threadIdx.x / S::T;
    const int gi[1] = {(int)threadIdx.x % S::T};
    const int iy = blockIdx.x * S::ROWS + rb;
    const float scale = in_scale(probs[prob], 0, g.fscale);
    float a[S::P / 2];
    float2 nu[S::P / 2];
#pragma unroll
    for (int i = 0; i < S::P / 2; ++i) {
        const int ix = cell_of(gi[0] + cell_q<S::P>(i) * S::T, LOG, g.cx);
        a[i] = 0.f;
        nu[i] = make_float2(0.f, 0.f);
        if (iy < g.ny && ix >= 0 && ix < g.nx) {
            const size_t at = (size_t)iy * g.nx + ix;
            const int j = g.cell[at];
            if (j >= 0) {
                a[i] = __double2float_rn(X[j]) * scale * g.amp[at];
                nu[i] = g.nu[at];
            }
        }
    }
    float2* smr = sm_rows + rb * L;
    int par = 0;
    const int q1 = min(np, (int)(blockIdx.y + 1) * GR_PCH);
    for (int p = blockIdx.y * GR_PCH; p < q1; ++p) {
        const float2 w = g.wp[p0 + p];
        float2 v[1][S::P];
#pragma unroll
        for (int i = 0; i < S::P / 2; ++i) {
            const float2 e = plane_phase(w, nu[i]);
            v[0][cell_q<S::P>(i)] = make_float2(a[i] * e.x, a[i] * e.y);
        }
        fft_pass_all<LOG, -1, 1, 1, true, false, S::BUF>(v, gi, 0, smr, par, g.twx);
        if (iy < g.ny) {
            float2* dst = g.g1 + ((size_t)p * g.ny + iy) * L;
#pragma unroll
            for (int q = 0; q < S::P; ++q) dst[gi[0] + q * S::T] = v[0][q];
        }
    }
}

// Adjoint, rows: g1 transformed back along x; Re(exp(+2 pi i w_p nu) z) summed
// over the CTA's planes (FP32 over GR_PCH planes) into the chunk's partial slots,
// which a later pass over the planes adds to.
template <int LOG>
__global__ void __launch_bounds__(RowShape<LOG>::THREADS, RowShape<LOG>::CTAS)
grid_rows_adj_kernel(const DevProblem* __restrict__ probs, int prob, const GridOp g, int p0, int np, int n_pix,
                     int n_pix_pad, double* __restrict__ partial)
{
    using S = RowShape<LOG>;
    constexpr int L = 1 << LOG;
    extern __shared__ __align__(16) float2 sm_rows[];         // two buffers of BUF
    const double2* R;
    if (!adj_role(probs[prob], R)) return;
    const int rb = threadIdx.x / S::T;
    const int gi[1] = {(int)threadIdx.x % S::T};
    const int iy = blockIdx.x * S::ROWS + rb;
    const float unscale = __frcp_rn(in_scale(probs[prob], 1, g.ascale));     // (a power of two)
    float acc[S::P / 2];
    float2 nu[S::P / 2];
#pragma unroll
    for (int i = 0; i < S::P / 2; ++i) {
        const int ix = cell_of(gi[0] + cell_q<S::P>(i) * S::T, LOG, g.cx);
        acc[i] = 0.f;
        nu[i] = (iy < g.ny && ix >= 0 && ix < g.nx) ? g.nu[(size_t)iy * g.nx + ix] : make_float2(0.f, 0.f);
    }
    float2* smr = sm_rows + rb * L;
    int par = 0;
    const int q1 = min(np, (int)(blockIdx.y + 1) * GR_PCH);
    for (int p = blockIdx.y * GR_PCH; p < q1; ++p) {
        const float2 w = g.wp[p0 + p];
        float2 v[1][S::P];
        const float2* src = g.g1 + ((size_t)p * g.ny + min(iy, g.ny - 1)) * L;
        const unsigned char* act = g.colact + (size_t)(p0 + p) * (L / GR_TILE);
#pragma unroll
        for (int q = 0; q < S::P; ++q) {          // columns without a visibility were not written
            const int e = gi[0] + q * S::T;
            v[0][q] = act[e / GR_TILE] ? src[e] : make_float2(0.f, 0.f);
        }
        fft_pass_all<LOG, 1, 1, 1, false, true, S::BUF>(v, gi, 0, smr, par, g.twx);
#pragma unroll
        for (int i = 0; i < S::P / 2; ++i) {
            const float2 e = plane_phase(w, nu[i]);                  // conj(e) z, real part
            acc[i] += fmaf(e.x, v[0][cell_q<S::P>(i)].x, e.y * v[0][cell_q<S::P>(i)].y);
        }
    }
    if (iy < g.ny) {
#pragma unroll
        for (int i = 0; i < S::P / 2; ++i) {
            const int ix = cell_of(gi[0] + cell_q<S::P>(i) * S::T, LOG, g.cx);
            if (ix < 0 || ix >= g.nx) continue;
            const size_t at = (size_t)iy * g.nx + ix;
            const int j = g.cell[at];
            if (j >= 0) {
                double& slot = partial[((size_t)(j / BLK) * g.n_chunk + blockIdx.y) * BLK + j % BLK];
                const double v = (double)acc[i] * ((double)g.amp[at] * (double)unscale);
                slot = p0 > 0 ? slot + v : v;
            }
        }
    }
    if (blockIdx.x == 0)                       // padding slots of the last pixel granule
        for (int j = n_pix + threadIdx.x; j < n_pix_pad; j += S::THREADS)
            partial[((size_t)(j / BLK) * g.n_chunk + blockIdx.y) * BLK + j % BLK] = 0.0;
}

// Columns: CB adjacent columns of one plane per CTA, so a row of the tile is
// 8 CB contiguous bytes.  Forward (SGN -1): the ny rows of g1, zero-padded,
// into the 2^LOG rows of g2; adjoint (SGN +1): g2 back, its ny lattice rows
// into g1.
template <int LOG>
struct ColShape {
    static constexpr int P = grid_radix(LOG);
    static constexpr int CB = LOG >= 11 ? 4 : 8;
    static constexpr int NB = 16 / P;                         // 16 elements per thread
    static constexpr int THREADS = CB * (1 << LOG) / 16;
    static constexpr int SMEM = CB * (1 << LOG) * (int)sizeof(float2);
};
template <int LOG, int SGN>
__global__ void __launch_bounds__(ColShape<LOG>::THREADS, ColShape<LOG>::THREADS >= 512 && LOG < 12 ? 2 : 1)
grid_cols_kernel(const DevProblem* __restrict__ probs, int prob, const GridOp g, int p0)
{
    using S = ColShape<LOG>;
    constexpr int P = S::P, E = (1 << LOG) / P;
    extern __shared__ __align__(16) float2 sm_cols[];
    __shared__ unsigned char s_act[(1 << LOG) / GR_TILE];      // tiles of these columns with a visibility
    if (SGN < 0) {
        const double* X;
        if (!fwd_role(probs[prob], X)) return;
    } else {
        const double2* R;
        if (!adj_role(probs[prob], R)) return;
    }
    {
        const int ty = (1 << LOG) / GR_TILE;
        const unsigned char* act = g.act + ((size_t)(p0 + blockIdx.y) * ((1 << g.lx) / GR_TILE) +
                                            blockIdx.x * S::CB / GR_TILE) * ty;
        int any = 0;
        for (int t = threadIdx.x; t < ty; t += S::THREADS) any |= (s_act[t] = act[t]);
        if (!__syncthreads_or(any)) return;
    }
    const int c = threadIdx.x % S::CB;
    int gi[S::NB];
#pragma unroll
    for (int n = 0; n < S::NB; ++n) gi[n] = threadIdx.x / S::CB + n * (E / S::NB);
    const size_t col = (size_t)blockIdx.x * S::CB + c, Lx = (size_t)1 << g.lx;
    float2* g1 = g.g1 + (size_t)blockIdx.y * g.ny * Lx + col;
    float2* g2 = g.g2 + ((size_t)blockIdx.y << LOG) * Lx + col;
    float2 v[S::NB][P];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int n = i / P, q = i % P;
        const int e = gi[n] + q * E;
        if (SGN > 0) {
            v[n][q] = s_act[e / GR_TILE] ? g2[(size_t)e * Lx] : make_float2(0.f, 0.f);
        } else if (q < P / 4 || q >= 3 * P / 4) {
            const int iy = cell_of(e, LOG, g.cy);
            v[n][q] = (iy >= 0 && iy < g.ny) ? g1[(size_t)iy * Lx] : make_float2(0.f, 0.f);
        }
    }
    float2* sm = sm_cols;
    int par = 0;
    fft_pass_all<LOG, SGN, S::CB, S::NB, (SGN < 0), (SGN > 0), 0>(v, gi, c, sm, par, g.twy);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int n = i / P, q = i % P;
        const int e = gi[n] + q * E;
        if (SGN < 0) {
            if (s_act[e / GR_TILE]) g2[(size_t)e * Lx] = v[n][q];
        } else if (q < P / 4 || q >= 3 * P / 4) {
            const int iy = cell_of(e, LOG, g.cy);
            if (iy >= 0 && iy < g.ny) g1[(size_t)iy * Lx] = v[n][q];
        }
    }
}

// ------------------------------------------------- gathering and spreading

// Forward: each visibility from its 8 x 8 cells of 8 planes, one warp per
// visibility (lane = 8 cells in x by 4 rows, twice): a plane's share is 8
// segments of 64 bytes.  Visibilities are taken by tile and first plane, so the
// warps of a CTA find each other's cells in L1.  ALL: one pass holds every
// plane, so the 16 loads of a lane need no test and are in flight together.
template <bool ALL>
__global__ void __launch_bounds__(256, 4)
grid_gather_kernel(const DevProblem* __restrict__ probs, int prob, const GridOp g, int p0, int np, int n_vis_pad,
                   double2* __restrict__ partial)
{
    const double* X;
    if (!fwd_role(probs[prob], X)) return;
    const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (i >= n_vis_pad) return;
    const int k = g.order[i];
    const float unscale = __frcp_rn(in_scale(probs[prob], 0, g.fscale));     // (a power of two)
    const int4 ps = g.pos[k];
    if (!ALL && (ps.z >= p0 + np || ps.z + GRW <= p0) && p0 > 0) return;     // nothing to add
    const float* wt = g.wts + (size_t)k * (3 * GRW);
    const int tx = lane & 7, ty = lane >> 3;
    const int Lx = 1 << g.lx, Ly = 1 << g.ly;
    const int x = (ps.x + tx) & (Lx - 1);
    const size_t y0 = (size_t)((ps.y + ty) & (Ly - 1)) * Lx + x, y1 = (size_t)((ps.y + ty + 4) & (Ly - 1)) * Lx + x;
    const size_t plane = (size_t)Ly * Lx;
    const float2* pl = g.g2 + (size_t)(ALL ? ps.z : 0) * plane;
    float2 a[GRW], b[GRW];
#pragma unroll
    for (int t = 0; t < GRW; ++t) {
        if (ALL) {
            a[t] = pl[t * plane + y0];
            b[t] = pl[t * plane + y1];
        } else {
            const int p = ps.z + t - p0;
            const bool in = p >= 0 && p < np;
            a[t] = in ? pl[p * plane + y0] : make_float2(0.f, 0.f);
            b[t] = in ? pl[p * plane + y1] : make_float2(0.f, 0.f);
        }
    }
    const float wx = wt[tx], wy0 = wt[GRW + ty], wy1 = wt[GRW + ty + 4];
    const float4 wa = *reinterpret_cast<const float4*>(wt + 2 * GRW), wb = *reinterpret_cast<const float4*>(wt + 2 * GRW + 4);
    const float ww[GRW] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
    float2 s0 = make_float2(0.f, 0.f), s1 = s0;
#pragma unroll
    for (int t = 0; t < GRW; ++t) {
        s0.x = fmaf(ww[t], a[t].x, s0.x);
        s0.y = fmaf(ww[t], a[t].y, s0.y);
        s1.x = fmaf(ww[t], b[t].x, s1.x);
        s1.y = fmaf(ww[t], b[t].y, s1.y);
    }
    float sr = wx * fmaf(wy0, s0.x, wy1 * s1.x), si = wx * fmaf(wy0, s0.y, wy1 * s1.y);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        sr += __shfl_xor_sync(0xffffffffu, sr, o);
        si += __shfl_xor_sync(0xffffffffu, si, o);
    }
    if (lane == 0) {
        const float2 e = g.rot[k];
        const double inv = (double)unscale;
        double2 v = make_double2((double)fmaf(e.x, sr, -e.y * si) * inv, (double)fmaf(e.x, si, e.y * sr) * inv);
        if (ps.w) v.y = -v.y;                  // taken at the mirrored point
        if (!ALL && p0 > 0) {                  // a later pass over the planes
            const double2 o = partial[k];
            v.x += o.x;
            v.y += o.y;
        }
        partial[k] = v;
    }
}

constexpr int GR_SEG = GR_TILE * GR_TILE;      // planes of a spreading segment at most

// Adjoint: a CTA owns the GR_TILE^2 cells (one per thread) of a tile and walks
// the visibilities that touch it in the order of their first plane, with a ring
// of 8 accumulators per cell, the planes the current point reaches: once the
// points move on to a later first plane, the planes left behind are complete
// and are written.  So every point is visited once per tile, no atomics are
// needed and the sums are the same every time.  A warp (8 x 4 cells) visits
// only the points that meet it.  Points are staged 32 at a time, the next ones
// loaded while the current ones are added (a CTA has few, and each is two
// dependent loads away).  blockIdx.y cuts the planes into segments of
// seg_planes; a point that reaches into two segments is visited in both.
__global__ void __launch_bounds__(GR_TILE * GR_TILE, 4)
grid_spread_kernel(const DevProblem* __restrict__ probs, int prob, const GridOp g, int p0, int np, int seg_planes)
{
    constexpr int PB = 32;                     // points staged at a time, by 8 threads each
    __shared__ float4 s_pt[2][PB];             // {Re, Im of conj(rot) r, first x, first y}
    __shared__ __align__(16) float s_wx[2][PB][GRW], s_wy[2][PB][GRW], s_ww[2][PB][GRW];
    __shared__ int s_ip[2][PB];
    __shared__ unsigned char s_act[GR_SEG];    // planes of the segment that have to be written
    const double2* R;
    if (!adj_role(probs[prob], R)) return;
    const int Lx = 1 << g.lx, Ly = 1 << g.ly, tiles_x = Lx / GR_TILE;
    const int tile = blockIdx.x;
    const int ta = p0 + blockIdx.y * seg_planes, tb = min(ta + seg_planes, p0 + np);   // planes [ta, tb)
    const int ni = g.np - GRW + 1;             // values of a first plane
    const int* st = g.start + (size_t)tile * (ni + 1);
    const int b0 = st[max(0, min(ni, ta - GRW + 1))], b1 = st[max(0, min(ni, tb))];
    if (b0 >= b1) return;                      // no plane of the segment is touched here
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wx0 = (tile % tiles_x) * GR_TILE + (warp & 1) * 8, wy0 = (tile / tiles_x) * GR_TILE + (warp >> 1) * 4;
    const int x = wx0 + (lane & 7), y = wy0 + (lane >> 3);
    const size_t plane = (size_t)Ly * Lx;
    float2* const cell = g.g2 + (size_t)y * Lx + x;
    if ((int)threadIdx.x < tb - ta)            // (read after the loop's first barrier)
        s_act[threadIdx.x] = g.act[((size_t)(ta + threadIdx.x) * tiles_x + tile % tiles_x) * (Ly / GR_TILE) + tile / tiles_x];
    // this thread's part of the staging: point si, weights sf of each axis
    const int si = threadIdx.x >> 3, sf = threadIdx.x & 7;
    const float scale = in_scale(probs[prob], 1, g.ascale);
    float lwx = 0.f, lwy = 0.f, lww = 0.f;
    float4 lpt = make_float4(0.f, 0.f, 0.f, 0.f);
    int lip = 0;
    const auto fetch = [&](int b) {
        if (b + si >= b1) return;
        const int k = g.list[b + si];
        const float* wt = g.wts + (size_t)k * (3 * GRW);
        lwx = wt[sf];
        lwy = wt[GRW + sf];
        lww = wt[2 * GRW + sf];
        const int4 ps = g.pos[k];
        lip = ps.z;
        if (sf == 0) {
            const float2 o = g.rot[k];
            const double2 r = R[k];
            const float rr = (float)r.x * scale, ri = (float)(ps.w ? -r.y : r.y) * scale;
            lpt = make_float4(fmaf(o.x, rr, o.y * ri), fmaf(o.x, ri, -o.y * rr), __int_as_float(ps.x),
                              __int_as_float(ps.y));
        }
    };
    // acc[p mod 8] is plane p of [cur, cur + 8); the staged weights in w are
    // rotated to match, so the ring turns without moving a register
    float2 acc[GRW];
#pragma unroll
    for (int q = 0; q < GRW; ++q) acc[q] = make_float2(0.f, 0.f);
    int cur = max(0, ta - GRW + 1);
    const auto put = [&](int p, float2 v) {
        if (p >= ta && p < tb && s_act[p - ta]) cell[(size_t)(p - p0) * plane] = v;
    };
    // planes [cur, to) are complete
    const auto advance = [&](int to) {
        if (cur >= to) return;
        const int n = to - cur;
#pragma unroll
        for (int q = 0; q < GRW; ++q) {
            const int d = (q - cur) & (GRW - 1);           // acc[q] is plane cur + d
            if (d < n) {
                put(cur + d, acc[q]);
                acc[q] = make_float2(0.f, 0.f);
            }
        }
        for (int p = cur + GRW; p < to; ++p) put(p, make_float2(0.f, 0.f));
        cur = to;
    };
    fetch(b0);
    int buf = 0;
    for (int b = b0; b < b1; b += PB, buf ^= 1) {
        const int n = min(PB, b1 - b);
        s_wx[buf][si][sf] = lwx;
        s_wy[buf][si][sf] = lwy;
        s_ww[buf][si][(sf + lip) & (GRW - 1)] = lww;       // by plane mod 8
        if (sf == 0) {
            s_pt[buf][si] = lpt;
            s_ip[buf][si] = lip;
        }
        __syncthreads();                       // (the other buffer's readers are done, too)
        fetch(b + PB);
        // the staged points whose 8 x 8 cells meet the warp's (lane = point)
        const float4 pl = s_pt[buf][lane];
        const int ox = (__float_as_int(pl.z) - wx0 + GRW - 1) & (Lx - 1), oy = (__float_as_int(pl.w) - wy0 + GRW - 1) & (Ly - 1);
        unsigned todo = __ballot_sync(0xffffffffu, lane < n && ox < 8 + GRW - 1 && oy < 4 + GRW - 1);
        for (; todo; todo &= todo - 1) {
            const int i = __ffs(todo) - 1;
            const float4 pt = s_pt[buf][i];
            advance(s_ip[buf][i]);
            const int dx = (x - __float_as_int(pt.z)) & (Lx - 1), dy = (y - __float_as_int(pt.w)) & (Ly - 1);
            if (dx < GRW && dy < GRW) {
                const float w = s_wx[buf][i][dx] * s_wy[buf][i][dy];
                const float vr = w * pt.x, vi = w * pt.y;
                const float4 wa = *reinterpret_cast<const float4*>(s_ww[buf][i]);
                const float4 wb = *reinterpret_cast<const float4*>(s_ww[buf][i] + 4);
                const float ww[GRW] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
                for (int q = 0; q < GRW; ++q) {
                    acc[q].x = fmaf(ww[q], vr, acc[q].x);
                    acc[q].y = fmaf(ww[q], vi, acc[q].y);
                }
            }
        }
    }
    advance(tb);
}

// ------------------------------------------------------------------ set-up

__device__ __forceinline__ double es_kernel(double z)      // z in cells from the centre
{
    const double t = 2.0 * z / GRW, s = 1.0 - t * t;
    return s > 0.0 ? exp(GR_BETA * (sqrt(s) - 1.0)) : 0.0;
}

__global__ void grid_setup_vis_kernel(const d4* __restrict__ vd, int n_pad, GridOp g, double dl, double dm, double lc,
                                      double mc, double nc, double w0, double dw, int4* __restrict__ pos,
                                      float* __restrict__ wts, float2* __restrict__ rot)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n_pad) return;
    d4 v = vd[k];
    const bool mirror = v.z < 0.0;
    if (mirror) v = make_d4(-v.x, -v.y, -v.z, v.w);
    const int Lx = 1 << g.lx, Ly = 1 << g.ly;
    const double tx = v.x * dl, ty = v.y * dm;
    const double gx = (tx - floor(tx)) * Lx, gy = (ty - floor(ty)) * Ly, gw = (v.z - w0) / dw;
    const double ix = ceil(gx - 0.5 * GRW), iy = ceil(gy - 0.5 * GRW);
    const double iw = fmin(fmax(ceil(gw - 0.5 * GRW), 0.0), (double)(g.np - GRW));
    pos[k] = make_int4((int)ix & (Lx - 1), (int)iy & (Ly - 1), (int)iw, mirror ? 1 : 0);
    for (int t = 0; t < GRW; ++t) {
        wts[(size_t)k * 3 * GRW + t] = (float)es_kernel(ix + t - gx);
        wts[(size_t)k * 3 * GRW + GRW + t] = (float)es_kernel(iy + t - gy);
        wts[(size_t)k * 3 * GRW + 2 * GRW + t] = (float)es_kernel(iw + t - gw);
    }
    double a = v.x * lc, b = v.y * mc, c = v.z * nc;
    a -= rint(a);
    b -= rint(b);
    c -= rint(c);
    double s, co;
    sincospi(2.0 * (a + b + c), &s, &co);
    rot[k] = make_float2((float)co, (float)-s);
}

// amp = (1/n) / (transforms of the kernel in x, y and w); cxy: [nx] then [ny]
// reciprocal transforms, quad: GR_NQ nodes (cells) and weights times the
// kernel, for the transform in w.
__global__ void grid_setup_cells_kernel(const d4* __restrict__ pd, GridOp g, const double* __restrict__ cxy,
                                        const double* __restrict__ quad, double nc, double dw, float* __restrict__ amp,
                                        float2* __restrict__ nu)
{
    const size_t n = (size_t)g.nx * g.ny;
    for (size_t at = (size_t)blockIdx.x * blockDim.x + threadIdx.x; at < n; at += (size_t)gridDim.x * blockDim.x) {
        const int j = g.cell[at];
        if (j < 0) {
            amp[at] = 0.f;
            nu[at] = make_float2(0.f, 0.f);
            continue;
        }
        const d4 d = pd[j];
        const double v = d.z - nc, xi = v * dw;
        double hat = 0.0;
        for (int q = 0; q < GR_NQ; ++q) hat += quad[GR_NQ + q] * cospi(2.0 * xi * quad[q]);
        hat *= 2.0;
        amp[at] = (float)(d.w * cxy[at % g.nx] * cxy[g.nx + at / g.nx] / hat);
        const float hi = (float)v;
        nu[at] = make_float2(hi, (float)(v - (double)hi));
    }
}

cudaError_t grid_setup_vis(const d4* vd, int n_pad, GridOp g, double dl, double dm, double lc, double mc, double nc,
                           double w0, double dw, int4* pos, float* wts, float2* rot, cudaStream_t st)
{
    grid_setup_vis_kernel<<<(n_pad + 127) / 128, 128, 0, st>>>(vd, n_pad, g, dl, dm, lc, mc, nc, w0, dw, pos, wts,
                                                               rot);
    return cudaGetLastError();
}
cudaError_t grid_setup_cells(const d4* pd, GridOp g, const double* cxy, const double* quad, double nc, double dw,
                             float* amp, float2* nu, cudaStream_t st)
{
    const size_t n = (size_t)g.nx * g.ny;
    grid_setup_cells_kernel<<<(unsigned)std::min<size_t>(4096, (n + 127) / 128), 128, 0, st>>>(pd, g, cxy, quad, nc,
                                                                                               dw, amp, nu);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- launchers

template <int LOG>
static void rows_fwd(const DevProblem* probs, int p, const GridOp& g, int p0, int np, cudaStream_t st)
{
    using S = RowShape<LOG>;
    const dim3 grid((unsigned)((g.ny + S::ROWS - 1) / S::ROWS), (unsigned)((np + GR_PCH - 1) / GR_PCH));
    grid_rows_fwd_kernel<LOG><<<grid, S::THREADS, S::SMEM, st>>>(probs, p, g, p0, np);
}
template <int LOG>
static void rows_adj(const DevProblem* probs, int p, const GridOp& g, int p0, int np, int n_pix, int n_pix_pad,
                     double* partial, cudaStream_t st)
{
    using S = RowShape<LOG>;
    const dim3 grid((unsigned)((g.ny + S::ROWS - 1) / S::ROWS), (unsigned)((np + GR_PCH - 1) / GR_PCH));
    grid_rows_adj_kernel<LOG><<<grid, S::THREADS, S::SMEM, st>>>(probs, p, g, p0, np, n_pix, n_pix_pad, partial);
}
template <int LOG, int SGN>
static void cols(const DevProblem* probs, int p, const GridOp& g, int p0, int np, cudaStream_t st)
{
    using S = ColShape<LOG>;
    const dim3 grid((1u << g.lx) / S::CB, (unsigned)np);
    grid_cols_kernel<LOG, SGN><<<grid, S::THREADS, S::SMEM, st>>>(probs, p, g, p0);
}

// Calls F<LOG>::go(args...) for the run-time length lg.
#define GRID_DISPATCH(lg, CALL)                  \
    switch (lg) {                                \
    case 6: { constexpr int LOG = 6; CALL; break; }   \
    case 7: { constexpr int LOG = 7; CALL; break; }   \
    case 8: { constexpr int LOG = 8; CALL; break; }   \
    case 9: { constexpr int LOG = 9; CALL; break; }   \
    case 10: { constexpr int LOG = 10; CALL; break; } \
    case 11: { constexpr int LOG = 11; CALL; break; } \
    case 12: { constexpr int LOG = 12; CALL; break; } \
    default: return cudaErrorInvalidValue;       \
    }

cudaError_t grid_forward(const DevProblem* probs, int p, const GridOp& g, int n_vis_pad, double2* partial,
                         cudaStream_t st, long long* n_launch)
{
    for (int p0 = 0; p0 < g.np; p0 += g.np_pass) {
        const int np = std::min(g.np_pass, g.np - p0);
        GRID_DISPATCH(g.lx, (rows_fwd<LOG>(probs, p, g, p0, np, st)));
        GRID_DISPATCH(g.ly, (cols<LOG, -1>(probs, p, g, p0, np, st)));
        if (g.np_pass >= g.np)
            grid_gather_kernel<true><<<(n_vis_pad + 7) / 8, 256, 0, st>>>(probs, p, g, p0, np, n_vis_pad, partial);
        else
            grid_gather_kernel<false><<<(n_vis_pad + 7) / 8, 256, 0, st>>>(probs, p, g, p0, np, n_vis_pad, partial);
        *n_launch += 3;
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t grid_adjoint(const DevProblem* probs, int p, const GridOp& g, int n_pix, int n_pix_pad, double* partial,
                         cudaStream_t st, long long* n_launch)
{
    for (int p0 = 0; p0 < g.np; p0 += g.np_pass) {
        const int np = std::min(g.np_pass, g.np - p0);
        // segments of planes: enough CTAs for a few waves, no fewer planes than 32
        // and no more than GR_SEG
        const int tiles = grid_tiles(g);
        const int nseg = std::max((np + GR_SEG - 1) / GR_SEG, std::max(1, std::min((np + 31) / 32, 4096 / tiles)));
        const int seg = (np + nseg - 1) / nseg;
        const dim3 sg((unsigned)tiles, (unsigned)((np + seg - 1) / seg));
        grid_spread_kernel<<<sg, GR_TILE * GR_TILE, 0, st>>>(probs, p, g, p0, np, seg);
        GRID_DISPATCH(g.ly, (cols<LOG, 1>(probs, p, g, p0, np, st)));
        GRID_DISPATCH(g.lx, (rows_adj<LOG>(probs, p, g, p0, np, n_pix, n_pix_pad, partial, st)));
        *n_launch += 3;
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <int LOG>
static cudaError_t raise_limits()
{
    cudaError_t e = cudaFuncSetAttribute(grid_cols_kernel<LOG, -1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         ColShape<LOG>::SMEM);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(grid_cols_kernel<LOG, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             ColShape<LOG>::SMEM);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(grid_rows_fwd_kernel<LOG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             RowShape<LOG>::SMEM);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(grid_rows_adj_kernel<LOG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                RowShape<LOG>::SMEM);
}
cudaError_t grid_prepare_kernels(int lx, int ly)
{
    cudaError_t e = cudaSuccess;
    GRID_DISPATCH(lx, (e = raise_limits<LOG>()));
    if (e != cudaSuccess || lx == ly) return e;
    GRID_DISPATCH(ly, (e = raise_limits<LOG>()));
    return e;
}

}  // namespace sl1m
