// sl1m_fp64.cu -- the "plain" FP64 forward operator and adjoint of SL1M
// (Hardy 2013, Sect. 2 and 3.1): the same stream-K decomposition of work as
// the mixed kernels, every step in FP64 (phase, sine and cosine, exponential,
// accumulation).  Gaussian pixels use the real split form of Eq. samlm4/samlm5
// given in sl1m_mixed.cu; gains multiply by G[j][a_k] conj(G[j][b_k]).
//
// The SM executes 2 FP64 multiply-adds per clock (1/64 of its FP32 rate), so
// these kernels are bound by the number of FP64 instructions of a pair and
// everything else hides behind them:
//   - sine and cosine come from a table of 2048 points of the circle (32 KB,
//     in shared memory) and the Taylor polynomials of the rest of the angle,
//     |theta| <= pi/2048, where two terms each reach 2^-53: 8 instructions
//     after the reduction, 4 of them the rotation, instead of sincospi's
//     two polynomials on a quarter turn; the exponential likewise from 2^(i/2048);
//   - the phase is carried in 1/2048 turns, so its reduction and the table index
//     are one add of 1.5 2^52, two subtracts and an integer mask;
//   - the adjoint (real output) takes r in polar form and the cosine alone;
//   - what depends on one side only is formed once per tile.
// Counted FP64 instructions per pair: forward 16 (Dirac), 32 (Gaussian);
// adjoint 14 and 30; before, about 40 and 80.  Measured on GB300: 16,384
// multiscale pixels x 8,064 visibilities, adjoint 16.68 -> 6.78 ms, which is
// 1.8 of the 2 instructions per clock; 1024 x 2208 Dirac, forward 91 and
// adjoint 68 us (floors 61 and 53 us).
//
// A unit is an owned block of 512 elements times one streamed element (the
// mixed kernels': times a granule of 64): a pair costs so much here that small
// problems have to split evenly over all SMs (1024 pixels x 2208 visibilities:
// 80 units of a whole granule kept half the SMs idle).
#include "sl1m_dev.h"
#include "sl1m_devfn.cuh"
#include "sl1m_kernels.h"

namespace sl1m {

constexpr int CIRC = (int)R64_TURN;                 // table points of the circle, and of [1, 2) for 2^x
static_assert(FP64_SUB == G, "a unit streams one element");

// e^{2 pi i k / CIRC} and 2^(k / CIRC), filled for a device's first context (fp64_init_tables).
__device__ double2 g_circ[CIRC];
__device__ double g_exp2[CIRC];

__global__ void fp64_tables_kernel()
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= CIRC) return;
    double s, c;
    sincospi(2.0 * k / CIRC, &s, &c);
    g_circ[k] = make_double2(c, s);
    g_exp2[k] = exp2((double)k / CIRC);
}
cudaError_t fp64_init_tables(cudaStream_t st)
{
    fp64_tables_kernel<<<CIRC / 256, 256, 0, st>>>();
    return cudaGetLastError();
}

#define FP64_MAGIC 6755399441055744.0      // 1.5 2^52: adding it rounds to an integer

// The nearest table point (its index) and the rest of x, a multiple of 1/CIRC.
__device__ __forceinline__ double split_rest(double x, int& k)
{
    const double m = __dadd_rn(x, FP64_MAGIC);
    k = __double2loint(m);
    return __dadd_rn(x, -__dadd_rn(m, -FP64_MAGIC));
}

// Taylor coefficients of the angle theta = A0 d, d in 1/CIRC turns, |d| <= 1/2:
// sin theta = d (A0 + A1 d^2) to theta^5/120 < 7e-17, cos theta - 1 =
// d^2 (B1 + B2 d^2) to theta^6/720 < 2e-20.
constexpr double C_A0 = 6.283185307179586476925286766559 / CIRC;
constexpr double C_A1 = -C_A0 * C_A0 * C_A0 / 6.0;
constexpr double C_B1 = -C_A0 * C_A0 / 2.0;
constexpr double C_B2 = C_A0 * C_A0 * C_A0 * C_A0 / 24.0;

// cos and sin of x / CIRC turns, |x| < 2^51.
__device__ __forceinline__ void cis_circ(double x, const double2* __restrict__ circ, double& c, double& s)
{
    int k;
    const double d = split_rest(x, k);
    const double2 t = circ[k & (CIRC - 1)];
    const double z = d * d;
    const double sd = d * fma(C_A1, z, C_A0), cz = z * fma(C_B2, z, C_B1);
    c = fma(-t.y, sd, fma(t.x, cz, t.x));
    s = fma(t.x, sd, fma(t.y, cz, t.y));
}
__device__ __forceinline__ double cos_circ(double x, const double2* __restrict__ circ)
{
    int k;
    const double d = split_rest(x, k);
    const double2 t = circ[k & (CIRC - 1)];
    const double z = d * d;
    const double sd = d * fma(C_A1, z, C_A0), cz = z * fma(C_B2, z, C_B1);
    return fma(-t.y, sd, fma(t.x, cz, t.x));
}

// 2^(x / CIRC) for x <= 0 (below 2^-1022: 0).  2^(d / CIRC), |d| <= 1/2, to
// (ln 2 / 4096)^4 / 24 < 4e-17.
constexpr double E_1 = 0.693147180559945309417232121458 / CIRC;
constexpr double E_2 = E_1 * E_1 / 2.0, E_3 = E_1 * E_1 * E_1 / 6.0;
__device__ __forceinline__ double exp2_circ(double x, const double* __restrict__ tab)
{
    const bool gone = !(x > -1022.0 * CIRC);             // (NaN: caught by the phase)
    int k;
    const double d = split_rest(gone ? -1022.0 * CIRC : x, k);
    const double t = tab[k & (CIRC - 1)];
    const double p = fma(d * fma(d, fma(d, E_3, E_2), E_1), t, t);
    const int hi = __double2hiint(p) + ((k >> 11) << 20);   // times 2^(k div CIRC): the exponent field
    return gone ? 0.0 : __hiloint2double(hi, __double2loint(p));
}
static_assert(CIRC == 1 << 11, "the exponent shift in exp2_circ");

// Constants of one (visibility, Gaussian scale) pair; u, v, w and the phase in
// 1/CIRC turns (u = CIRC u_k and so on).
struct Gauss64 {
    double beta, id;     // beta = w s^2, id = 1/(1 + beta^2)
    double gam;          // beta^2 id
    double cph;          // + id beta s^2 (u^2 + v^2) / 2 of the phase
    double coef;         // exponent (1/CIRC of a power of two) = coef |(u,v) - w (l,m)|^2
};
__device__ __forceinline__ Gauss64 gauss64(double u, double v, double w, double sigma)
{
    Gauss64 g;
    const double s2 = sigma * sigma;
    g.beta = w * (1.0 / CIRC) * s2;
    g.id = 1.0 / (1.0 + g.beta * g.beta);
    g.gam = g.beta * g.beta * g.id;
    g.cph = 0.5 * g.id * g.beta * s2 * (u * u + v * v) * (1.0 / CIRC);
    // -pi s^2 id |.|^2 / ln 2, |.|^2 in units of CIRC^2, the exponent in 1/CIRC
    g.coef = -4.532360141827193809627682945717 * s2 * g.id / CIRC;
    return g;
}

// log2 amplitude (1/CIRC) and phase (1/CIRC turns, plus add) of a Gaussian
// pair, the factor id (1 + i beta) left out.  pg = {l, m, r^2/2, nu}; phi: the
// Dirac phase, by far the largest term, so the others are summed first.
template <bool PAR>
__device__ __forceinline__ void gauss_pair64(double u, double v, double w, const d4& pg, double phi, double gam,
                                             double coef, double add, double& ex, double& ph)
{
    const double e1 = fma(-w, pg.x, u), e2 = fma(-w, pg.y, v);
    ex = coef * fma(e1, e1, e2 * e2);
    const double t = fma(-w, pg.w, phi);                  // u l + v m - w r^2/2
    ph = (PAR ? t : phi) + fma(-gam, t, add);             // paraxial: without w nu
}

extern __shared__ __align__(16) unsigned char s_fp64[];

// Shared memory: the circle, the powers of two (GAUSS), then the kernel's own.
template <bool GAUSS>
__device__ __forceinline__ void load_tables(double2*& circ, double*& ex, unsigned char*& rest)
{
    circ = reinterpret_cast<double2*>(s_fp64);
    ex = reinterpret_cast<double*>(s_fp64 + CIRC * 16);
    rest = s_fp64 + CIRC * (GAUSS ? 24 : 16);
    for (int i = threadIdx.x; i < CIRC; i += NTHREADS) {
        circ[i] = g_circ[i];
        if (GAUSS) ex[i] = g_exp2[i];
    }
}

constexpr int FWD64_OWN = G * (32 + 32);                        // {l, m, n-1, x/n}, {l, m, r^2/2, nu}
constexpr int ADJ64_OWN = G * (32 + 16 + 8);                    // {u, v, w, W}, r, antennas
constexpr int ADJ64_REC = BLK_GRAN * G * 32;                    // per warp: Gaussian records

__device__ __forceinline__ d4 to_circ(d4 v) { return make_d4(v.x * CIRC, v.y * CIRC, v.z * CIRC, v.w); }

template <int KIND, bool GAINS>
__device__ __forceinline__ void fwd64_tile(const DevProblem& P, int e0, int n, const d4* __restrict__ s_pd,
                                           const d4* __restrict__ s_pg, const double2* __restrict__ circ,
                                           const double* __restrict__ ex2, const d4 (&vd)[2], const Gauss64 (&gc)[2],
                                           const int2 (&ant)[2], double (&sr)[2], double (&si)[2])
{
#pragma unroll 2
    for (int j = 0; j < n; ++j) {
        const d4 pd = s_pd[j];
        d4 pg = pd;
        if (KIND != DIRAC) pg = s_pg[j];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            double m = pd.w, ph = fma(vd[r].z, pd.z, fma(vd[r].y, pd.y, vd[r].x * pd.x));
            if (KIND != DIRAC) {
                double ex;
                gauss_pair64<KIND == PARAXIAL>(vd[r].x, vd[r].y, vd[r].z, pg, ph, gc[r].gam, gc[r].coef, gc[r].cph,
                                               ex, ph);
                m *= exp2_circ(ex, ex2);
            }
            double c, s;
            cis_circ(ph, circ, c, s);
            if (GAINS) {
                const double2* gj = P.gains64 + (size_t)(e0 + j) * P.n_ant;
                const double2 ga = gj[ant[r].x], gb = gj[ant[r].y];
                const double gr = fma(ga.x, gb.x, ga.y * gb.y), gi = fma(ga.y, gb.x, -ga.x * gb.y);
                const double t = fma(gr, c, gi * s);       // (gr + i gi)(c - i s)
                s = fma(gr, s, -gi * c);
                c = t;
            }
            sr[r] = fma(m, c, sr[r]);
            si[r] = fma(-m, s, si[r]);
        }
    }
}

template <bool GAUSS, bool GAINS>
__global__ void __launch_bounds__(NTHREADS, 2)
fwd_fp64_kernel(const DevProblem* __restrict__ probs, const Plan* __restrict__ plp, double2* __restrict__ partial)
{
    double2* circ;
    double* ex2;
    unsigned char* rest;
    load_tables<GAUSS>(circ, ex2, rest);
    d4* s_pd = reinterpret_cast<d4*>(rest);                 // {l, m, n-1, a = x/n}
    d4* s_pg = s_pd + G;                                    // {l, m, r^2/2, nu}
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const Plan pl = *plp;
    const long long c = blockIdx.x;
    long long u, u_end;
    cta_range(pl, c, u, u_end);
    while (u < u_end) {
        const int p = find_prob(pl, u);
        const DevProblem& P = probs[p];
        const long long loc = u - pl.prob_u0[p];
        const double* X;
        if (!fwd_role(P, X)) {                    // problem not in this step: skip its units
            u = min(u_end, pl.prob_u0[p + 1]);
            continue;
        }
        const int upb = P.pix.n_gran * FP64_SUB;
        const int blk = (int)(loc / upb);
        const int g0 = (int)(loc % upb);
        const int g1 = (int)min((long long)upb, (long long)g0 + (u_end - u));
        const int vg = blk * BLK_GRAN + warp;
        const bool vg_ok = vg < P.vis.n_gran;
        d4 vd[2];
        int2 ant[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            vd[r] = make_d4(0.0, 0.0, 0.0, 0.0);
            ant[r] = make_int2(0, 0);
            if (vg_ok) {
                const int e = vg * G + lane + 32 * r;
                vd[r] = to_circ(P.vis.d[e]);
                if (GAINS) ant[r] = P.ant[e];
            }
        }
        double tr[2] = {0.0, 0.0}, ti[2] = {0.0, 0.0};
        // g0, g1 are pixels; runs within one granule (its kind and sigma are uniform)
        for (int e = g0, e1; e < g1; e = e1) {
            const int g = e / G;
            e1 = min(g1, (g + 1) * G);
            const int n = e1 - e;
            __syncthreads();
            const int kind = GAUSS ? P.gkind[g] : DIRAC;
            if (threadIdx.x < n) {
                d4 d = P.pix.d[e + threadIdx.x];
                d.w = X[e + threadIdx.x] * d.w;
                s_pd[threadIdx.x] = d;
                if (GAUSS && kind != DIRAC) s_pg[threadIdx.x] = P.pgauss64[e + threadIdx.x];
            }
            __syncthreads();
            Gauss64 gc[2] = {};
            if (!GAUSS || kind == DIRAC) {
                fwd64_tile<DIRAC, GAINS>(P, e, n, s_pd, s_pg, circ, ex2, vd, gc, ant, tr, ti);
            } else {
                const double sigma = P.gsig64[g];
                double sr[2] = {0.0, 0.0}, si[2] = {0.0, 0.0};
#pragma unroll
                for (int r = 0; r < 2; ++r) gc[r] = gauss64(vd[r].x, vd[r].y, vd[r].z, sigma);
                if (kind == PARAXIAL) fwd64_tile<PARAXIAL, GAINS>(P, e, n, s_pd, s_pg, circ, ex2, vd, gc, ant, sr, si);
                else fwd64_tile<WIDE, GAINS>(P, e, n, s_pd, s_pg, circ, ex2, vd, gc, ant, sr, si);
#pragma unroll
                for (int r = 0; r < 2; ++r) {             // id (1 + i beta)
                    tr[r] = fma(gc[r].id, fma(-gc[r].beta, si[r], sr[r]), tr[r]);
                    ti[r] = fma(gc[r].id, fma(gc[r].beta, sr[r], si[r]), ti[r]);
                }
            }
        }
        if (vg_ok) {
            const int gb = pl.prob_b0[p] + blk;
            double2* dst = partial + (size_t)slot_of(pl, gb) * BLK + warp * G + lane;
#pragma unroll
            for (int r = 0; r < 2; ++r) dst[32 * r] = make_double2(tr[r], ti[r]);
        }
        u += g1 - g0;
    }
}

// One run of streamed visibilities for a warp's pixel granule.  s_rec (Gaussian
// owners): {arg r' + constant phase (1/CIRC turns), |r'|, gam, coef}, r' =
// id (1 - i beta) r; Dirac owners read r itself in polar form.  With gains r
// stays Cartesian (r' for Gaussian owners too).
template <int KIND, bool GAINS>
__device__ __forceinline__ void adj64_tile(const DevProblem& P, int n, const d4* __restrict__ s_vd,
                                           const double2* __restrict__ s_r, const int2* __restrict__ s_ant,
                                           const d4* __restrict__ s_rec, const double2* __restrict__ circ,
                                           const double* __restrict__ ex2, const d4 (&pd)[2], const d4 (&pg)[2],
                                           const int (&eidx)[2], double sigma, double (&tot)[2])
{
#pragma unroll 2
    for (int k = 0; k < n; ++k) {
        const d4 vd = s_vd[k];
        const double2 rr = s_r[k];
        d4 rec = vd;
        if (KIND != DIRAC && !GAINS) rec = s_rec[k];
        Gauss64 gc = {};
        if (KIND != DIRAC && GAINS) gc = gauss64(vd.x, vd.y, vd.z, sigma);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            // (Dirac, polar r: arg r starts the chain)
            const double x0 = KIND == DIRAC && !GAINS ? fma(vd.x, pd[r].x, rr.x) : vd.x * pd[r].x;
            double ph = fma(vd.z, pd[r].z, fma(vd.y, pd[r].y, x0));
            double m = KIND == DIRAC ? rr.y : rec.y, ex;
            if (KIND != DIRAC) {
                gauss_pair64<KIND == PARAXIAL>(vd.x, vd.y, vd.z, pg[r], ph, GAINS ? gc.gam : rec.z,
                                               GAINS ? gc.coef : rec.w, GAINS ? gc.cph : rec.x, ex, ph);
                const double a = exp2_circ(ex, ex2);
                m = GAINS ? a : m * a;
            }
            if (!GAINS) {
                tot[r] = fma(m, cos_circ(ph, circ), tot[r]);
            } else {
                double c, s;
                cis_circ(ph, circ, c, s);
                // e = (1 + i beta) id a (c - i s) times g = G_a conj(G_b); Re(conj(e g) r)
                double er = c, ei = -s;
                if (KIND != DIRAC) {
                    const double f = m * gc.id;
                    er = f * fma(gc.beta, s, c);
                    ei = f * fma(gc.beta, c, -s);
                }
                const int2 ab = s_ant[k];
                const double2* gj = P.gains64 + (size_t)eidx[r] * P.n_ant;
                const double2 ga = gj[ab.x], gb = gj[ab.y];
                const double gr = fma(ga.x, gb.x, ga.y * gb.y), gi = fma(ga.y, gb.x, -ga.x * gb.y);
                const double hr = fma(er, gr, -ei * gi), hi = fma(er, gi, ei * gr);
                tot[r] = fma(hr, rr.x, fma(hi, rr.y, tot[r]));
            }
        }
    }
}

template <bool GAUSS, bool GAINS>
__global__ void __launch_bounds__(NTHREADS, 2)
adj_fp64_kernel(const DevProblem* __restrict__ probs, const Plan* __restrict__ plp, double* __restrict__ partial)
{
    double2* circ;
    double* ex2;
    unsigned char* rest;
    load_tables<GAUSS>(circ, ex2, rest);
    d4* s_vd = reinterpret_cast<d4*>(rest);                 // {u, v, w (times CIRC), W}
    double2* s_r = reinterpret_cast<double2*>(s_vd + G);    // r in polar form {arg (1/CIRC turns), |r|}; gains: r
    int2* s_ant = reinterpret_cast<int2*>(s_r + G);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    d4* s_rec = reinterpret_cast<d4*>(rest + ADJ64_OWN) + warp * G;   // GAUSS, no gains
    const Plan pl = *plp;
    const long long c = blockIdx.x;
    long long u, u_end;
    cta_range(pl, c, u, u_end);
    while (u < u_end) {
        const int p = find_prob(pl, u);
        const DevProblem& P = probs[p];
        const long long loc = u - pl.prob_u0[p];
        const double2* R;
        if (!adj_role(P, R)) {                    // problem not in this step: skip its units
            u = min(u_end, pl.prob_u0[p + 1]);
            continue;
        }
        const int upb = P.vis.n_gran * FP64_SUB;
        const int blk = (int)(loc / upb);
        const int g0 = (int)(loc % upb);
        const int g1 = (int)min((long long)upb, (long long)g0 + (u_end - u));
        const int pgi = blk * BLK_GRAN + warp;
        const bool pg_ok = pgi < P.pix.n_gran;
        const int kind = GAUSS && pg_ok ? P.gkind[pgi] : DIRAC;
        const double sigma = pg_ok ? P.gsig64[pgi] : 0.0;
        d4 pd[2], pg[2];
        int eidx[2] = {0, 0};
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            pd[r] = pg[r] = make_d4(0.0, 0.0, 0.0, 0.0);
            if (pg_ok) {
                const int e = pgi * G + lane + 32 * r;
                eidx[r] = e;
                pd[r] = P.pix.d[e];
                if (GAUSS && kind != DIRAC) pg[r] = P.pgauss64[e];
            }
        }
        double tot[2] = {0.0, 0.0};
        for (int e = g0, e1; e < g1; e = e1) {
            e1 = min(g1, (e / G + 1) * G);
            const int n = e1 - e;
            __syncthreads();
            if (threadIdx.x < n) {
                const int k = e + threadIdx.x;
                s_vd[threadIdx.x] = to_circ(P.vis.d[k]);
                s_r[threadIdx.x] = GAINS ? R[k] : P.r64[k];
                if (GAINS) s_ant[threadIdx.x] = P.ant[k];
            }
            __syncthreads();
            if (!GAUSS || kind == DIRAC) {
                adj64_tile<DIRAC, GAINS>(P, n, s_vd, s_r, s_ant, s_rec, circ, ex2, pd, pg, eidx, sigma, tot);
                continue;
            }
            if (!GAINS) {                         // this warp's records of the run
                for (int k = lane; k < n; k += 32) {
                    const d4 v = s_vd[k];
                    const Gauss64 gc = gauss64(v.x, v.y, v.z, sigma);
                    const double2 rr = s_r[k];
                    // |r'| = |r| sqrt(id), arg r' = arg r - atan(beta)
                    s_rec[k] = make_d4(rr.x + gc.cph - atan(gc.beta) * (0.15915494309189533577 * CIRC),
                                       rr.y * sqrt(gc.id), gc.gam, gc.coef);
                }
                __syncwarp();
            }
            if (kind == PARAXIAL)
                adj64_tile<PARAXIAL, GAINS>(P, n, s_vd, s_r, s_ant, s_rec, circ, ex2, pd, pg, eidx, sigma, tot);
            else
                adj64_tile<WIDE, GAINS>(P, n, s_vd, s_r, s_ant, s_rec, circ, ex2, pd, pg, eidx, sigma, tot);
        }
        if (pg_ok) {
            const int gb = pl.prob_b0[p] + blk;
            double* dst = partial + (size_t)slot_of(pl, gb) * BLK + warp * G + lane;
#pragma unroll
            for (int r = 0; r < 2; ++r) dst[32 * r] = tot[r] * pd[r].w;
        }
        u += g1 - g0;
    }
}

// ------------------------------------------------------------- launchers

cudaError_t launch_forward_mixed(bool gains, int n_ant, int nst, const DevProblem* probs, const Plan* plp, int C,
                                 double2* partial, cudaStream_t st);
cudaError_t launch_adjoint_mixed(bool gains, int n_ant, int nst, const DevProblem* probs, const Plan* plp, int C,
                                 double* partial, cudaStream_t st);
int occupancy_mixed(int op, bool gains, int n_ant, int nst);

static int fwd64_smem(bool gauss) { return CIRC * (gauss ? 24 : 16) + FWD64_OWN; }
static int adj64_smem(bool gauss) { return CIRC * (gauss ? 24 : 16) + ADJ64_OWN + (gauss ? ADJ64_REC : 0); }
using Fwd64 = void (*)(const DevProblem*, const Plan*, double2*);
using Adj64 = void (*)(const DevProblem*, const Plan*, double*);
// The instance without the Gaussian tiles for batches without Gaussian pixels
// (SHAPE_DIRAC_ONLY in the shape code).
static Fwd64 fwd64_of(bool gauss, bool gains)
{
    return gauss ? (gains ? fwd_fp64_kernel<true, true> : fwd_fp64_kernel<true, false>)
                 : (gains ? fwd_fp64_kernel<false, true> : fwd_fp64_kernel<false, false>);
}
static Adj64 adj64_of(bool gauss, bool gains)
{
    return gauss ? (gains ? adj_fp64_kernel<true, true> : adj_fp64_kernel<true, false>)
                 : (gains ? adj_fp64_kernel<false, true> : adj_fp64_kernel<false, false>);
}

cudaError_t launch_forward(int precision, bool gains, int n_ant, const DevProblem* probs,
                           const Plan* plp, int C, double2* partial, cudaStream_t st, int nst)
{
    if (precision == 0) {
        const bool gauss = !shape_dirac_only(nst);
        fwd64_of(gauss, gains)<<<C, NTHREADS, fwd64_smem(gauss), st>>>(probs, plp, partial);
        return cudaGetLastError();
    }
    return launch_forward_mixed(gains, n_ant, nst, probs, plp, C, partial, st);
}

cudaError_t launch_adjoint(int precision, bool gains, int n_ant, const DevProblem* probs, const Plan* plp, int C,
                           double* partial, cudaStream_t st, int nst)
{
    if (precision == 0) {
        const bool gauss = !shape_dirac_only(nst);
        adj64_of(gauss, gains)<<<C, NTHREADS, adj64_smem(gauss), st>>>(probs, plp, partial);
        return cudaGetLastError();
    }
    return launch_adjoint_mixed(gains, n_ant, nst, probs, plp, C, partial, st);
}

int occupancy(int which, bool gains, int n_ant, int nst)
{
    if (which >= 2) return occupancy_mixed(which - 2, gains, n_ant, nst);
    // (raises the shared-memory limits: batches are built outside captures)
    const bool gauss = !shape_dirac_only(nst);
    const int sm = which == 0 ? fwd64_smem(gauss) : adj64_smem(gauss);
    const void* k = which == 0 ? (const void*)fwd64_of(gauss, gains) : (const void*)adj64_of(gauss, gains);
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, NTHREADS, sm);
    return n < 1 ? 1 : n;
}

}  // namespace sl1m
