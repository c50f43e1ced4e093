// sl1m_kernels.h -- launch wrappers of the libsl1m kernels (internal).
#pragma once
#include "sl1m_dev.h"

namespace sl1m {

enum FinishMode : int { FIN_OP = 0, FIN_POWER = 1, FIN_SOLVE = 2, FIN_INIT = 3 };

// operator kernels (sl1m_mixed.cu, sl1m_fp64.cu); precision 0 = FP64, 1 = mixed.
// plp: device-resident plan; C: its grid size (known on the host).
// nst: streamed granules per shared-memory stage of the mixed no-gains
// kernels (2, 4 or 8; the tile shape the autotuner picks).
constexpr int NST_DEFAULT = 4;
// Tile-shape code carried as `nst` below: streamed granules per stage (2, 4
// or 8) plus 16 x npoly, the pairs of every 8 whose sincos runs on the FMA
// pipe (0, 1 or 2; Dirac tiles without gains).
// Bit 8: the batch has no Gaussian pixels, so the no-gains mixed kernels may
// run an instance compiled without the Gaussian tiles.
constexpr int SHAPE_DIRAC_ONLY = 1 << 8;
constexpr int shape_code(int nst, int npoly) { return nst | (npoly << 4); }
constexpr int shape_nst(int code) { return code & 15; }
constexpr int shape_npoly(int code) { return (code >> 4) & 15; }
constexpr bool shape_dirac_only(int code) { return (code & SHAPE_DIRAC_ONLY) != 0; }
// The shape code of a launch over pixels that may (gauss) or may not hold
// Gaussian pixels.
constexpr int shape_for(int code, bool gauss) { return gauss ? (code & ~SHAPE_DIRAC_ONLY) : (code | SHAPE_DIRAC_ONLY); }
cudaError_t launch_forward(int precision, bool gains, int n_ant, const DevProblem* probs,
                           const Plan* plp, int C, double2* partial, cudaStream_t st, int nst = NST_DEFAULT);
cudaError_t launch_adjoint(int precision, bool gains, int n_ant, const DevProblem* probs, const Plan* plp, int C,
                           double* partial, cudaStream_t st, int nst = NST_DEFAULT);
// which: 0 fwd fp64, 1 adj fp64, 2 fwd mixed, 3 adj mixed
int occupancy(int which, bool gains, int n_ant, int nst = NST_DEFAULT);
int fwd_smem_bytes(int n_ant, bool gains, int nst);
// Writes the FP64 kernels' tables on the current device; called for its first context.
cudaError_t fp64_init_tables(cudaStream_t st);
// Owned granules per block of a plan.  A CTA of the mixed gains adjoint works on
// one pixel granule at a time with all its warps, so its blocks are granules:
// a CTA's range is then a long run of visibility granules for its 8 warps,
// where 8 granules x a short run left some of them idle on small problems.
constexpr int own_granules(int precision, int op, bool gains)
{
    return precision != 0 && op == 1 && gains ? 1 : BLK_GRAN;
}
constexpr int own_blocks(int precision, int op, bool gains, int n_gran)
{
    return (n_gran + own_granules(precision, op, gains) - 1) / own_granules(precision, op, gains);
}
// Streamed granules as the plans count them: the FP64 kernels' units
// stream one element, FP64_SUB per granule.
constexpr int stream_units(int precision, int n_gran) { return precision == 0 ? n_gran * FP64_SUB : n_gran; }
// The adjoints without FP64 gains read r in polar form too, {|r|, arg r in turns}
// in FP32 (r32) or {arg r in 1/R64_TURN turns, |r|} in FP64 (r64).  Whatever writes r
// writes it: `polar` below is 0 (the lattice operator, FP64 gains), 1 r32 or 2 r64.
// Per-visibility constants of up to GCLS_MAX Gaussian scales.
constexpr int GCLS_MAX = 4;
cudaError_t launch_gauss_class(const d4* vd, int n_pad, const double* sigma, int n_cls, float4* gcls, cudaStream_t st);
// The mixed gains kernels' bounded waits for their bulk copies set a device
// flag when they give up; read it into *host_flag (asynchronously on st: valid
// after the stream is synchronised) and clear it.
cudaError_t wait_fault_read(unsigned* host_flag, cudaStream_t st);
cudaError_t wait_fault_clear(cudaStream_t st);
// Self-test: n_blocks CTAs each wait on an mbarrier nobody arrives on; the
// waits give up after wait_limit_ns() and set the flag above; waited_ns
// [n_blocks] (device) receives how long each CTA's thread 0 waited.
cudaError_t launch_wait_selftest(unsigned long long* waited_ns, int n_blocks, cudaStream_t st);
unsigned long long wait_limit_ns();

// solver kernels (sl1m_solver.cu)
// huge (may be null): set where a value is GR_HUGE or more (sl1m_grid.h).
cudaError_t launch_gather_real(const double* src, double* dst, const int* orig, int n_pad,
                               double scale, int* huge, cudaStream_t st);
// P: the problem's descriptor on the device.
cudaError_t launch_gather_resid(const double2* src, const DevProblem* P, int n_pad, int polar, double2* dst,
                                cudaStream_t st);
cudaError_t launch_scatter_real(const double* src, double* dst, const int* orig, int n_pad,
                                cudaStream_t st);
cudaError_t launch_scatter_cplx(const double2* src, double2* dst, const int* orig, int n_pad,
                                cudaStream_t st);
cudaError_t launch_fill_valid(double* dst, const int* orig, int n_pad, double val, cudaStream_t st);
cudaError_t launch_weighted_vis(const DevProblem* P, int n_pad, int polar, double2* r, cudaStream_t st);
// pl: host copy of the plan's header.  user_out: where an operator call's result
// goes, in the caller's order (null: the descriptor's array, in the library's).
cudaError_t launch_fwd_finish(const DevProblem* probs, const Plan* plp, const Plan& pl, int num_sms,
                              const double2* partial, int polar, double2* user_out, cudaStream_t st);
cudaError_t launch_adj_finish(const DevProblem* probs, const Plan* plp, const Plan& pl, int num_sms,
                              const double* partial, double* user_out, cudaStream_t st);
cudaError_t launch_mfista_mix(const DevProblem* probs, const Plan* fplp, const Plan* aplp, int grid, int polar,
                              cudaStream_t st);
// evals (may be null): [0] += pairs the forward and [1] += pairs the adjoint
// evaluated in this tick, summed over the problems that took part.
cudaError_t launch_scalars(const DevProblem* probs, const int* n_probs, int grid, double* evals, cudaStream_t st);
cudaError_t launch_phases(const DevProblem* probs, const int* n_probs, int grid, int* out, cudaStream_t st);

}  // namespace sl1m
