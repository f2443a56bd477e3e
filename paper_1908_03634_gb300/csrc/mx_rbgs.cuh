// Single-pass red-black Gauss-Seidel sweep and the per-cell update it shares
// with the two-pass colour kernels.
#pragma once

#include <climits>

#include "mx_stencil.cuh"

enum { RB_PLAIN = 0, RB_ZERO = 1, RB_PROLONG = 2 };

// Rounded arithmetic without contraction: every kernel that updates a cell
// (two-pass colour passes, the single-pass sweep, the batched and coarse-end
// kernels) evaluates the update with exactly these operations, so they agree
// bit for bit whatever FMA contractions the compiler would choose in each.
// FP32 multiplies with the hardware's approximate reciprocal of the diagonal (1
// ulp; subnormal sums, far below any face-coefficient sum here, count as 0), FP64
// with a correctly rounded one.  The smoother only sets the V-cycle's
// contraction, the refinement loop the accuracy.
__device__ __forceinline__ float rmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double rmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float radd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double radd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float rfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double rfma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float rinv(float a) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}
__device__ __forceinline__ double rinv(double a) { return __drcp_rn(a); }

// 1 / sum_f b_f of a cell's row
template <typename T>
__device__ __forceinline__ T gs_inverse(const T b[6]) {
    return rinv(radd(radd(radd(b[0], b[1]), radd(b[2], b[3])), radd(b[4], b[5])));
}

// Exact solve of cell c's row: e_c = (sum_f b_f e_nb - h^2 f_c) / sum_f b_f, with
// inv = gs_inverse(b).
template <typename T>
__device__ __forceinline__ T gs_numerator(const T b[6], const T v[6], T f, T h2) {
    T num = rmul(b[0], v[0]);
    num = rfma(b[1], v[1], num);
    num = rfma(b[2], v[2], num);
    num = rfma(b[3], v[3], num);
    num = rfma(b[4], v[4], num);
    num = rfma(b[5], v[5], num);
    return rfma(-h2, f, num);
}
template <typename T>
__device__ __forceinline__ T gs_update(const T b[6], const T v[6], T f, T h2, T inv) {
    return rmul(gs_numerator(b, v, f, h2), inv);
}
__device__ __forceinline__ float gs_update(const float b[6], const float v[6], float f, float h2) {
    return gs_update(b, v, f, h2, gs_inverse(b));
}

// FP32 levels of at least so many cells smooth by single-pass sweeps.  A sweep moves
// half the bytes of two colour passes but takes more of the SMs' shared-memory
// pipe, so the line lies where e, f and the coefficients (20 B per cell) outgrow the
// 126 MB L2: measured, 256^3 96 us a sweep against 112 us, 160x192x224 42 against
// 46, and 128^3, out of L2, 21 against 18.
constexpr long long SWEEP_MIN_CELLS = 6LL << 20;

// With mx_opts.fused = 1 they do from so many.
constexpr long long FUSED_MIN_CELLS = 1LL << 18;
// The cells from which a level smooths by sweeps under mx_opts.fused (2: none does).
inline long long sweep_from(int fused) {
    return fused == 2 ? LLONG_MAX : (fused ? FUSED_MIN_CELLS : SWEEP_MIN_CELLS);
}

// Whether the single-pass sweep supports this level (n_x a multiple of 4, at least 32).
bool rbgs_fused_ok(const DGeom &g);

// Allow the sweep kernels their shared memory (once per device, outside any capture).
cudaError_t rbgs_init();

// e_out = one red+black sweep applied to e_in (mode RB_ZERO: e_in = 0;
// RB_PROLONG: e_in + piecewise-constant prolongation of coarse->e).
void k_rbgs_fused(cudaStream_t s, const Level<float> &L, const float *ein, float *eout, int mode,
                  const Level<float> *coarse);

// The same over a batch: work entries (box, tile x, tile y, chunk) of
// rbgs_sweep_grid(level geometry, zk), zk from rbgs_sweep_zk over the boxes; e -> e2
// (to_e2) or e2 -> e
dim3 rbgs_sweep_grid(const DGeom &g, int zk);
int rbgs_sweep_zk(int nbox, const DGeom *g);
void k_rbgs_sweep_batch(cudaStream_t s, const Level<float> *levs, const int4 *work, int nwork, const SolveState *st,
                        int level, int zero, int to_e2, int zk);
