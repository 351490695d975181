// Launch wrappers of the SP-MPS CUDA kernels (sm_103a).  All take device task arrays built
// by the host planner and a table of slot base pointers, and launch on the given stream.
#pragma once

#include <cuda_runtime.h>

#include "core.h"

namespace spmps {

// Launch item `id` of n list entries (the first n0 operator 0's) times ng beta points: operator 0's entries of
// every beta point come first, so that the long reductions of H are not left for the end of a launch.
struct LaunchItem {
    int entry, g, op;
};
__host__ __device__ inline LaunchItem launch_item(int id, int n, int n0, int ng) {
    const int first = n0 * ng;
    LaunchItem it;
    it.op = id >= first ? 1 : 0;
    const int count = it.op ? n - n0 : n0, rel = id - (it.op ? first : 0);
    it.g = rel / count;
    it.entry = rel - it.g * count + (it.op ? n0 : 0);
    return it;
}
// Entries of operator 0 among the n from `from` on.
inline int op0_entries(const BetaRun& b, int from, int n) {
    const int k = b.split - from;
    return k < 0 ? 0 : (k > n ? n : k);
}

// Grouped FP64 GEMM: one warp per tile of the task list (register tiles of 256 outputs, warp blocks of up to 256).
cudaError_t launch_gemm_f64(const Slots& slots, const GemmTask* tasks, const GemmSeg* segs,
                            const GemmTile* tiles, const int* cmaps, int n_tiles, cudaStream_t st,
                            const BetaRun& beta = BetaRun());

// out[i] = sum_{g < G} w[g] sum_{k < ks} partial[(g * ks + k) * n + i] (fixed order; w null: 1) for one or
// two outputs (a null output is left out).
cudaError_t launch_sum_partials(const double* partial0, const double* partial1, const double* w, int G, int ks0, int ks1,
                                int64_t n, double* out0, double* out1, cudaStream_t st);

// Operand buffers in pre-split TF32 form (float2 = (hi, lo) per element), indexed by the same slot
// handles as the FP64 buffers.
struct SlotsF {
    float2* p[kMaxSlots];
};
// out[i] = (tf32(float(x[i])), tf32(float(x[i]) - hi)).
cudaError_t launch_split_tf32(const double* x, int64_t n, float2* out, cudaStream_t st);
// The same task lists on the tensor cores (m16n8k8 TF32, FP32 accumulation; split3 != 0 uses the 3xTF32
// split hi*hi + hi*lo + lo*hi) with every A and B operand read from the pre-split buffers of the same
// slots; C written in FP64.
cudaError_t launch_gemm_tf32s(const Slots& slots, const SlotsF& split, const GemmTask* tasks, const GemmSeg* segs,
                              const GemmTile* tiles, const int* cmaps, int n_tiles, int split3, cudaStream_t st,
                              const BetaRun& beta);

// Linear combination of equally shaped blocks (the MPO-leg contraction).
cudaError_t launch_comb_f64(const Slots& slots, const CombOut* outs, const CombTerm* terms, int n_outs,
                            cudaStream_t st);

// Diagonal of the projected H and N operators on the two-site row-block layout.
cudaError_t launch_diag_f64(const Slots& slots, const DiagBlock* blocks, const DiagTerm* terms, int n_blocks,
                            double* dh, double* dn, cudaStream_t st);

// ---- dense vector kernels for the Davidson solver (length n, column-major bases) ----------

// out[j] = sum_i V[j*ldv + i] * x[i] for j < m (plus a scale); multi-dot with block reduction.
// `partial` is a per-caller scratch of kPartialDoubles doubles.
constexpr int kPartialDoubles = 2 * 64 * 32;
constexpr int kNormBlocks = 304;  // partial sums of launch_ritz_vectors / launch_project (two CTAs per SM)
cudaError_t launch_multidot(const double* V, int64_t ldv, int m, const double* x, int64_t n, double* out,
                            double* partial, cudaStream_t st);
// y[i] = sum_j V[j*ldv + i] * c[j]  (c on the device), optionally y -= (when sub != 0).
cudaError_t launch_gemv(const double* V, int64_t ldv, int m, const double* c, int64_t n, double* y, int sub,
                        cudaStream_t st);
// dst[:, j] = sum_i src[:, i] * Q[i + j*ldq]  for j < k (dst and src must differ).
cudaError_t launch_basis_rotate(const double* src, int64_t ld, int m, const double* Q, int ldq, int k,
                                int64_t n, double* dst, cudaStream_t st);

// Incremental Ritz step of the Davidson solver (one CTA) on the stored subspace
// matrices h, n (m x m, leading dim ldm, upper triangles column by column): lowest Ritz pair in the
// range of n kept above eps_metric * max diag(n).  The state is kept across the iterations of one
// solve; reset != 0 rebuilds it from the m stored columns.  Writes coef[0..32) (zeros beyond m; the previous
// contents go to coef_prev) and scal[0] = theta, scal[1] = number of kept metric directions (0 = singular).
struct RitzState {
    static constexpr int kR = 32;
    double X[kR * kR];   // n-orthonormal coefficient basis, X[i + j*kR]
    double hp[kR * kR];  // X^T h X
    float C[kR * kR];    // eigenvectors of hp (columns)
    int k, m, kc, pad;
};
cudaError_t launch_ritz_inc(const double* h, const double* nmat, int ldm, int m, int reset, double eps_metric,
                            RitzState* state, double* coef, double* coef_prev, double* scal, cudaStream_t st);

// One pass over the bases (leading dimension n): x = V c, hx = HV c, nx = NV c, r = hx - theta nx (theta =
// scal[0]), t = -r / (diag H - theta diag N) clamped (also into t2 unless null), block sums of |r|^2.
cudaError_t launch_ritz_vectors(const double* V, const double* HV, const double* NV, int64_t n, int m, const double* coef,
                                const double* dh, const double* dn, const double* scal, double clamp, double* x,
                                double* hx, double* nx, double* r, double* t, double* t2, double* sums, cudaStream_t st);
// y -= V V^T y (one pass of classical Gram-Schmidt against m vectors); block sums of |y|^2 unless null.
cudaError_t launch_project(const double* V, int64_t n, int m, double* y, double* partial, double* sums, cudaStream_t st);
// *out = sum of the block sums of a vector of length n.
cudaError_t launch_sum_blocks(const double* sums, int64_t n, double* out, cudaStream_t st);
// y /= |y| from the block sums of |y|^2 (their sum to *yy); the sum of rsums (unless null) to *rr.
cudaError_t launch_normalise(double* y, int64_t n, const double* ysums, const double* rsums, double* yy, double* rr,
                             cudaStream_t st);
// out0[j] = V_j . x0 and out1[j] = V_j . x1 for j < m.
cudaError_t launch_multidot2(const double* V, int64_t ldv, int m, const double* x0, const double* x1, int64_t n,
                             double* out0, double* out1, double* partial, cudaStream_t st);
// sum of squares into *out (two-pass deterministic reduction).
cudaError_t launch_norm2(const double* x, int64_t n, double* out, double* partial, cudaStream_t st);
// x *= 1/sqrt(*nrm2) (device scalar)
cudaError_t launch_scale_inv_sqrt(double* x, int64_t n, const double* nrm2, cudaStream_t st);
// x += alpha * y, alpha = sign * num / den from device scalars (for CG)
// out = v / (diag H - theta diag N) (denominator clamped to |.| >= clamp; theta = scal[0])
cudaError_t launch_precond_apply(const double* v, const double* dh, const double* dn, const double* scal,
                                 double clamp, int64_t n, double* out, cudaStream_t st);
cudaError_t launch_axpy_ratio(double* x, const double* y, int64_t n, const double* num, const double* den,
                              double sign, cudaStream_t st);
// p = r + (num/den) p
cudaError_t launch_xpby_ratio(double* p, const double* r, int64_t n, const double* num, const double* den,
                              cudaStream_t st);
// Two-vector orthonormal restart coefficients in the current basis: Qout (m x 2) from the
// Ritz coefficients c_new and c_old (m each); the count to scal_out[0]; c_new (32 entries) becomes the
// coefficients of the same vector in the restarted basis.
cudaError_t launch_restart_coef(double* c_new, const double* c_old, int m, double* Qout, double* scal_out,
                                cudaStream_t st);

// ---- decimation -------------------------------------------------------------------------------

// Ordered truncation of the singular values sqrt(max(evals, 0)): evals holds the values of all labels
// in label order (label l from val_off[l]), labels ascending in (n, 2m).  Values within tie_rtol * max of
// their sorted predecessor form a cluster ordered by (n, 2m, index); values below drop_abs are dropped;
// the first D kept.  keep_count[label] receives the number kept per label, keep_total[0] the total and
// discarded[0] the discarded weight.  Scratch: 3 total ints and 2 total doubles.
cudaError_t launch_truncate(const double* evals, const int64_t* val_off, int n_labels, int total, int D, double tie_rtol,
                            double drop_abs, int* keep_count, int* keep_total, double* discarded, int* scratch_idx,
                            double* scratch_val, cudaStream_t st);

// Gather/scatter of sub-blocks: dst[(r)*ld_dst + c] = src[(r)*ld_src + c] * scale for a list.
struct CopyBlock {
    uint64_t src, dst;
    int rows, cols, ld_src, ld_dst;
    int transpose;  // 1: dst(r, c) = src(c, r)
    int pad;
};
cudaError_t launch_copy_blocks(const Slots& slots, const CopyBlock* blocks, int n, cudaStream_t st);

// FP64 FMA throughput of the current device (TFLOP/s), from a kernel of independent chains.
cudaError_t measure_fp64_peak(double* tflops);

}  // namespace spmps
