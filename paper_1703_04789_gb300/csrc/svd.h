// Batched singular vectors of the decimation blocks (svd.cu).
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <vector>

namespace spmps {

constexpr int kSvdConv = 256;           // sweep flags per block and precision
constexpr int kSvdMaxSweeps = 250;      // of the FP64 finish: 5 in the blocks of random states, up to 90 in 700 rows with
                                        // singular values over 14 decades
constexpr int kSvdMaxRows = 1024;       // rows that a block's rotations may act on (their list in shared memory)
constexpr int kSvdSmemFloats = 56000;   // FP32 start in shared memory: [Z | I] and the row norms (219 KB)
constexpr int kSvdSmemDefault = 112;    // limit on the dimension at which no limit is meant

// A block X of dim x other; the left singular vectors (dim of them) are wanted.
struct SvdShape {
    int dim, other;
};
struct SvdBlock {
    int R, C, dim;   // rows and columns that the rotations act on
    int companion;   // 1: rows are X's, their rotations are the vectors; 0: rows are X^T's
    int smem;        // FP32 start in shared memory
    int pad;
    int64_t z_off, j_off, f_off, w_off, n_off;  // input, J, Z', FP32 work, row norms
    int64_t m_off, e_off;                       // vectors (dim x dim) and values (dim)
};
struct SvdGemm {
    int64_t a, b, c;
    int M, N, K, lda, ldb, ldc, transb, pad;
    double alpha, diag;
};

struct SvdPlan {
    std::vector<SvdBlock> blocks;
    std::vector<SvdGemm> gemms;
    std::vector<int3> tiles;
    std::vector<int> gemm_rng;
    int64_t z_size = 0, j_size = 0, f_size = 0, w_size = 0, n_size = 0;
    int smem_floats = 0, max_rows = 0;  // of the blocks that start in shared memory
    int most_rows = 0;                  // of all blocks
    int max_sweeps = kSvdMaxSweeps;     // of the FP64 finish
    bool any_smem = false, any_global = false, any_companion = false;
    // blocks of dimension up to smem_dim may start in shared memory (kSvdSmemDefault: all that fit)
    void build(const std::vector<SvdShape>& shapes, int smem_dim);
    size_t workspace() const;             // bytes of launch_svd's workspace
    double* z_buffer(void* ws) const;     // the input rows inside it: block b's R x C at z_off, row-major
};

// Singular values squared (descending, dim per block at e_off) and left singular vectors (columns of the
// dim x dim row-major matrix at m_off, in the same order; zero columns beyond the rank when the
// transpose was the smaller side) of every block.  The caller has written the rows (X, or X^T where
// companion is 0) into z_buffer(ws).  *unsettled (device) becomes 1 where a block still had coupled rows when
// its sweeps ended: its vectors are then not orthonormal to rounding.  cudaErrorInvalidValue, and nothing
// launched, for a block of more than kSvdMaxRows rows or more than kSvdConv sweeps.
cudaError_t launch_svd(const SvdPlan& P, void* ws, double* mats, double* evals, int* unsettled, cudaStream_t st);

}  // namespace spmps
