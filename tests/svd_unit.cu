// C entries over one block of svd.cu, for tests/test_svd_unit.py.
#include "svd.h"

using namespace spmps;

// launch_svd of a block of dim x other without any buffer.
extern "C" int svd_launch_empty(int dim, int other, int max_sweeps) {
    SvdPlan P;
    P.build({{dim, other}}, kSvdSmemDefault);
    P.max_sweeps = max_sweeps;
    return launch_svd(P, nullptr, nullptr, nullptr, nullptr, nullptr);
}

// Singular values squared and left vectors (columns of dim x dim) of x (dim x other, row-major, host).
extern "C" int svd_block(int dim, int other, int max_sweeps, const double* x, double* evals, double* mats, int* unsettled) {
    SvdPlan P;
    P.build({{dim, other}}, kSvdSmemDefault);
    P.max_sweeps = max_sweeps;
    std::vector<double> z(static_cast<size_t>(dim) * other);
    const SvdBlock& B = P.blocks[0];
    for (int r = 0; r < B.R; ++r)
        for (int c = 0; c < B.C; ++c) z[static_cast<size_t>(r) * B.C + c] = B.companion ? x[r * other + c] : x[c * other + r];
    void *ws = nullptr, *m = nullptr, *e = nullptr, *u = nullptr;
    const size_t mb = sizeof(double) * dim * dim, eb = sizeof(double) * dim;
    cudaError_t st = cudaMalloc(&ws, P.workspace());
    if (st == cudaSuccess) st = cudaMalloc(&m, mb);
    if (st == cudaSuccess) st = cudaMalloc(&e, eb);
    if (st == cudaSuccess) st = cudaMalloc(&u, sizeof(int));
    if (st == cudaSuccess) st = cudaMemset(u, 0, sizeof(int));
    if (st == cudaSuccess) st = cudaMemcpy(P.z_buffer(ws), z.data(), z.size() * sizeof(double), cudaMemcpyHostToDevice);
    if (st == cudaSuccess) st = launch_svd(P, ws, static_cast<double*>(m), static_cast<double*>(e), static_cast<int*>(u), nullptr);
    if (st == cudaSuccess) st = cudaMemcpy(evals, e, eb, cudaMemcpyDeviceToHost);
    if (st == cudaSuccess) st = cudaMemcpy(mats, m, mb, cudaMemcpyDeviceToHost);
    if (st == cudaSuccess) st = cudaMemcpy(unsettled, u, sizeof(int), cudaMemcpyDeviceToHost);
    cudaFree(ws);
    cudaFree(m);
    cudaFree(e);
    cudaFree(u);
    return st;
}
