// CUDA kernels of the SP-MPS library (sm_103a, FP64).
//
// The contractions of the projected action and of the environment updates are lists of small
// dense block products produced by the host planner (Abelian (N, M) blocks on the bra side,
// N-only blocks on the rotated ket side).  They run as grouped launches: one warp per output
// tile of any task, every task of every beta point in the same launch.
#include <cfloat>
#include <cmath>

#include "kernels.h"
#include "tc_gemm.h"

namespace spmps {

namespace {

__device__ __forceinline__ double* resolve(const Slots& S, uint64_t h) {
    return S.p[h >> 56] + static_cast<int64_t>(h & 0x00FFFFFFFFFFFFFFull);
}

__device__ __forceinline__ void cp_async8(double* dst, const double* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
                 "l"(src));
}

__device__ __forceinline__ double* resolve(double* const* base, uint64_t h) {
    return base[h >> 56] + static_cast<int64_t>(h & 0x00FFFFFFFFFFFFFFull);
}

// This warp's base pointers (its beta point and operator) into its row of a shared table.
__device__ __forceinline__ double* const* warp_bases(const Slots& S, const BetaStride& B, int op, int g,
                                                     double* (*table)[kMaxSlots]) {
    const int lane = threadIdx.x & 31;
    double** mine = table[threadIdx.x >> 5];
    if (lane < kMaxSlots) mine[lane] = S.p[lane] + g * B.s[op][lane];
    __syncwarp();
    return mine;
}

// ---- grouped FP64 GEMM ----------------------------------------------------------------------
// Tile shapes (rows x cols per warp; each lane owns RM x CN outputs on a LR x LC lane grid):
//   0: 16 x 16  (LR 8, LC 4, RM 2, CN 4)      1: 4 x 64  (LR 4, LC 8, RM 1, CN 8)
//   2: 64 x 4   (LR 8, LC 4, RM 8, CN 1)      3: 32 x 8  (LR 8, LC 4, RM 4, CN 2)
//   4: 8 x 32   (LR 4, LC 8, RM 2, CN 4)
template <int LR, int LC, int RM, int CN>
__device__ __forceinline__ void gemm_tile(double* const* S, const GemmTask& T, const GemmSeg* __restrict__ segs,
                                          const int* __restrict__ cmaps, int m0, int n0, int lane) {
    const int lr = lane / LC, lc = lane % LC;
    int rows[RM], cols[CN];
    bool rv[RM], cv[CN];
#pragma unroll
    for (int i = 0; i < RM; ++i) {
        rows[i] = m0 + lr + i * LR;
        rv[i] = rows[i] < T.M;
    }
#pragma unroll
    for (int j = 0; j < CN; ++j) {
        cols[j] = n0 + lc + j * LC;
        cv[j] = cols[j] < T.N;
    }
    double acc[RM][CN];
#pragma unroll
    for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < CN; ++j) acc[i][j] = 0.0;

    for (int sgi = 0; sgi < T.nseg; ++sgi) {
        const GemmSeg sg = segs[T.seg0 + sgi];
        const double* __restrict__ A = resolve(S, sg.a);
        const double* __restrict__ B = resolve(S, sg.b);
        for (int k = 0; k < sg.K; ++k) {
            double a[RM], b[CN];
#pragma unroll
            for (int i = 0; i < RM; ++i)
                a[i] = rv[i] ? __ldg(A + static_cast<int64_t>(rows[i]) * sg.a_rs + static_cast<int64_t>(k) * sg.a_cs)
                             : 0.0;
#pragma unroll
            for (int j = 0; j < CN; ++j)
                b[j] = cv[j] ? __ldg(B + static_cast<int64_t>(k) * sg.b_rs + static_cast<int64_t>(cols[j]) * sg.b_cs)
                             : 0.0;
#pragma unroll
            for (int i = 0; i < RM; ++i)
#pragma unroll
                for (int j = 0; j < CN; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
        }
    }
    double* C = resolve(S, T.c);
    const int* cm = T.cmap >= 0 ? cmaps + T.cmap : nullptr;
#pragma unroll
    for (int j = 0; j < CN; ++j) {
        if (!cv[j]) continue;
        const int64_t cc = cm ? cm[cols[j]] : cols[j];
#pragma unroll
        for (int i = 0; i < RM; ++i)
            if (rv[i]) C[static_cast<int64_t>(rows[i]) * T.ldc + cc] = acc[i][j];
    }
}

// Warp-block tile (shape 5): one warp computes a whole tm x tn output block (tm, tn <= 32,
// tm * tn <= 256).  K is staged in chunks of 8 through the warp's two shared-memory slices by asynchronous
// copies (four rows of 8 k per warp step), the next chunk (of the same or the next segment) in flight while
// every lane accumulates its flattened outputs o = lane + 32 q (q < NQ) from the current one, so the
// operand rows are read once per block and no FMA is spent on padding beyond the last partial row of 32
// outputs.
constexpr int kWbK = 8;                     // K chunk
constexpr int kWbStride = kWbK + 1;         // padded row stride of the staged chunks
constexpr int kWbSlice = 2 * 32 * kWbStride;     // doubles of one stage (A rows and B rows)
constexpr int kWbWarpSmem = 2 * kWbSlice;        // per warp

template <int NQ>
__device__ __forceinline__ void gemm_tile_wb(double* const* S, const GemmTask& T, const GemmSeg* __restrict__ segs,
                                             const int* __restrict__ cmaps, int m0, int n0, int tm, int tn, int lane,
                                             double* __restrict__ sm) {
    const int nout = tm * tn;
    double v[NQ];
    int oa[NQ], ob[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        v[q] = 0.0;
        const int o = lane + 32 * q;
        const int oo = o < nout ? o : 0;
        oa[q] = (oo / tn) * kWbStride;
        ob[q] = (32 + oo % tn) * kWbStride;
    }
    const int kl = lane & (kWbK - 1), rl = lane >> 3;
    GemmSeg sg{};
    if (T.nseg > 0) sg = segs[T.seg0];
    // chunk k0 of segment sg into slice buf
    auto issue = [&](int k0, int buf) {
        const double* A = resolve(S, sg.a) + static_cast<int64_t>(m0 + rl) * sg.a_rs + static_cast<int64_t>(k0 + kl) * sg.a_cs;
        const double* B = resolve(S, sg.b) + static_cast<int64_t>(n0 + rl) * sg.b_cs + static_cast<int64_t>(k0 + kl) * sg.b_rs;
        const bool kv = k0 + kl < sg.K;
        double* As = sm + buf * kWbSlice + rl * kWbStride + kl;
#pragma unroll 4
        for (int i = 0; i < 8; ++i) {
            if (rl + 4 * i < tm) {
                if (kv)
                    cp_async8(As + 4 * i * kWbStride, A + static_cast<int64_t>(4 * i) * sg.a_rs);
                else
                    As[4 * i * kWbStride] = 0.0;
            }
            if (rl + 4 * i < tn) {
                double* Bs = As + 32 * kWbStride;
                if (kv)
                    cp_async8(Bs + 4 * i * kWbStride, B + static_cast<int64_t>(4 * i) * sg.b_cs);
                else
                    Bs[4 * i * kWbStride] = 0.0;
            }
        }
    };
    int sgi = 0, k0 = 0, kc = 0;  // kc: length of the chunk in flight
    for (int t = 0;; ++t) {
        int next = 0;
        if (sgi < T.nseg) {
            issue(k0, t & 1);
            next = min(kWbK, sg.K - k0);
            k0 += kWbK;
            if (k0 >= sg.K) {
                ++sgi;
                k0 = 0;
                if (sgi < T.nseg) sg = segs[T.seg0 + sgi];
            }
        }
        asm volatile("cp.async.commit_group;");
        if (t > 0) {
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            __syncwarp();
            const double* st = sm + ((t - 1) & 1) * kWbSlice;
#pragma unroll 2
            for (int kk = 0; kk < kc; ++kk) {
#pragma unroll
                for (int q = 0; q < NQ; ++q) v[q] = fma(st[oa[q] + kk], st[ob[q] + kk], v[q]);
            }
            __syncwarp();
        }
        if (next == 0) break;
        kc = next;
    }
    double* C = resolve(S, T.c);
    const int* cm = T.cmap >= 0 ? cmaps + T.cmap : nullptr;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const int o = lane + 32 * q;
        if (o < nout) {
            const int i = o / tn, j = o % tn;
            const int64_t cc = cm ? cm[n0 + j] : n0 + j;
            C[static_cast<int64_t>(m0 + i) * T.ldc + cc] = v[q];
        }
    }
}

__global__ void __launch_bounds__(128, 5) k_gemm_f64(const __grid_constant__ Slots P, const __grid_constant__ BetaStride Bs,
                                                     int n0, int g0, int ng, const GemmTask* __restrict__ tasks,
                                                     const GemmSeg* __restrict__ segs, const GemmTile* __restrict__ tiles,
                                                     const int* __restrict__ cmaps, int n_tiles) {
    __shared__ double wb_smem[4 * kWbWarpSmem];
    __shared__ double* table[4][kMaxSlots];
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (warp >= n_tiles * ng) return;
    const LaunchItem it = launch_item(warp, n_tiles, n0, ng);
    const GemmTile tl = tiles[it.entry];
    const GemmTask T = tasks[tl.task];
    double* const* S = warp_bases(P, Bs, it.op, g0 + it.g, table);
    if (tl.shape == 5) {
        double* sm = wb_smem + (threadIdx.x >> 5) * kWbWarpSmem;
        const int nq = (tl.tm * tl.tn + 31) / 32;
        switch (nq) {
            case 1: gemm_tile_wb<1>(S, T, segs, cmaps, tl.m0, tl.n0, tl.tm, tl.tn, lane, sm); break;
            case 2: gemm_tile_wb<2>(S, T, segs, cmaps, tl.m0, tl.n0, tl.tm, tl.tn, lane, sm); break;
            case 3: gemm_tile_wb<3>(S, T, segs, cmaps, tl.m0, tl.n0, tl.tm, tl.tn, lane, sm); break;
            case 4: gemm_tile_wb<4>(S, T, segs, cmaps, tl.m0, tl.n0, tl.tm, tl.tn, lane, sm); break;
            case 5: gemm_tile_wb<5>(S, T, segs, cmaps, tl.m0, tl.n0, tl.tm, tl.tn, lane, sm); break;
            case 6: gemm_tile_wb<6>(S, T, segs, cmaps, tl.m0, tl.n0, tl.tm, tl.tn, lane, sm); break;
            case 7: gemm_tile_wb<7>(S, T, segs, cmaps, tl.m0, tl.n0, tl.tm, tl.tn, lane, sm); break;
            default: gemm_tile_wb<8>(S, T, segs, cmaps, tl.m0, tl.n0, tl.tm, tl.tn, lane, sm); break;
        }
        return;
    }
    switch (tl.shape) {
        case 1: gemm_tile<4, 8, 1, 8>(S, T, segs, cmaps, tl.m0, tl.n0, lane); break;
        case 2: gemm_tile<8, 4, 8, 1>(S, T, segs, cmaps, tl.m0, tl.n0, lane); break;
        case 3: gemm_tile<8, 4, 4, 2>(S, T, segs, cmaps, tl.m0, tl.n0, lane); break;
        case 4: gemm_tile<4, 8, 2, 4>(S, T, segs, cmaps, tl.m0, tl.n0, lane); break;
        default: gemm_tile<8, 4, 2, 4>(S, T, segs, cmaps, tl.m0, tl.n0, lane); break;
    }
}

// ---- stacked FP64 GEMM ------------------------------------------------------------------------
// The stacks of tc_gemm.h on the FP64 pipe, for the long reductions of phase C: every output row of all
// blocks that read the same rows of the right environment, so that a warp's tile (tm x tn outputs of a
// stack, <= 256) is full although most blocks are only a few rows high.  The K segments (one per channel)
// are walked as one reduction in chunks of 8: lane kl of a chunk keeps its own position (segment, k), so
// no chunk is cut short at a segment's end.  Double-buffered asynchronous copies as in gemm_tile_wb.  Bound by
// the FP64 pipe.  Measured (GB300, phase C of the middle action of the L = 24, D = 256
// chain, 494 Mflop): 0.494 ms; one block at a time per warp took 0.647 ms (28 % of the lanes idle).
template <int NQ>
__device__ __forceinline__ void stack_tile(double* const* S, const TcStack& st, const TcRow* __restrict__ rows,
                                           const TcSeg* __restrict__ segs, const uint64_t* __restrict__ atab,
                                           const int* __restrict__ cmaps, int m0, int n0, int tm, int tn, int lane,
                                           double* __restrict__ sm) {
    const int nout = tm * tn;
    double v[NQ];
    int oa[NQ], ob[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        v[q] = 0.0;
        const int o = lane + 32 * q;
        const int oo = o < nout ? o : 0;
        oa[q] = (oo / tn) * kWbStride;
        ob[q] = (32 + oo % tn) * kWbStride;
    }
    const int kl = lane & (kWbK - 1), rl = lane >> 3;
    int s = -1, k = kl, K = 0;  // this lane's segment and position in it; past the end: s = nseg
    const double* B = nullptr;
    int64_t b_ks = 0, b_ns = 0;
    int left = st.ktot;  // of the whole reduction
    int kc = 0;
    for (int t = 0;; ++t) {
        if (left > 0) {
            while (s < st.nseg && k >= K) {
                k -= K;
                if (++s < st.nseg) {
                    const TcSeg sg = segs[st.seg0 + s];
                    K = sg.K;
                    b_ks = sg.b_ks;
                    b_ns = sg.b_ns;
                    B = resolve(S, sg.b);
                }
            }
            const bool kv = s < st.nseg;
            const uint64_t* at = atab + st.atab0 + static_cast<int64_t>(m0 + rl) * st.nseg + (kv ? s : 0);
            const double* bp = kv ? B + static_cast<int64_t>(n0 + rl) * b_ns + k * b_ks : nullptr;
            double* As = sm + (t & 1) * kWbSlice + rl * kWbStride + kl;
#pragma unroll 4
            for (int i = 0; i < 8; ++i) {
                if (rl + 4 * i < tm) {
                    const uint64_t h = kv ? __ldg(at + static_cast<int64_t>(4 * i) * st.nseg) : kNoOperand;
                    if (h != kNoOperand)
                        cp_async8(As + 4 * i * kWbStride, resolve(S, h) + k);
                    else
                        As[4 * i * kWbStride] = 0.0;
                }
                if (rl + 4 * i < tn) {
                    double* Bs = As + 32 * kWbStride;
                    if (kv)
                        cp_async8(Bs + 4 * i * kWbStride, bp + 4 * i * b_ns);
                    else
                        Bs[4 * i * kWbStride] = 0.0;
                }
            }
            k += kWbK;
        }
        asm volatile("cp.async.commit_group;");
        if (t > 0) {
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            __syncwarp();
            const double* sc = sm + ((t - 1) & 1) * kWbSlice;
#pragma unroll 2
            for (int kk = 0; kk < kc; ++kk) {
#pragma unroll
                for (int q = 0; q < NQ; ++q) v[q] = fma(sc[oa[q] + kk], sc[ob[q] + kk], v[q]);
            }
            __syncwarp();
        }
        if (left <= 0) break;
        kc = min(kWbK, left);
        left -= kWbK;
    }
    const int* cm = st.cmap >= 0 ? cmaps + st.cmap : nullptr;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const int o = lane + 32 * q;
        if (o < nout) {
            const int i = o / tn, n = n0 + o % tn;
            resolve(S, rows[st.row0 + m0 + i].c)[cm ? cm[n] : n] = v[q];
        }
    }
}

__global__ void __launch_bounds__(128, 5) k_gemm_f64_stack(const __grid_constant__ Slots P,
                                                           const __grid_constant__ BetaStride Bs, int n0, int g0, int ng,
                                                           const TcStack* __restrict__ stacks,
                                                           const TcRow* __restrict__ rows, const TcSeg* __restrict__ segs,
                                                           const uint64_t* __restrict__ atab, const int* __restrict__ cmaps,
                                                           const int4* __restrict__ units, int u0, int u1) {
    __shared__ double smem[4 * kWbWarpSmem];
    __shared__ double* table[4][kMaxSlots];
    const int id = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (id >= (u1 - u0) * ng) return;
    const LaunchItem it = launch_item(id, u1 - u0, n0, ng);
    const int4 U = units[u0 + it.entry];
    const TcStack st = stacks[U.x];
    const int tm = U.w & 0xFFFF, tn = U.w >> 16;
    double* const* S = warp_bases(P, Bs, it.op, g0 + it.g, table);
    double* sm = smem + (threadIdx.x >> 5) * kWbWarpSmem;
    switch ((tm * tn + 31) / 32) {
        case 1: stack_tile<1>(S, st, rows, segs, atab, cmaps, U.y, U.z, tm, tn, lane, sm); break;
        case 2: stack_tile<2>(S, st, rows, segs, atab, cmaps, U.y, U.z, tm, tn, lane, sm); break;
        case 3:
        case 4: stack_tile<4>(S, st, rows, segs, atab, cmaps, U.y, U.z, tm, tn, lane, sm); break;
        case 5:
        case 6: stack_tile<6>(S, st, rows, segs, atab, cmaps, U.y, U.z, tm, tn, lane, sm); break;
        case 7: stack_tile<7>(S, st, rows, segs, atab, cmaps, U.y, U.z, tm, tn, lane, sm); break;
        default: stack_tile<8>(S, st, rows, segs, atab, cmaps, U.y, U.z, tm, tn, lane, sm); break;
    }
}

// ---- beta reduction of the output partials ------------------------------------------------------
// Partials of beta point g: ks consecutive slices of n values (the slices of the channels).
__global__ void __launch_bounds__(256) k_sum_partials(const double* __restrict__ p0, const double* __restrict__ p1,
                                                      const double* __restrict__ w, int G, int ks0, int ks1, int64_t n,
                                                      double* __restrict__ out0, double* __restrict__ out1) {
    const double* __restrict__ partial = blockIdx.y == 0 ? p0 : p1;
    double* __restrict__ out = blockIdx.y == 0 ? out0 : out1;
    const int ks = blockIdx.y == 0 ? ks0 : ks1;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        double acc = 0.0;
        for (int g = 0; g < G; ++g) {
            const double* __restrict__ p = partial + static_cast<int64_t>(g) * ks * n + i;
            double s = p[0];
#pragma unroll 4
            for (int k = 1; k < ks; ++k) s += p[k * n];
            acc = fma(w ? __ldg(w + g) : 1.0, s, acc);
        }
        out[i] = acc;
    }
}

// ---- block linear combination (MPO legs) ------------------------------------------------------
__global__ void __launch_bounds__(256) k_comb_f64(const __grid_constant__ Slots S, const CombOut* __restrict__ outs,
                                                  const CombTerm* __restrict__ terms, int n_outs) {
    const int ob = blockIdx.x;
    if (ob >= n_outs) return;
    const CombOut o = outs[ob];
    double* dst = resolve(S, o.dst);
    const int n = o.rows * o.cols;
    for (int e = threadIdx.x; e < n; e += blockDim.x) {
        const int r = e / o.cols, c = e - r * o.cols;
        double acc = 0.0;
        for (int t = 0; t < o.nterm; ++t) {
            const CombTerm tm = terms[o.term0 + t];
            acc = fma(tm.coef, __ldg(resolve(S, tm.src) + static_cast<int64_t>(r) * tm.ld + c), acc);
        }
        dst[static_cast<int64_t>(r) * o.ld + c] = acc;
    }
}

// ---- diagonal of the projected operators ------------------------------------------------------
__global__ void __launch_bounds__(256) k_diag_f64(const __grid_constant__ Slots S, const DiagBlock* __restrict__ blocks,
                                                  const DiagTerm* __restrict__ terms, int n_blocks, double* dh,
                                                  double* dn) {
    const int bi = blockIdx.x;
    if (bi >= n_blocks) return;
    const DiagBlock b = blocks[bi];
    double* out = b.out == 0 ? dh : dn;
    const int n = b.rows * b.cols;
    for (int e = threadIdx.x; e < n; e += blockDim.x) {
        const int i = e / b.cols, j = e - i * b.cols;
        double acc = 0.0;
        for (int t = 0; t < b.nterm; ++t) {
            const DiagTerm tm = terms[b.term0 + t];
            acc = fma(tm.coef * resolve(S, tm.l)[static_cast<int64_t>(i) * tm.l_step],
                      resolve(S, tm.r)[static_cast<int64_t>(j) * tm.r_step], acc);
        }
        out[b.off + static_cast<int64_t>(i) * b.ld + j] = acc;
    }
}

// ---- reductions and vector kernels ------------------------------------------------------------
__device__ double block_sum(double v, double* sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) sh[w] = v;
    __syncthreads();
    const int nw = (blockDim.x + 31) >> 5;
    v = threadIdx.x < nw ? sh[threadIdx.x] : 0.0;
    if (w == 0)
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    __syncthreads();
    return v;  // valid in thread 0
}

constexpr int kRedBlocks = 64;

// partial[j * kRedBlocks + b] = sum over chunk b of V[:, j] . x
__global__ void __launch_bounds__(256) k_multidot_partial(const double* __restrict__ V, int64_t ldv,
                                                          const double* __restrict__ x, int64_t n,
                                                          double* __restrict__ partial) {
    __shared__ double sh[32];
    const int j = blockIdx.y;
    const double* v = V + j * ldv;
    double acc = 0.0;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        acc = fma(v[i], x[i], acc);
    acc = block_sum(acc, sh);
    if (threadIdx.x == 0) partial[j * kRedBlocks + blockIdx.x] = acc;
}
__global__ void k_multidot_final(const double* __restrict__ partial, int nb, double* __restrict__ out) {
    // one warp per output, fixed summation order
    const int j = blockIdx.x;
    const int lane = threadIdx.x;
    double acc = 0.0;
    for (int b = lane; b < nb; b += 32) acc += partial[j * kRedBlocks + b];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (lane == 0) out[j] = acc;
}

// The same for two right-hand sides (blockIdx.z) in one launch each.
__global__ void __launch_bounds__(256) k_multidot2_partial(const double* __restrict__ V, int64_t ldv,
                                                           const double* __restrict__ x0, const double* __restrict__ x1,
                                                           int64_t n, double* __restrict__ partial) {
    __shared__ double sh[32];
    const int j = blockIdx.y;
    const double* v = V + j * ldv;
    const double* x = blockIdx.z == 0 ? x0 : x1;
    double acc = 0.0;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        acc = fma(v[i], x[i], acc);
    acc = block_sum(acc, sh);
    if (threadIdx.x == 0) partial[(blockIdx.z * gridDim.y + j) * kRedBlocks + blockIdx.x] = acc;
}
__global__ void k_multidot2_final(const double* __restrict__ partial, int nb, double* __restrict__ out0,
                                  double* __restrict__ out1) {
    const int j = blockIdx.x, lane = threadIdx.x;
    const double* p = partial + (blockIdx.y * gridDim.x + j) * kRedBlocks;
    double acc = 0.0;
    for (int b = lane; b < nb; b += 32) acc += p[b];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (lane == 0) (blockIdx.y == 0 ? out0 : out1)[j] = acc;
}

__global__ void __launch_bounds__(256) k_gemv(const double* __restrict__ V, int64_t ldv, int m,
                                              const double* __restrict__ c, int64_t n, double* __restrict__ y,
                                              int sub) {
    __shared__ double cs[64];
    if (threadIdx.x < m) cs[threadIdx.x] = c[threadIdx.x];
    __syncthreads();
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        double acc = 0.0;
        for (int j = 0; j < m; ++j) acc = fma(V[j * ldv + i], cs[j], acc);
        y[i] = sub ? y[i] - acc : acc;
    }
}

__global__ void __launch_bounds__(256) k_basis_rotate(const double* __restrict__ src, int64_t ld, int m,
                                                      const double* __restrict__ Q, int ldq, int k, int64_t n,
                                                      double* __restrict__ dst) {
    __shared__ double qs[64 * 4];
    for (int e = threadIdx.x; e < m * k; e += blockDim.x) {
        const int i = e % m, j = e / m;
        qs[j * 64 + i] = Q[i + j * ldq];
    }
    __syncthreads();
    for (int64_t r = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; r < n;
         r += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        for (int j = 0; j < k; ++j) {
            double acc = 0.0;
            for (int i = 0; i < m; ++i) acc = fma(src[i * ld + r], qs[j * 64 + i], acc);
            dst[j * ld + r] = acc;
        }
    }
}

__global__ void __launch_bounds__(256) k_norm2_partial(const double* __restrict__ x, int64_t n,
                                                       double* __restrict__ partial) {
    __shared__ double sh[32];
    double acc = 0.0;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        acc = fma(x[i], x[i], acc);
    acc = block_sum(acc, sh);
    if (threadIdx.x == 0) partial[blockIdx.x] = acc;
}

__global__ void __launch_bounds__(256) k_scale_inv_sqrt(double* __restrict__ x, int64_t n,
                                                        const double* __restrict__ nrm2) {
    const double v = *nrm2;
    const double s = v > 1e-300 ? 1.0 / sqrt(v) : 0.0;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        x[i] *= s;
}

// The vectors of one Davidson iteration in one pass over the bases: x = V c, H x = HV c, N x = NV c, the
// residual r, its diagonal correction t (also into t2 where given) and block sums of |r|^2.  Bound by the
// 3 m vectors it reads (L2 at the sizes of a chain).  Measured (GB300, L = 16, D = 64 step): the vector
// kernels of an iteration take 39 us in 6 launches, 79 us in 14 launches and copies before.
__global__ void __launch_bounds__(256) k_ritz_vectors(const double* __restrict__ V, const double* __restrict__ HV,
                                                      const double* __restrict__ NV, int64_t n, int m,
                                                      const double* __restrict__ coef, const double* __restrict__ dh,
                                                      const double* __restrict__ dn, const double* __restrict__ scal,
                                                      double clamp, double* __restrict__ x, double* __restrict__ hx,
                                                      double* __restrict__ nx, double* __restrict__ r,
                                                      double* __restrict__ t, double* __restrict__ t2,
                                                      double* __restrict__ sums) {
    __shared__ double cs[32], sh[32];
    if (threadIdx.x < m) cs[threadIdx.x] = coef[threadIdx.x];
    __syncthreads();
    const double theta = scal[0];
    double rr = 0.0;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        double a = 0.0, b = 0.0, c = 0.0;
#pragma unroll 4
        for (int j = 0; j < m; ++j) {
            a = fma(V[j * n + i], cs[j], a);
            b = fma(HV[j * n + i], cs[j], b);
            c = fma(NV[j * n + i], cs[j], c);
        }
        x[i] = a;
        hx[i] = b;
        nx[i] = c;
        const double ri = b - theta * c;
        r[i] = ri;
        double den = dh[i] - theta * dn[i];
        if (fabs(den) < clamp) den = den < 0.0 ? -clamp : clamp;
        const double ti = -ri / den;
        t[i] = ti;
        if (t2) t2[i] = ti;
        rr = fma(ri, ri, rr);
    }
    rr = block_sum(rr, sh);
    if (threadIdx.x == 0) sums[blockIdx.x] = rr;
}

// y -= V d with d_j the sum of the nb block sums of k_multidot_partial (same order as k_multidot_final);
// block sums of |y|^2 where `sums` is given.
__global__ void __launch_bounds__(256) k_project(const double* __restrict__ V, int64_t n, int m,
                                                 const double* __restrict__ partial, int nb, double* __restrict__ y,
                                                 double* __restrict__ sums) {
    __shared__ double cs[32], sh[32];
    const int lane = threadIdx.x & 31;
    for (int j = threadIdx.x >> 5; j < m; j += 8) {
        double d = 0.0;
        for (int b = lane; b < nb; b += 32) d += partial[j * kRedBlocks + b];
        for (int o = 16; o > 0; o >>= 1) d += __shfl_down_sync(0xffffffffu, d, o);
        if (lane == 0) cs[j] = d;
    }
    __syncthreads();
    double yy = 0.0;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        double acc = 0.0;
#pragma unroll 4
        for (int j = 0; j < m; ++j) acc = fma(V[j * n + i], cs[j], acc);
        const double v = y[i] - acc;
        y[i] = v;
        yy = fma(v, v, yy);
    }
    if (sums) {
        yy = block_sum(yy, sh);
        if (threadIdx.x == 0) sums[blockIdx.x] = yy;
    }
}

// Sum of nb block sums by one warp, fixed order (valid in lane 0).
__device__ __forceinline__ double sum_blocks(const double* __restrict__ s, int nb) {
    double v = 0.0;
    for (int b = threadIdx.x & 31; b < nb; b += 32) v += s[b];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// out[0] = sum of the block sums.
__global__ void k_sum_blocks(const double* __restrict__ s, int nb, double* __restrict__ out) {
    const double v = sum_blocks(s, nb);
    if (threadIdx.x == 0) out[0] = v;
}

// y scaled to norm 1 by the block sums of |y|^2 (nyb of them), which also goes to yy; where rsums is
// given, the sum of those goes to rr.
__global__ void __launch_bounds__(256) k_normalise(double* __restrict__ y, int64_t n, const double* __restrict__ ysums,
                                                   int nyb, const double* __restrict__ rsums, int nrb,
                                                   double* __restrict__ yy, double* __restrict__ rr) {
    __shared__ double sc;
    if (threadIdx.x < 32) {
        const double v = sum_blocks(ysums, nyb);
        if (threadIdx.x == 0) {
            sc = v > 1e-300 ? 1.0 / sqrt(v) : 0.0;
            if (blockIdx.x == 0) *yy = v;
        }
    } else if (threadIdx.x < 64 && blockIdx.x == 0 && rsums) {
        const double v = sum_blocks(rsums, nrb);
        if (threadIdx.x == 32) *rr = v;
    }
    __syncthreads();
    const double s = sc;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        y[i] *= s;
}

// out = v / (diag H - theta diag N), the denominator clamped as in k_ritz_vectors
__global__ void __launch_bounds__(256) k_precond_apply(const double* __restrict__ v, const double* __restrict__ dh,
                                                       const double* __restrict__ dn,
                                                       const double* __restrict__ scal, double clamp, int64_t n,
                                                       double* __restrict__ out) {
    const double theta = scal[0];
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        double den = dh[i] - theta * dn[i];
        if (fabs(den) < clamp) den = den < 0.0 ? -clamp : clamp;
        out[i] = v[i] / den;
    }
}

__global__ void __launch_bounds__(256) k_axpy_ratio(double* __restrict__ x, const double* __restrict__ y, int64_t n,
                                                    const double* __restrict__ num, const double* __restrict__ den,
                                                    double sign) {
    const double d = *den;
    const double a = d != 0.0 ? sign * (*num) / d : 0.0;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        x[i] = fma(a, y[i], x[i]);
}

__global__ void __launch_bounds__(256) k_xpby_ratio(double* __restrict__ p, const double* __restrict__ r, int64_t n,
                                                    const double* __restrict__ num, const double* __restrict__ den) {
    const double d = *den;
    const double b = d != 0.0 ? (*num) / d : 0.0;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        p[i] = fma(b, p[i], r[i]);
}

constexpr int kRitzMax = 32;

// ---- incremental Ritz step --------------------------------------------------------------------
// Keeps, across the iterations of one Davidson solve, an n-orthonormal coefficient basis X
// (Y = V X has Y^T N Y = I), the projected matrix hp = X^T h X and the eigenvectors C of hp.
// Adding basis vector v_m: classical Gram-Schmidt of e_m against X in the n inner product,
// twice; the direction is kept when its n-norm^2 exceeds eps * max(diag n) (numerically null
// directions of the metric are dropped, as in canonical orthogonalisation).  hp grows by one row
// and column; its eigenbasis is re-solved by FP32 Jacobi started from the previous eigenvectors (so only
// the new coupling has to be rotated away), and the lowest pair is refined in FP64 against hp (below).
//
// One CTA of 16 warps, bound by latency: every FP64 instruction of a warp holds its sub-partition's FP64
// pipe for 64 clocks.  The FP64 products of vectors of 32 run on four warps, one per sub-partition, each
// taking a quarter of the sum; every thread of the CTA owns two elements of the FP32 matrices, so a Jacobi
// round (the two rotations of an element's row and column, recomputed by each thread) is one barrier.
// Measured (GB300, ncu, L = 16, D = 64 step, subspaces up to 20): 46 us (49 us with IEEE division and root in the
// Jacobi rotations); one warp took 93 us.
__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

constexpr double kMetricFloor = 1e-14;
constexpr int kRitzThreads = 512;
constexpr int kRitzLd = RitzState::kR + 1;

// sum_l M[lane, l] v_l for l < n (v_l held by lane l; M[lane, l] = mat[lane * rs + l * cs]) on the four warps
// of threads 0 .. 127, whose `slot` of shared memory (128 doubles) no warp may still be reading.
__device__ __forceinline__ double matvec4(const double* mat, int rs, int cs, double v, int n, double* slot) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    double acc = 0.0;
    for (int l = w; l < n; l += 4) acc = fma(mat[lane * rs + l * cs], __shfl_sync(0xffffffffu, v, l), acc);
    slot[w * 32 + lane] = acc;
    asm volatile("bar.sync 1, 128;" ::: "memory");
    return (slot[lane] + slot[32 + lane]) + (slot[64 + lane] + slot[96 + lane]);
}

// Cyclic Jacobi (round-robin pairs) on the n x n symmetric matrix in a (row stride kRitzLd), the rotations
// accumulated in v (the identity at first); a2, v2: second buffers.  Returns with the results in a and v.
__device__ void jacobi_cta_f32(float*& a, float*& v, float*& a2, float*& v2, int n, float* red) {
    const int tid = threadIdx.x, np = (n + 1) & ~1;
    if (n <= 1) return;
    // the two elements of this thread and the round-robin positions of their row and column
    int ei[2], ej[2], ki[2], kj[2];
    bool own[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int e = tid + q * kRitzThreads;
        own[q] = e < n * n;
        ei[q] = own[q] ? e / n : 0;
        ej[q] = own[q] ? e - ei[q] * n : 0;
    }
    float off_prev = INFINITY;
    for (int sweep = 0; sweep < 30; ++sweep) {
        float off = 0.0f, tot = 0.0f;
#pragma unroll
        for (int q = 0; q < 2; ++q)
            if (own[q]) {
                const float x = a[ei[q] * kRitzLd + ej[q]];
                tot = fmaf(x, x, tot);
                if (ei[q] != ej[q]) off = fmaf(x, x, off);
            }
        for (int o = 16; o > 0; o >>= 1) {
            off += __shfl_xor_sync(0xffffffffu, off, o);
            tot += __shfl_xor_sync(0xffffffffu, tot, o);
        }
        if ((tid & 31) == 0) {
            red[tid >> 5] = off;
            red[16 + (tid >> 5)] = tot;
        }
        __syncthreads();
        off = tot = 0.0f;
#pragma unroll
        for (int w = 0; w < kRitzThreads / 32; ++w) {
            off += red[w];
            tot += red[16 + w];
        }
        // off-diagonal below 3e-5 of the matrix (the FP64 refinement of the lowest pair reduces
        // its error by about that factor per correction), or no longer decreasing
        if (off <= 1e-9f * tot || off == 0.0f || (off <= 1e-6f * tot && off > 0.25f * off_prev)) break;
        off_prev = off;
        const float tiny = 1e-10f * sqrtf(tot);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            ki[q] = ei[q];
            kj[q] = ej[q];
        }
        for (int round = 0; round < np - 1; ++round) {
            // the player at position k plays the one at np - 1 - k; position 0 is player 0, positions
            // 1 .. np - 1 move on by one player per round
            auto opponent = [&](int k) {
                const int o = np - 1 - k;
                if (o == 0) return 0;
                const int x = o - 1 + round;
                return 1 + (x >= np - 1 ? x - (np - 1) : x);
            };
            // rotation of index i with p: its own factor, and the one of its opponent's entry
            auto rotation = [&](int i, int p, float& c, float& s) {
                c = 1.0f;
                s = 0.0f;
                if (p >= n || p == i) return;
                const int lo = min(i, p), hi = max(i, p);
                const float apq = a[lo * kRitzLd + hi];
                if (!(fabsf(apq) > tiny)) return;
                const float z = __fdividef(a[hi * kRitzLd + hi] - a[lo * kRitzLd + lo], 2.0f * apq);
                const float w = fminf(fabsf(z), 1e18f), q2 = fmaf(w, w, 1.0f);
                const float t = copysignf(__fdividef(1.0f, fmaf(q2, rsqrtf(q2), w)), z);
                c = rsqrtf(fmaf(t, t, 1.0f));
                s = i == lo ? -t * c : t * c;
            };
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                if (own[q]) {
                    const int i = ei[q], j = ej[q];
                    const int pi = opponent(ki[q]), pj = opponent(kj[q]);
                    float ci, si, cj, sj;
                    rotation(i, pi, ci, si);
                    rotation(j, pj, cj, sj);
                    const int ii = i * kRitzLd, pp = (pi < n ? pi : i) * kRitzLd, jj = pj < n ? pj : j;
                    const float x = fmaf(sj, a[ii + jj], cj * a[ii + j]), y = fmaf(sj, a[pp + jj], cj * a[pp + j]);
                    a2[ii + j] = fmaf(si, y, ci * x);
                    v2[ii + j] = fmaf(sj, v[ii + jj], cj * v[ii + j]);
                    ki[q] = ki[q] == 0 ? 0 : (ki[q] == 1 ? np - 1 : ki[q] - 1);
                    kj[q] = kj[q] == 0 ? 0 : (kj[q] == 1 ? np - 1 : kj[q] - 1);
                }
            }
            __syncthreads();
            float* t = a;
            a = a2;
            a2 = t;
            t = v;
            v = v2;
            v2 = t;
        }
    }
}

__global__ void __launch_bounds__(kRitzThreads) k_ritz_inc(const double* __restrict__ h, const double* __restrict__ nm,
                                                           int ldm, int m, int reset, double eps,
                                                           RitzState* __restrict__ st, double* __restrict__ coef,
                                                           double* __restrict__ coef_prev, double* __restrict__ scal) {
    constexpr int R = RitzState::kR, L = kRitzLd, MM = R * L;
    extern __shared__ double rs_smem[];
    double* X = rs_smem;      // n-orthonormal coefficient basis, X[i * L + j]
    double* HP = X + MM;      // X^T h X
    double* NS = HP + MM;     // n, full symmetric; later the eigenbasis in FP64
    double* HS = NS + MM;     // h, full symmetric
    float* Af = reinterpret_cast<float*>(HS + MM);
    float* A2 = Af + MM;
    float* Vf = A2 + MM;
    float* V2 = Vf + MM;
    float* W0 = V2 + MM;      // start basis
    float* Hf = W0 + MM;      // X^T h X in FP32
    __shared__ double slots[2][128];
    __shared__ float red[32];
    __shared__ int k_sh;
    const int tid = threadIdx.x, lane = tid & 31;
    int k = 0, m0 = 0, kc = 0;
    if (!reset) {
        k = st->k;
        m0 = st->m;
        kc = st->kc;
    }
    for (int e = tid; e < R * R; e += kRitzThreads) {
        const int i = e / R, j = e % R;
        X[i * L + j] = reset ? 0.0 : st->X[i + j * R];
        HP[i * L + j] = reset ? 0.0 : st->hp[e];
        W0[i * L + j] = i < kc && j < kc ? st->C[e] : (i == j ? 1.0f : 0.0f);
        const bool in = i < m && j < m;
        const int hi = i > j ? i : j, lo = i > j ? j : i;
        NS[i * L + j] = in ? nm[hi * ldm + lo] : 0.0;
        HS[i * L + j] = in ? h[hi * ldm + lo] : 0.0;
    }
    // the coefficients of the previous Ritz vector, kept for the restart
    if (tid < R) coef_prev[tid] = coef[tid];
    __syncthreads();
    int turn = 0;
    if (tid < 128) {  // four warps with the same values
        auto mv = [&](const double* mat, int rs, int cs, double v, int n) {
            turn ^= 1;
            return matvec4(mat, rs, cs, v, n, slots[turn]);
        };
        double dmax = lane < m ? NS[lane * L + lane] : 0.0;
        for (int o = 16; o > 0; o >>= 1) dmax = fmax(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
        for (int col = m0; col < m; ++col) {
            // y = e_col - X (X^T n y), twice, in the n inner product (lane i holds y_i, i <= col)
            double y = lane == col ? 1.0 : 0.0, ny;
            for (int pass = 0; pass < 2; ++pass) {
                ny = mv(NS, L, 1, y, col + 1);
                if (lane > col) ny = 0.0;
                const double c = mv(X, 1, L, ny, col + 1);  // lane j: X_j . n y
                const double corr = mv(X, L, 1, c, k);
                if (lane <= col) y -= corr;
            }
            ny = mv(NS, L, 1, y, col + 1);
            const double nu2 = warp_sum(lane <= col ? y * ny : 0.0);
            // the basis vectors have unit norm and |N_eff| <= 1: below kMetricFloor the metric is
            // numerically zero (no state of the target spin is reachable), whatever eps says
            if (nu2 > eps * dmax && nu2 > kMetricFloor) {
                const double xk = lane <= col ? y * (1.0 / sqrt(nu2)) : 0.0;
                double hx = mv(HS, L, 1, xk, col + 1);
                if (lane > col) hx = 0.0;
                if (tid < 32) X[lane * L + k] = xk;
                asm volatile("bar.sync 1, 128;" ::: "memory");
                const double hk = mv(X, 1, L, hx, col + 1);  // lane j: X_j . h x_k
                if (tid < 32 && lane <= k) {
                    HP[lane * L + k] = hk;
                    HP[k * L + lane] = hk;
                }
                ++k;
                asm volatile("bar.sync 1, 128;" ::: "memory");
            }
        }
        if (tid == 0) k_sh = k;
    }
    __syncthreads();
    k = k_sh;
    // The Ritz pair.  FP32 Jacobi on W0^T HP W0, W0 = previous eigenvectors padded with the
    // identity (so only the new row and column have to be rotated away), gives the eigenbasis W of
    // HP to FP32 accuracy; the lowest pair is then refined in FP64 against HP itself: Rayleigh
    // quotient y^T HP y / y^T y, residual r = HP y - theta y, and the correction
    // sum_{j != min} w_j (w_j^T r) / (theta - lambda_j) through W's spectrum, up to three times, so theta
    // and the coefficients are FP64-accurate while the O(k^3) work runs in FP32.
    for (int e = tid; e < k * k; e += kRitzThreads) {
        const int i = e / k, j = e - i * k;
        Hf[i * L + j] = static_cast<float>(HP[i * L + j]);
    }
    __syncthreads();
    for (int e = tid; e < k * k; e += kRitzThreads) {  // HP W0
        const int i = e / k, j = e - i * k;
        float acc = 0.0f;
        for (int l = 0; l < k; ++l) acc = fmaf(Hf[i * L + l], W0[l * L + j], acc);
        A2[i * L + j] = acc;
    }
    __syncthreads();
    for (int e = tid; e < k * k; e += kRitzThreads) {  // W0^T (HP W0), one triangle
        const int i = e / k, j = e - i * k;
        if (i <= j) {
            float acc = 0.0f;
            for (int l = 0; l < k; ++l) acc = fmaf(W0[l * L + i], A2[l * L + j], acc);
            Af[i * L + j] = acc;
            Af[j * L + i] = acc;
        }
        Vf[i * L + j] = i == j ? 1.0f : 0.0f;
    }
    __syncthreads();
    jacobi_cta_f32(Af, Vf, A2, V2, k, red);
    __syncthreads();
    for (int e = tid; e < k * k; e += kRitzThreads) {  // W = W0 V
        const int i = e / k, j = e - i * k;
        float acc = 0.0f;
        for (int l = 0; l < k; ++l) acc = fmaf(W0[i * L + l], Vf[l * L + j], acc);
        Hf[i * L + j] = acc;
        NS[i * L + j] = static_cast<double>(acc);
    }
    __syncthreads();
    if (tid < 128) {
        auto mv = [&](const double* mat, int rs, int cs, double v, int n) {
            turn ^= 1;
            return matvec4(mat, rs, cs, v, n, slots[turn]);
        };
        // lowest diagonal entry of the rotated matrix
        const float lam = lane < k ? Af[lane * L + lane] : INFINITY;
        float best = lam;
        int jmin = lane < k ? lane : R;
        for (int o = 16; o > 0; o >>= 1) {
            const float ob = __shfl_xor_sync(0xffffffffu, best, o);
            const int oj = __shfl_xor_sync(0xffffffffu, jmin, o);
            if (ob < best || (ob == best && oj < jmin)) {
                best = ob;
                jmin = oj;
            }
        }
        double y = (lane < k && jmin < R) ? NS[lane * L + jmin] : 0.0;
        double theta = 0.0;
        bool last = false;
        for (int it = 0;; ++it) {
            double hy = mv(HP, L, 1, y, k);
            if (lane >= k) hy = 0.0;
            double yy = y * y, yhy = y * hy;
            for (int o = 16; o > 0; o >>= 1) {
                yy += __shfl_xor_sync(0xffffffffu, yy, o);
                yhy += __shfl_xor_sync(0xffffffffu, yhy, o);
            }
            theta = yy > 0.0 ? yhy / yy : 0.0;
            if (last) {
                y = yy > 0.0 ? y / sqrt(yy) : 0.0;
                break;
            }
            const double r = lane < k ? hy - theta * y : 0.0;
            double c = mv(NS, 1, L, r, k);  // lane j: w_j^T r
            const double den = theta - static_cast<double>(lam);
            // components (nearly) degenerate with the lowest one are left as they are
            const bool use = lane < k && lane != jmin && fabs(den) > 1e-7 * (fabs(theta) + fabs(static_cast<double>(lam)) + 1e-300);
            c = use ? c / den : 0.0;
            const double d = mv(NS, L, 1, c, k);
            if (lane < k) y += d;
            // a correction leaves 3e-5 of itself: below 1e-11 the next one is rounding
            last = it == 2 || !__any_sync(0xffffffffu, fabsf(static_cast<float>(c)) > 1e-11f);
        }
        if (tid == 0) {
            scal[0] = k > 0 ? theta : 0.0;
            scal[1] = static_cast<double>(k);
        }
        // coefficients of the Ritz vector in the basis V: X y
        const double acc = mv(X, L, 1, y, k);
        if (tid < R) coef[tid] = tid < m && k > 0 ? acc : 0.0;
    }
    for (int e = tid; e < R * R; e += kRitzThreads) {
        const int i = e / R, j = e % R;
        st->C[e] = (i < k && j < k) ? Hf[i * L + j] : 0.0f;
        st->X[i + j * R] = X[i * L + j];
        st->hp[e] = HP[i * L + j];
    }
    if (tid == 0) {
        st->k = k;
        st->m = m;
        st->kc = k;
    }
}

// Orthonormal restart coefficients from [c_new, c_old] (Gram-Schmidt, twice); c_new is replaced by the
// coefficients of the same vector in the restarted basis.
__global__ void k_restart_coef(double* __restrict__ cn, const double* __restrict__ co, int m,
                               double* __restrict__ Q, double* __restrict__ out) {
    if (threadIdx.x != 0) return;
    double a[kRitzMax], b[kRitzMax];
    double na = 0.0;
    for (int i = 0; i < m; ++i) { a[i] = cn[i]; na += a[i] * a[i]; }
    na = sqrt(na);
    for (int i = 0; i < m; ++i) a[i] /= na;
    for (int i = 0; i < m; ++i) b[i] = co[i];
    for (int pass = 0; pass < 2; ++pass) {
        double d = 0.0;
        for (int i = 0; i < m; ++i) d += a[i] * b[i];
        for (int i = 0; i < m; ++i) b[i] -= d * a[i];
    }
    double nb = 0.0;
    for (int i = 0; i < m; ++i) nb += b[i] * b[i];
    nb = sqrt(nb);
    int k = 1;
    for (int i = 0; i < m; ++i) Q[i] = a[i];
    if (nb > 1e-10) {
        k = 2;
        for (int i = 0; i < m; ++i) Q[m + i] = b[i] / nb;
    } else {
        for (int i = 0; i < m; ++i) Q[m + i] = 0.0;  // a zero second column (dropped downstream)
    }
    out[0] = k;
    // coefficients of the current Ritz vector in the rotated basis: Q^T c_new
    double d0 = 0.0, d1 = 0.0;
    for (int i = 0; i < m; ++i) { d0 += Q[i] * cn[i]; if (k == 2) d1 += Q[m + i] * cn[i]; }
    for (int i = 0; i < kRitzMax; ++i) cn[i] = i == 0 ? d0 : (i == 1 ? d1 : 0.0);
}

// ---- ordered truncation ---------------------------------------------------------------------------
// Rank sort of the singular values sqrt(max(evals, 0)), descending, ties by flat index: one warp per
// value (non-negative doubles compare as integers, which spares the FP64 pipe).
__global__ void __launch_bounds__(256) k_trunc_rank(const double* __restrict__ evals, int total,
                                                    int* __restrict__ order, double* __restrict__ sorted) {
    const int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (i >= total) return;
    auto key = [&](int j) -> long long {
        const double v = evals[j];
        return __double_as_longlong(v > 0.0 ? v : 0.0);
    };
    const long long ki = key(i);
    int rank = 0;
    for (int j = lane; j < total; j += 32) {
        const long long kj = key(j);
        rank += (kj > ki || (kj == ki && j < i)) ? 1 : 0;
    }
    rank = __reduce_add_sync(0xffffffffu, rank);
    if (lane == 0) {
        order[rank] = i;
        sorted[rank] = sqrt(__longlong_as_double(ki));
    }
}

// Inclusive block scan of one int per thread (sum, or maximum); *total receives the last value.
template <bool MAX>
__device__ int block_scan(int v, int* sh, int* total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v = MAX ? max(v, u) : v + u;
    }
    if (lane == 31) sh[w] = v;
    __syncthreads();
    if (w == 0) {
        int t = lane < static_cast<int>(blockDim.x >> 5) ? sh[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t = MAX ? max(t, u) : t + u;
        }
        sh[lane] = t;
    }
    __syncthreads();
    if (w > 0) v = MAX ? max(v, sh[w - 1]) : v + sh[w - 1];
    *total = sh[(blockDim.x >> 5) - 1];
    __syncthreads();
    return v;
}

// Tie clusters, the cut at D and the counts per label, every step parallel over the values.  The flat
// indices ascend in (n, 2m, index), so the order inside a cluster is the order of the indices.  Measured
// on the canonicalisation of the random L = 24, D = 256 state (about 1000 values, half of them the tied
// zeros of a full-rank cut): 5.5 ms for the form it replaces, which walked the values and sorted
// the clusters by insertion on one thread.
__global__ void __launch_bounds__(1024) k_trunc_select(const int64_t* __restrict__ val_off, int n_labels, int total, int D,
                                                       double tie_rtol, double drop_abs, int* __restrict__ keep_count,
                                                       int* __restrict__ keep_total, double* __restrict__ discarded,
                                                       const int* __restrict__ order, int* __restrict__ start,
                                                       int* __restrict__ order2, double* __restrict__ sorted,
                                                       double* __restrict__ sig2) {
    __shared__ int sh[32];
    __shared__ double shd[32];
    const int tid = threadIdx.x, nt = blockDim.x;
    for (int l = tid; l < n_labels; l += nt) keep_count[l] = 0;
    const double gap = total > 0 ? tie_rtol * sorted[0] : 0.0;
    int carry = 0, last = 0;
    for (int base = 0; base < total; base += nt) {  // first position of every value's cluster
        const int r = base + tid;
        int s = 0;
        if (r < total && r > 0 && sorted[r - 1] - sorted[r] > gap) s = r;
        s = max(block_scan<true>(s, sh, &last), carry);
        carry = max(carry, last);
        if (r < total) start[r] = s;
    }
    __syncthreads();
    for (int r = tid; r < total; r += nt) {
        const int cs = start[r], i = order[r];
        int before = 0;
        // a cluster of dropped values needs no order (the null directions of all labels are one: hundreds of
        // dependent loads a thread, 49 us a launch of the L = 24, D = 256 canonicalisation, 8 us without)
        if (sorted[cs] < drop_abs)
            before = r - cs;
        else
            for (int j = cs; j < total && start[j] == cs; ++j) before += order[j] < i ? 1 : 0;
        order2[cs + before] = i;
        sig2[cs + before] = sorted[r];
    }
    __syncthreads();
    double disc = 0.0;
    carry = 0;
    for (int base = 0; base < total; base += nt) {
        const int r = base + tid;
        const double s = r < total ? sig2[r] : 0.0;
        const int ok = r < total && s >= drop_abs ? 1 : 0;
        const int upto = carry + block_scan<false>(ok, sh, &last);
        carry += last;
        if (ok && upto <= D) {
            const int i = order2[r];
            int lo = 0, hi = n_labels - 1;  // last label whose values start at or before i
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (val_off[mid] <= i) lo = mid; else hi = mid - 1;
            }
            atomicAdd(keep_count + lo, 1);
        } else {
            disc = fma(s, s, disc);
        }
    }
    disc = block_sum(disc, shd);
    if (tid == 0) {
        keep_total[0] = min(carry, D);
        discarded[0] = disc;
    }
}

// ---- block copies ------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_copy_blocks(const __grid_constant__ Slots S, const CopyBlock* __restrict__ blocks, int n) {
    const int bi = blockIdx.x;
    if (bi >= n) return;
    const CopyBlock b = blocks[bi];
    const double* src = resolve(S, b.src);
    double* dst = resolve(S, b.dst);
    const int tot = b.rows * b.cols;
    for (int e = threadIdx.x; e < tot; e += blockDim.x) {
        const int r = e / b.cols, c = e - r * b.cols;
        const double v = b.transpose ? src[static_cast<int64_t>(c) * b.ld_src + r] : src[static_cast<int64_t>(r) * b.ld_src + c];
        dst[static_cast<int64_t>(r) * b.ld_dst + c] = v;
    }
}

// FP64 throughput probe: 8 independent FMA chains per thread.
__global__ void __launch_bounds__(256) k_fp64_peak(double* out, int iters, double a, double b) {
    double x0 = threadIdx.x * 1e-7, x1 = x0 + 1e-8, x2 = x0 + 2e-8, x3 = x0 + 3e-8;
    double x4 = x0 + 4e-8, x5 = x0 + 5e-8, x6 = x0 + 6e-8, x7 = x0 + 7e-8;
    for (int i = 0; i < iters; ++i) {
        x0 = fma(x0, a, b); x1 = fma(x1, a, b); x2 = fma(x2, a, b); x3 = fma(x3, a, b);
        x4 = fma(x4, a, b); x5 = fma(x5, a, b); x6 = fma(x6, a, b); x7 = fma(x7, a, b);
    }
    const double r = x0 + x1 + x2 + x3 + x4 + x5 + x6 + x7;
    if (r == 12345.678) out[0] = r;  // keeps the chains live
}

int grid_for(int64_t n, int threads, int cap) {
    int64_t g = (n + threads - 1) / threads;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return static_cast<int>(g);
}

// Blocks of the elementwise kernels that also sum (one partial sum each): up to kNormBlocks.
int norm_blocks(int64_t n) { return grid_for(n, 256, kNormBlocks); }

}  // namespace

// ---- launch wrappers ----------------------------------------------------------------------------

cudaError_t launch_gemm_f64(const Slots& slots, const GemmTask* tasks, const GemmSeg* segs, const GemmTile* tiles,
                            const int* cmaps, int n_tiles, cudaStream_t st, const BetaRun& beta) {
    if (n_tiles <= 0) return cudaSuccess;
    const int warps_per_cta = 4;
    const int grid = (n_tiles * beta.ng + warps_per_cta - 1) / warps_per_cta;
    k_gemm_f64<<<grid, 32 * warps_per_cta, 0, st>>>(slots, beta.stride, op0_entries(beta, 0, n_tiles), beta.g0, beta.ng, tasks,
                                                    segs, tiles, cmaps, n_tiles);
    return cudaGetLastError();
}

cudaError_t launch_gemm_f64_stack(const Slots& slots, const TcStack* stacks, const TcRow* rows, const TcSeg* segs,
                                  const uint64_t* atab, const int* cmaps, const int4* units, int u0, int u1, cudaStream_t st,
                                  const BetaRun& beta) {
    if (u1 <= u0) return cudaSuccess;
    k_gemm_f64_stack<<<((u1 - u0) * beta.ng + 3) / 4, 128, 0, st>>>(slots, beta.stride, op0_entries(beta, u0, u1 - u0), beta.g0,
                                                                    beta.ng, stacks, rows, segs, atab, cmaps, units, u0, u1);
    return cudaGetLastError();
}

cudaError_t launch_sum_partials(const double* partial0, const double* partial1, const double* w, int G, int ks0, int ks1,
                                int64_t n, double* out0, double* out1, cudaStream_t st) {
    if (n <= 0 || (!out0 && !out1)) return cudaSuccess;
    const bool both = out0 && out1;
    const dim3 grid(grid_for(n, 256, 4096), both ? 2 : 1);
    if (out0)
        k_sum_partials<<<grid, 256, 0, st>>>(partial0, partial1, w, G, ks0, ks1, n, out0, out1);
    else
        k_sum_partials<<<grid, 256, 0, st>>>(partial1, partial1, w, G, ks1, ks1, n, out1, out1);
    return cudaGetLastError();
}

cudaError_t launch_comb_f64(const Slots& slots, const CombOut* outs, const CombTerm* terms, int n_outs,
                            cudaStream_t st) {
    if (n_outs <= 0) return cudaSuccess;
    k_comb_f64<<<n_outs, 256, 0, st>>>(slots, outs, terms, n_outs);
    return cudaGetLastError();
}

cudaError_t launch_diag_f64(const Slots& slots, const DiagBlock* blocks, const DiagTerm* terms, int n_blocks,
                            double* dh, double* dn, cudaStream_t st) {
    if (n_blocks <= 0) return cudaSuccess;
    k_diag_f64<<<n_blocks, 256, 0, st>>>(slots, blocks, terms, n_blocks, dh, dn);
    return cudaGetLastError();
}

cudaError_t launch_multidot(const double* V, int64_t ldv, int m, const double* x, int64_t n, double* out,
                            double* partial, cudaStream_t st) {
    if (m <= 0) return cudaSuccess;
    if (m > kRitzMax) return cudaErrorInvalidValue;
    const int nb = grid_for(n, 256, kRedBlocks);
    k_multidot_partial<<<dim3(nb, m), 256, 0, st>>>(V, ldv, x, n, partial);
    k_multidot_final<<<m, 32, 0, st>>>(partial, nb, out);
    return cudaGetLastError();
}

cudaError_t launch_gemv(const double* V, int64_t ldv, int m, const double* c, int64_t n, double* y, int sub,
                        cudaStream_t st) {
    if (m > 64) return cudaErrorInvalidValue;
    k_gemv<<<grid_for(n, 256, 2048), 256, 0, st>>>(V, ldv, m, c, n, y, sub);
    return cudaGetLastError();
}

cudaError_t launch_basis_rotate(const double* src, int64_t ld, int m, const double* Q, int ldq, int k, int64_t n,
                                double* dst, cudaStream_t st) {
    if (m > 64 || k > 4) return cudaErrorInvalidValue;
    k_basis_rotate<<<grid_for(n, 256, 2048), 256, 0, st>>>(src, ld, m, Q, ldq, k, n, dst);
    return cudaGetLastError();
}


cudaError_t launch_ritz_inc(const double* h, const double* nmat, int ldm, int m, int reset, double eps_metric,
                            RitzState* state, double* coef, double* coef_prev, double* scal, cudaStream_t st) {
    if (m > RitzState::kR) return cudaErrorInvalidValue;
    constexpr int smem = RitzState::kR * kRitzLd * (4 * static_cast<int>(sizeof(double)) + 6 * static_cast<int>(sizeof(float)));
    static int attr_device = -1;  // the attribute is per device; set it once per device in use
    int dev = 0;
    cudaGetDevice(&dev);
    if (attr_device != dev) {
        cudaError_t e = cudaFuncSetAttribute(k_ritz_inc, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        attr_device = dev;
    }
    k_ritz_inc<<<1, kRitzThreads, smem, st>>>(h, nmat, ldm, m, reset, eps_metric, state, coef, coef_prev, scal);
    return cudaGetLastError();
}

cudaError_t launch_ritz_vectors(const double* V, const double* HV, const double* NV, int64_t n, int m, const double* coef,
                                const double* dh, const double* dn, const double* scal, double clamp, double* x,
                                double* hx, double* nx, double* r, double* t, double* t2, double* sums, cudaStream_t st) {
    if (m > kRitzMax) return cudaErrorInvalidValue;
    k_ritz_vectors<<<norm_blocks(n), 256, 0, st>>>(V, HV, NV, n, m, coef, dh, dn, scal, clamp, x, hx, nx, r, t, t2, sums);
    return cudaGetLastError();
}

cudaError_t launch_project(const double* V, int64_t n, int m, double* y, double* partial, double* sums, cudaStream_t st) {
    if (m > kRitzMax) return cudaErrorInvalidValue;
    const int nb = grid_for(n, 256, kRedBlocks);
    if (m > 0) k_multidot_partial<<<dim3(nb, m), 256, 0, st>>>(V, n, y, n, partial);
    k_project<<<norm_blocks(n), 256, 0, st>>>(V, n, m, partial, nb, y, sums);
    return cudaGetLastError();
}

cudaError_t launch_sum_blocks(const double* sums, int64_t n, double* out, cudaStream_t st) {
    k_sum_blocks<<<1, 32, 0, st>>>(sums, norm_blocks(n), out);
    return cudaGetLastError();
}

cudaError_t launch_normalise(double* y, int64_t n, const double* ysums, const double* rsums, double* yy, double* rr,
                             cudaStream_t st) {
    k_normalise<<<norm_blocks(n), 256, 0, st>>>(y, n, ysums, norm_blocks(n), rsums, norm_blocks(n), yy, rr);
    return cudaGetLastError();
}

cudaError_t launch_multidot2(const double* V, int64_t ldv, int m, const double* x0, const double* x1, int64_t n,
                             double* out0, double* out1, double* partial, cudaStream_t st) {
    if (m <= 0) return cudaSuccess;
    if (m > kRitzMax) return cudaErrorInvalidValue;
    const int nb = grid_for(n, 256, kRedBlocks);
    k_multidot2_partial<<<dim3(nb, m, 2), 256, 0, st>>>(V, ldv, x0, x1, n, partial);
    k_multidot2_final<<<dim3(m, 2), 32, 0, st>>>(partial, nb, out0, out1);
    return cudaGetLastError();
}

cudaError_t launch_precond_apply(const double* v, const double* dh, const double* dn, const double* scal,
                                 double clamp, int64_t n, double* out, cudaStream_t st) {
    k_precond_apply<<<grid_for(n, 256, 2048), 256, 0, st>>>(v, dh, dn, scal, clamp, n, out);
    return cudaGetLastError();
}

cudaError_t launch_norm2(const double* x, int64_t n, double* out, double* partial, cudaStream_t st) {
    const int nb = grid_for(n, 256, kRedBlocks);
    k_norm2_partial<<<nb, 256, 0, st>>>(x, n, partial);
    k_multidot_final<<<1, 32, 0, st>>>(partial, nb, out);
    return cudaGetLastError();
}

cudaError_t launch_scale_inv_sqrt(double* x, int64_t n, const double* nrm2, cudaStream_t st) {
    k_scale_inv_sqrt<<<grid_for(n, 256, 2048), 256, 0, st>>>(x, n, nrm2);
    return cudaGetLastError();
}

cudaError_t launch_axpy_ratio(double* x, const double* y, int64_t n, const double* num, const double* den,
                              double sign, cudaStream_t st) {
    k_axpy_ratio<<<grid_for(n, 256, 2048), 256, 0, st>>>(x, y, n, num, den, sign);
    return cudaGetLastError();
}

cudaError_t launch_xpby_ratio(double* p, const double* r, int64_t n, const double* num, const double* den,
                              cudaStream_t st) {
    k_xpby_ratio<<<grid_for(n, 256, 2048), 256, 0, st>>>(p, r, n, num, den);
    return cudaGetLastError();
}

cudaError_t launch_restart_coef(double* c_new, const double* c_old, int m, double* Qout, double* scal_out,
                                cudaStream_t st) {
    if (m > kRitzMax) return cudaErrorInvalidValue;
    k_restart_coef<<<1, 32, 0, st>>>(c_new, c_old, m, Qout, scal_out);
    return cudaGetLastError();
}

cudaError_t launch_truncate(const double* evals, const int64_t* val_off, int n_labels, int total, int D, double tie_rtol,
                            double drop_abs, int* keep_count, int* keep_total, double* discarded, int* scratch_idx,
                            double* scratch_val, cudaStream_t st) {
    if (total > 0) k_trunc_rank<<<(total + 7) / 8, 256, 0, st>>>(evals, total, scratch_idx, scratch_val);
    k_trunc_select<<<1, 1024, 0, st>>>(val_off, n_labels, total, D, tie_rtol, drop_abs, keep_count, keep_total, discarded,
                                       scratch_idx, scratch_idx + total, scratch_idx + 2 * total, scratch_val,
                                       scratch_val + total);
    return cudaGetLastError();
}

cudaError_t measure_fp64_peak(double* tflops) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    double* out = nullptr;
    cudaError_t e = cudaMalloc(&out, sizeof(double));
    if (e != cudaSuccess) return e;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    const int blocks = sms * 8, threads = 256, iters = 1 << 14;
    k_fp64_peak<<<blocks, threads>>>(out, 256, 0.999999, 1e-9);  // warm-up
    cudaEventRecord(e0);
    k_fp64_peak<<<blocks, threads>>>(out, iters, 0.999999, 1e-9);
    cudaEventRecord(e1);
    e = cudaEventSynchronize(e1);
    float ms = 0.0f;
    cudaEventElapsedTime(&ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(out);
    if (e != cudaSuccess) return e;
    const double flops = 2.0 * 8.0 * iters * static_cast<double>(blocks) * threads;
    *tflops = flops / (ms * 1e-3) / 1e12;
    return cudaGetLastError();
}

cudaError_t launch_copy_blocks(const Slots& slots, const CopyBlock* blocks, int n, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_copy_blocks<<<n, 256, 0, st>>>(slots, blocks, n);
    return cudaGetLastError();
}

}  // namespace spmps
