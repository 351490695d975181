// Singular vectors of the decimation blocks: one-sided Jacobi, started in FP32 and finished in FP64.
//
// The FP64 pipe of this part executes 2 FMA per clock and SM (FP32: 128), so an FP64 Jacobi is bound
// by that pipe of the few SMs a block occupies.  The bulk of the rotations therefore runs in FP32: for
// the rows of Z (the block, or its transpose),
//   1. k_osj<float>: one-sided Jacobi on an FP32 copy [Z | I] finds J with nearly orthogonal rows of J Z;
//   2. two Newton-Schulz steps J <- (3/2 - 1/2 J J^T) J in FP64 (k_block_gemm, all SMs) make J orthonormal
//      to FP64, and Z' = J Z is formed in FP64 from the unrounded block;
//   3. k_osj<double>: one-sided Jacobi on Z' to FP64 convergence (two or three sweeps as a rule: the FP32
//      start leaves relative couplings of 1e-6, and the convergence is quadratic).
// The singular values are the row norms of the result and come from Z itself, not from its Gram matrix,
// so small ones keep the FP64 noise floor of Z (1e-16, not 1e-8).
#include <cooperative_groups.h>

#include "svd.h"

namespace spmps {

namespace {

namespace cgx = cooperative_groups;

constexpr int kOsjC = 8;             // CTAs per block of the global-memory form
constexpr int kOsj32Threads = 640;   // shared-memory form: 80 pairs at once with up to 102 registers a thread
constexpr int kFp32Sweeps = 40;      // most sweeps of the FP32 start
constexpr double kNullRel = 1e-9;    // rows below this fraction of the block's norm are not separated further

template <class T>
__device__ __forceinline__ T ldc(const T* p) { return __ldcg(p); }

template <class T>
__device__ __forceinline__ T wsum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// The rows of [0, R) whose squared norm is above `least`, ascending, by the first warp of a CTA (R <= kSvdMaxRows).
// Rows beyond a block's rank shrink to the rounding noise of the large rows within two sweeps; without them a
// sweep has as many rounds as the block has rank.
constexpr int kFullSweeps = 2;
template <class Norm>
__device__ __forceinline__ void list_rows(unsigned short* list, int* count, int R, bool all, Norm above) {
    if (threadIdx.x >= 32) return;
    const int lane = threadIdx.x;
    int n = 0;
    for (int base = 0; base < R; base += 32) {
        const int r = base + lane;
        const bool in = r < R && (all || above(r));
        const unsigned m = __ballot_sync(0xffffffffu, in);
        if (in) list[n + __popc(m & ((1u << lane) - 1u))] = static_cast<unsigned short>(r);
        n += __popc(m);
    }
    if (lane == 0) *count = n;
}

// Place of row r among R rows by descending norm (ties by row), by a warp.
template <class Norm>
__device__ __forceinline__ int row_rank(int R, int r, Norm norm) {
    const auto v = norm(r);
    int before = 0;
    for (int j = threadIdx.x & 31; j < R; j += 32) {
        const auto o = norm(j);
        before += (o > v || (o == v && j < r)) ? 1 : 0;
    }
    return __reduce_add_sync(0xffffffffu, before);
}

// FP32 <-> FP64 by integer instructions: a conversion instruction runs on the FP64 pipe.  to_f32 truncates,
// divides by 2^shift first and clamps to [0, FLT_MAX]; to_f64 is exact (zero for subnormals).
__device__ __forceinline__ float to_f32(float v, int) { return v; }
__device__ __forceinline__ float to_f32(double v, int shift) {
    const int hi = __double2hiint(v), t = (hi & 0x7FFFFFFF) - ((896 + shift) << 20);
    const unsigned m = t < (1 << 20) ? 0u : (t >= (255 << 20) ? 0x7F7FFFFFu : __funnelshift_l(__double2loint(v), t, 3));
    return __uint_as_float(m | (static_cast<unsigned>(hi) & 0x80000000u));
}
__device__ __forceinline__ double to_f64(float v) {
    const unsigned u = __float_as_uint(v), m = u & 0x7FFFFFFFu;
    const unsigned hi = m < 0x00800000u ? 0u : (m >> 3) + (896u << 20);
    return __hiloint2double(static_cast<int>(hi | (u & 0x80000000u)), m < 0x00800000u ? 0 : static_cast<int>(m << 29));
}

// tan(theta) of the rotation that uncouples two rows: d the difference of their squared norms, g their product.
// For rows of very different norms it has to be right down to g / d, far below FP32's epsilon.
__device__ __forceinline__ float rotation_tan(float d, float g) {
    const float zeta = __fdividef(d, 2.0f * g), z = fabsf(zeta), q = fmaf(z, z, 1.0f);
    return z > 1e8f ? __fdividef(g, d) : copysignf(__fdividef(1.0f, fmaf(q, rsqrtf(q), z)), zeta);
}
__device__ __forceinline__ float half_tan(float t) {
    const float q = fmaf(t, t, 1.0f);
    return __fdividef(t, 1.0f + q * rsqrtf(q));
}

// sin(theta) for h = tan(theta / 2): 2 h / (1 + h^2) to the precision of T.  The rotation is applied as three
// shears x -= h y, y += s x, x -= h y, which is orthonormal for any h as far as s belongs to it: an error e of s
// leaves e between the two rows, so it has to be rounding of s itself; the angle may be rounded (the next sweep
// removes what it leaves).
__device__ __forceinline__ float shear_sin(float hf, float) { return __fdividef(2.0f * hf, fmaf(hf, hf, 1.0f)); }
__device__ __forceinline__ double shear_sin(float hf, double h) {
    const double h2 = to_f64(2.0f * hf);
    const float m = fabsf(hf);
    if (m < 7e-9f) return h2;                         // relative error h^2 < 5e-17
    const double q = h * h;
    if (m < 2e-3f) return fma(h2, fma(q, q, -q), h2);  // h^6 < 7e-17
    const double d = fma(h, h, 1.0);
    double y = to_f64(__fdividef(1.0f, fmaf(hf, hf, 1.0f)));
    y = fma(y, fma(-d, y, 1.0), y);
    y = fma(y, fma(-d, y, 1.0), y);
    return h2 * y;
}

// One-sided Jacobi on the rows of Z (R x W, row stride W): the first C columns are the block, the rest a
// companion that receives the same rotations.  Round-robin pairs, one warp per pair and round.
// A cluster of kOsjC CTAs with the rows in global memory (L2), a cluster barrier per round: in FP64 the
// FP64 pipes of 8 SMs share the work.  NCH > 0 keeps the two rows of a pair in registers (W <= 32 NCH)
// between the product and the update, NCH = 0 reads them twice.  The sweeps end after one that met no
// relative coupling above `done` (what it leaves is the square of that over the relative gap), or after `sweeps` of
// them with the result false.
// FP64: an instruction of a warp occupies its sub-partition's FP64 pipe for 64 cycles whether its lanes hold
// one number or 32, so a pair issues 3 per 32 elements for the shears, one for the product, 5 for its sum
// over the warp, 2 for the norms and at most 7 for the sine; comparisons, conversions and the angle are
// FP32 and integer instructions.  Measured (GB300): a launch
// of the canonicalisation below 0.38 ms on average, the middle decimation of L = 24, D = 256 2.0 ms; 0.81 and 2.7 ms
// with the comparisons, conversions and the angle's operands in FP64, 0.63 ms without the next two.  Rows beyond the
// block's rank leave the rounds after two sweeps (0.57 ms), and the FP32 start hands its rows over by descending norm.
template <class T, int NCH>
__device__ bool osj_sweeps(T* Z, T* nrm2, int R, int C, int W, T norm2_all, float done, int* conv, int rank, int ctas,
                           int sweeps) {
    const int lane = threadIdx.x & 31;
    const int warp = (threadIdx.x >> 5) * ctas + rank;  // pairs go round the CTAs: the FP64 pipes of all share them
    const int warps = (blockDim.x >> 5) * ctas;
    __shared__ unsigned short list[kSvdMaxRows];
    __shared__ int count;
    constexpr bool kF64 = sizeof(T) == 8;
    constexpr float tol = kF64 ? 1e-15f : 3e-7f;
    constexpr float floor_abs = kF64 ? 0.0f : 1e-12f;  // FP32: the noise of the block's largest rows
    constexpr float null2 = kF64 ? static_cast<float>(kNullRel * kNullRel) : 1e-13f;
    constexpr float least = kF64 ? 1e-28f : null2;
    // squared norms and products as FP32 numbers relative to the block's squared norm (to a factor of 2)
    int shift = 0;
    if constexpr (kF64) shift = norm2_all > T(0) ? ((__double2hiint(norm2_all) >> 20) & 2047) - 1023 : 0;
    auto barrier = [&]() { cgx::this_cluster().sync(); };
    auto ld = [&](const T* p) -> T { return ldc(p); };
    auto stg = [&](T* p, T v) { __stcg(p, v); };
    for (int sweep = 0; sweep < sweeps; ++sweep) {
        for (int r = warp; r < R; r += warps) {
            T s = T(0);
            for (int c = lane; c < C; c += 32) {
                const T v = ld(Z + static_cast<int64_t>(r) * W + c);
                s += v * v;
            }
            s = wsum(s);
            if (lane == 0) stg(nrm2 + r, s);
        }
        barrier();
        list_rows(list, &count, R, sweep < kFullSweeps, [&](int r) { return to_f32(ld(nrm2 + r), shift) > least; });
        barrier();  // every CTA has its list before a rotation moves a norm
        const int np = (count + 1) & ~1, half = np / 2, rows = count;
        bool rough = false;
        for (int round = 0; round < np - 1; ++round) {
            for (int i = warp; i < half; i += warps) {
                int p = i - 1 + round, q = np - 2 - i + round;  // both below 2 (np - 1)
                p = i == 0 ? 0 : 1 + (p >= np - 1 ? p - (np - 1) : p);
                q = 1 + (q >= np - 1 ? q - (np - 1) : q);
                if (p > q) {
                    const int t = p;
                    p = q;
                    q = t;
                }
                if (q >= rows) continue;
                p = list[p];
                q = list[q];
                T* zp = Z + static_cast<int64_t>(p) * W;
                T* zq = Z + static_cast<int64_t>(q) * W;
                const T a = ld(nrm2 + p), b = ld(nrm2 + q);
                const float af = to_f32(a, shift), bf = to_f32(b, shift);
                if (!(af > null2) && !(bf > null2)) continue;
                T x[NCH > 0 ? NCH : 1], y[NCH > 0 ? NCH : 1];
                T g = T(0);
                if constexpr (NCH > 0) {
#pragma unroll
                    for (int k = 0; k < NCH; ++k) {
                        const int c = lane + 32 * k;
                        x[k] = c < W ? ld(zp + c) : T(0);
                        y[k] = c < W ? ld(zq + c) : T(0);
                    }
#pragma unroll
                    for (int k = 0; k < NCH; ++k)
                        if (32 * k < C) g += lane + 32 * k < C ? x[k] * y[k] : T(0);
                } else {
                    for (int c = lane; c < C; c += 32) g += ld(zp + c) * ld(zq + c);
                }
                g = wsum(g);
                const float gf = to_f32(g, shift), gm = fabsf(gf), root = sqrtf(af) * sqrtf(bf);
                if (!(gm > tol * root) || !(gm > floor_abs)) continue;
                if (gm > done * root && af > null2 && bf > null2) rough = true;
                const float tf = rotation_tan(to_f32(b - a, shift), gf), hf = half_tan(tf);
                T hh;
                if constexpr (kF64)
                    hh = to_f64(hf);
                else
                    hh = hf;
                const T sn = shear_sin(hf, hh);
                auto turn = [&](T& u, T& v) {
                    u -= hh * v;
                    v += sn * u;
                    u -= hh * v;
                };
                if constexpr (NCH > 0) {
#pragma unroll
                    for (int k = 0; k < NCH; ++k) {
                        const int c = lane + 32 * k;
                        if (c < W) {
                            turn(x[k], y[k]);
                            stg(zp + c, x[k]);
                            stg(zq + c, y[k]);
                        }
                    }
                } else {
                    for (int c = lane; c < W; c += 32) {
                        T u = ld(zp + c), v = ld(zq + c);
                        turn(u, v);
                        stg(zp + c, u);
                        stg(zq + c, v);
                    }
                }
                // |p|^2 and |q|^2 move by tan(theta) g (summed anew at every sweep)
                T tl;
                if constexpr (kF64)
                    tl = to_f64(lane == 0 ? -tf : tf);
                else
                    tl = lane == 0 ? -tf : tf;
                const T moved = fma(tl, g, lane == 0 ? a : b);
                if (lane < 2) stg(nrm2 + (lane == 0 ? p : q), moved > T(0) ? moved : T(0));
            }
            barrier();
        }
        if (rough && lane == 0) atomicOr(conv + sweep, 1);
        __threadfence();
        barrier();
        if (!*reinterpret_cast<volatile int*>(conv + sweep)) return true;  // uniform: read after the barrier
    }
    return false;
}

// The FP32 start in one CTA's shared memory: 8 lanes per pair and four elements per access, so that a warp
// computes four angles and four sums at once.  The scheduler's issue slots bound it (a round of 26 pairs was
// 1200 of them per sub-partition with a warp per pair, half for the angle and the sum); measured (GB300): the
// middle decimation of L = 24, D = 256 3.1 ms and 0.31 ms on average in the canonicalisation below, 5.0 and 0.52 ms
// before.  The pairs of a sweep follow the order of the norms (3.4 and 0.34 ms by row).
__device__ __forceinline__ float sum8(float v) {
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ float dot4(float4 a, float4 b) { return fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, a.w * b.w))); }
__device__ __forceinline__ void turn4(float4& x, float4& y, float h, float s) {
    auto turn = [&](float& u, float& v) {
        u = fmaf(-h, v, u);
        v = fmaf(s, u, v);
        u = fmaf(-h, v, u);
    };
    turn(x.x, y.x);
    turn(x.y, y.y);
    turn(x.z, y.z);
    turn(x.w, y.w);
}

// Rows of V vectors of four, the first CV of them the block; NV > 0 keeps a pair in registers (V <= 8 NV).
template <int NV>
__device__ void osj32_sweeps(float4* Z, float* nrm2, int R, int CV, int V) {
    constexpr float tol = 3e-7f, floor_abs = 1e-12f, null2 = 1e-13f, done = 1e-3f;
    const int gl = threadIdx.x & 7, group = threadIdx.x >> 3, groups = blockDim.x >> 3;
    __shared__ unsigned short list[kSvdMaxRows];
    __shared__ int count;
    for (int sweep = 0; sweep < kFp32Sweeps; ++sweep) {
        for (int base = 0; base < R; base += groups) {
            const int r = base + group;
            float s = 0.0f;
            if (r < R)
                for (int v = gl; v < CV; v += 8) s += dot4(Z[r * V + v], Z[r * V + v]);
            s = sum8(s);
            if (r < R && gl == 0) nrm2[r] = s;
        }
        __syncthreads();
        list_rows(list, &count, R, sweep < kFullSweeps, [&](int r) { return nrm2[r] > null2; });
        __syncthreads();
        for (int r = threadIdx.x >> 5; r < R; r += blockDim.x >> 5) {
            const int to = row_rank(R, r, [&](int j) { return nrm2[j]; });
            if ((threadIdx.x & 31) == 0 && to < count) list[to] = static_cast<unsigned short>(r);
        }
        __syncthreads();
        const int np = (count + 1) & ~1, half = np / 2, rows = count;
        int rough = 0;
        for (int round = 0; round < np - 1; ++round) {
            for (int base = 0; base < half; base += groups) {
                const int i = base + group;
                int p = i - 1 + round, q = np - 2 - i + round;
                p = i == 0 ? 0 : 1 + (p >= np - 1 ? p - (np - 1) : p);
                q = 1 + (q >= np - 1 ? q - (np - 1) : q);
                if (p > q) {
                    const int t = p;
                    p = q;
                    q = t;
                }
                bool on = i < half && q < rows;
                if (on) {
                    p = list[p];
                    q = list[q];
                }
                const float a = on ? nrm2[p] : 0.0f, b = on ? nrm2[q] : 0.0f;
                on = on && (a > null2 || b > null2);
                float4* zp = Z + p * V;
                float4* zq = Z + q * V;
                const float4 zero = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                float4 x[NV > 0 ? NV : 1], y[NV > 0 ? NV : 1];
                float g = 0.0f;
                if constexpr (NV > 0) {
#pragma unroll
                    for (int k = 0; k < NV; ++k) {
                        const int v = gl + 8 * k;
                        x[k] = on && v < V ? zp[v] : zero;
                        y[k] = on && v < V ? zq[v] : zero;
                    }
#pragma unroll
                    for (int k = 0; k < NV; ++k)
                        if (gl + 8 * k < CV) g += dot4(x[k], y[k]);
                } else {
                    for (int v = gl; on && v < CV; v += 8) g += dot4(zp[v], zq[v]);
                }
                g = sum8(g);
                const float root = sqrtf(a) * sqrtf(b), gm = fabsf(g);
                if (on && gm > tol * root && gm > floor_abs) {
                    if (gm > done * root && a > null2 && b > null2) rough = 1;
                    const float t = rotation_tan(b - a, g), h = half_tan(t), s = shear_sin(h, 0.0f);
                    if constexpr (NV > 0) {
#pragma unroll
                        for (int k = 0; k < NV; ++k) {
                            const int v = gl + 8 * k;
                            if (v < V) {
                                turn4(x[k], y[k], h, s);
                                zp[v] = x[k];
                                zq[v] = y[k];
                            }
                        }
                    } else {
                        for (int v = gl; v < V; v += 8) {
                            float4 u = zp[v], w = zq[v];
                            turn4(u, w, h, s);
                            zp[v] = u;
                            zq[v] = w;
                        }
                    }
                    if (gl < 2) nrm2[gl == 0 ? p : q] = fmaxf(fmaf(gl == 0 ? -t : t, g, gl == 0 ? a : b), 0.0f);
                }
            }
            __syncthreads();
        }
        if (!__syncthreads_or(rough)) break;
    }
}

// 1 / norm of a block, by all threads of a CTA.
__device__ double block_scale(const double* __restrict__ Z, int n) {
    __shared__ double red[32];
    __shared__ double tot;
    double s = 0.0;
    for (int e = threadIdx.x; e < n; e += blockDim.x) s = fma(Z[e], Z[e], s);
    s = wsum(s);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int i = 0; i < static_cast<int>(blockDim.x >> 5); ++i) t += red[i];
        tot = t;
    }
    __syncthreads();
    return tot > 0.0 ? 1.0 / sqrt(tot) : 0.0;
}

// FP32 start: [Z | I] of a block scaled to norm 1; J (R x R) leaves in FP64.  However its sweeps end, the FP64
// finish takes what they leave.
__global__ void __launch_bounds__(kOsj32Threads) k_osj32_smem(const SvdBlock* __restrict__ blocks, const double* __restrict__ zraw,
                                                              double* __restrict__ J, int smem_floats) {
    extern __shared__ float4 sm32[];
    const SvdBlock B = blocks[blockIdx.x];
    if (B.R <= 0 || B.C <= 0 || B.smem == 0) return;
    const int R = B.R, C = B.C, CV = (C + 3) / 4, V = CV + (R + 3) / 4, W = 4 * V;
    if (R * W + R > smem_floats) return;  // never: the host marks only blocks that fit
    const double* Zr = zraw + B.z_off;
    const double scale = block_scale(Zr, R * C);
    float* work = reinterpret_cast<float*>(sm32);
    for (int e = threadIdx.x; e < R * W; e += blockDim.x) {
        const int r = e / W, c = e - r * W;
        work[e] = c < C ? static_cast<float>(Zr[r * C + c] * scale) : (c - 4 * CV == r ? 1.0f : 0.0f);
    }
    __syncthreads();
    float* nrm2 = work + R * W;
    if (V <= 32)
        osj32_sweeps<4>(sm32, nrm2, R, CV, V);
    else if (V <= 56)
        osj32_sweeps<7>(sm32, nrm2, R, CV, V);
    else
        osj32_sweeps<0>(sm32, nrm2, R, CV, V);
    for (int r = threadIdx.x >> 5; r < R; r += blockDim.x >> 5) {
        const int to = row_rank(R, r, [&](int j) { return nrm2[j]; });
        for (int c = threadIdx.x & 31; c < R; c += 32)
            J[B.j_off + static_cast<int64_t>(to) * R + c] = static_cast<double>(work[r * W + 4 * CV + c]);
    }
}

__global__ void __cluster_dims__(kOsjC, 1, 1) __launch_bounds__(256)
    k_osj32_global(const SvdBlock* __restrict__ blocks, const double* __restrict__ zraw, float* __restrict__ works,
                   float* __restrict__ nrm, double* __restrict__ J, int* __restrict__ conv) {
    const int b = blockIdx.x / kOsjC, rank = static_cast<int>(cgx::this_cluster().block_rank());
    const SvdBlock B = blocks[b];
    if (B.R <= 0 || B.C <= 0 || B.smem != 0) return;  // uniform over the cluster
    const int R = B.R, C = B.C, W = C + R;
    const double* Zr = zraw + B.z_off;
    float* work = works + B.w_off;
    const double scale = block_scale(Zr, R * C);
    for (int e = rank * blockDim.x + threadIdx.x; e < R * W; e += blockDim.x * kOsjC) {
        const int r = e / W, c = e - r * W;
        __stcg(work + e, c < C ? static_cast<float>(Zr[static_cast<int64_t>(r) * C + c] * scale) : (c - C == r ? 1.0f : 0.0f));
    }
    cgx::this_cluster().sync();
    int* cv = conv + b * kSvdConv;
    if (W <= 256)
        osj_sweeps<float, 8>(work, nrm + B.n_off, R, C, W, 1.0f, 1e-3f, cv, rank, kOsjC, kFp32Sweeps);
    else
        osj_sweeps<float, 0>(work, nrm + B.n_off, R, C, W, 1.0f, 1e-3f, cv, rank, kOsjC, kFp32Sweeps);
    for (int r = (threadIdx.x >> 5) * kOsjC + rank; r < R; r += (blockDim.x >> 5) * kOsjC) {
        const int to = row_rank(R, r, [&](int j) { return __ldcg(nrm + B.n_off + j); });
        for (int c = threadIdx.x & 31; c < R; c += 32)
            J[B.j_off + static_cast<int64_t>(to) * R + c] = static_cast<double>(__ldcg(work + static_cast<int64_t>(r) * W + C + c));
    }
}

// FP64 finish on Z' (R x W, W = C, or C + R with the companion J): singular values squared, sorted
// descending, into evals (dim of them, zeros beyond the rank), and the wanted vectors as the columns of
// mats (dim x dim): the companion's rows, or the normalised rows of Z'.
__global__ void __cluster_dims__(kOsjC, 1, 1) __launch_bounds__(256)
    k_osj64(const SvdBlock* __restrict__ blocks, double* __restrict__ z, double* __restrict__ nrm, int* __restrict__ conv,
            double* __restrict__ mats, double* __restrict__ evals, int max_sweeps, int* __restrict__ unsettled) {
    __shared__ double red[32];
    __shared__ double tot;
    const int b = blockIdx.x / kOsjC;
    const SvdBlock B = blocks[b];
    if (B.dim <= 0) return;  // uniform over the cluster
    const int rank = static_cast<int>(cgx::this_cluster().block_rank());
    const int R = B.R, C = B.C, W = B.companion ? C + R : C;
    double* Z = z + B.f_off;
    double* nr = nrm + B.n_off;
    double s = 0.0;
    for (int e = threadIdx.x; e < R * C; e += blockDim.x) {
        const int r = e / C, c = e - r * C;
        const double v = __ldcg(Z + static_cast<int64_t>(r) * W + c);
        s = fma(v, v, s);
    }
    s = wsum(s);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int i = 0; i < static_cast<int>(blockDim.x >> 5); ++i) t += red[i];
        tot = t;
    }
    cgx::this_cluster().sync();  // every CTA has read Z before any rotates it
    if (!(tot < INFINITY)) {  // the block overflowed (the same sum in every CTA): no values, none of them is kept
        for (int rk = rank * blockDim.x + threadIdx.x; rk < B.dim; rk += blockDim.x * kOsjC) evals[B.e_off + rk] = 0.0;
        return;
    }
    int* cv = conv + (gridDim.x / kOsjC + b) * kSvdConv;
    // the companion is orthonormal by construction; normalised rows only as far as they are uncoupled
    const float done = B.companion ? 1e-11f : 1e-13f;
    bool settled;
    if (W <= 160)
        settled = osj_sweeps<double, 5>(Z, nr, R, C, W, tot, done, cv, rank, kOsjC, max_sweeps);
    else if (W <= 320)
        settled = osj_sweeps<double, 10>(Z, nr, R, C, W, tot, done, cv, rank, kOsjC, max_sweeps);
    else
        settled = osj_sweeps<double, 0>(Z, nr, R, C, W, tot, done, cv, rank, kOsjC, max_sweeps);
    if (!settled && rank == 0 && threadIdx.x == 0) *unsettled = 1;
    // exact norms of the final rows, then the vectors by descending norm (ties by row)
    const int lane = threadIdx.x & 31, warp = (threadIdx.x >> 5) * kOsjC + rank;
    const int warps = (blockDim.x >> 5) * kOsjC;
    for (int r = warp; r < R; r += warps) {
        double t = 0.0;
        for (int c = lane; c < C; c += 32) {
            const double v = __ldcg(Z + static_cast<int64_t>(r) * W + c);
            t = fma(v, v, t);
        }
        t = wsum(t);
        if (lane == 0) __stcg(nr + r, t);
    }
    cgx::this_cluster().sync();
    double* M = mats + B.m_off;
    double* ev = evals + B.e_off;
    const int n = B.dim;
    for (int r = warp; r < R; r += warps) {
        const double vr = __ldcg(nr + r);
        int rk = 0;
        for (int j = lane; j < R; j += 32) {
            const double vj = __ldcg(nr + j);
            rk += (vj > vr || (vj == vr && j < r)) ? 1 : 0;
        }
        rk = wsum(rk);
        if (rk >= n) continue;  // rows beyond the rank of the block (more rows than columns): noise
        if (lane == 0) ev[rk] = vr;
        const double inv = B.companion ? 1.0 : (vr > 0.0 ? 1.0 / sqrt(vr) : 0.0);
        const double* src = Z + static_cast<int64_t>(r) * W + (B.companion ? C : 0);
        for (int c = lane; c < n; c += 32) M[static_cast<int64_t>(c) * n + rk] = __ldcg(src + c) * inv;
    }
    for (int rk = R + warp; rk < n; rk += warps) {  // fewer rows than the dimension: the rest is null
        if (lane == 0) ev[rk] = 0.0;
        for (int c = lane; c < n; c += 32) M[static_cast<int64_t>(c) * n + rk] = 0.0;
    }
}

// Grouped FP64 products of the Newton-Schulz steps and of Z' = J Z: C = alpha A op(B) + diag 1, one CTA
// per 16 x 16 tile, K staged through shared memory in chunks of 32.  The FP64 pipe of an SM (2 FMA per clock)
// bounds a tile, so blocks of some tens of rows need tiles small enough for all SMs; a launch of the
// canonicalisation below takes 12 us (30 us with 32 x 32 tiles), of the middle decimation of L = 24, D = 256 26 us (66 us).
constexpr int kGemmTile = 16;
__global__ void __launch_bounds__(128) k_block_gemm(const double* __restrict__ a, const double* __restrict__ bm,
                                                    double* __restrict__ cm, const SvdGemm* __restrict__ gs,
                                                    const int3* __restrict__ tiles) {
    constexpr int KC = 32;
    __shared__ double As[KC][kGemmTile + 1], Bs[KC][kGemmTile + 1];
    const int3 tl = tiles[blockIdx.x];
    const SvdGemm G = gs[tl.x];
    const int m0 = tl.y, n0 = tl.z, tid = threadIdx.x;
    const double* A = a + G.a;
    const double* Bp = bm + G.b;
    const int tr = tid >> 3, tc = tid & 7;  // 16 x 8 threads, 1 x 2 outputs each
    double acc[2] = {0.0, 0.0};
    for (int k0 = 0; k0 < G.K; k0 += KC) {
#pragma unroll
        for (int e = tid; e < KC * kGemmTile; e += 128) {
            const int r = e / KC, k = e % KC;
            As[k][r] = (m0 + r < G.M && k0 + k < G.K) ? A[static_cast<int64_t>(m0 + r) * G.lda + k0 + k] : 0.0;
            if (G.transb) Bs[k][r] = (n0 + r < G.N && k0 + k < G.K) ? Bp[static_cast<int64_t>(n0 + r) * G.ldb + k0 + k] : 0.0;
        }
        if (!G.transb) {
#pragma unroll
            for (int e = tid; e < KC * kGemmTile; e += 128) {
                const int k = e / kGemmTile, c = e % kGemmTile;
                Bs[k][c] = (n0 + c < G.N && k0 + k < G.K) ? Bp[static_cast<int64_t>(k0 + k) * G.ldb + n0 + c] : 0.0;
            }
        }
        __syncthreads();
#pragma unroll 8
        for (int k = 0; k < min(KC, G.K - k0); ++k) {
            const double x = As[k][tr];
            acc[0] = fma(x, Bs[k][tc], acc[0]);
            acc[1] = fma(x, Bs[k][tc + 8], acc[1]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int r = m0 + tr, c = n0 + tc + 8 * j;
        if (r < G.M && c < G.N)
            cm[G.c + static_cast<int64_t>(r) * G.ldc + c] = G.alpha * acc[j] + (r == c ? G.diag : 0.0);
    }
}

// The companion columns of Z' of the blocks that keep J.
__global__ void __launch_bounds__(256) k_companion(const SvdBlock* __restrict__ blocks, const double* __restrict__ J,
                                                   double* __restrict__ z) {
    const SvdBlock B = blocks[blockIdx.x];
    if (!B.companion) return;
    const int W = B.C + B.R;
    for (int e = threadIdx.x; e < B.R * B.R; e += blockDim.x) {
        const int r = e / B.R, c = e - r * B.R;
        z[B.f_off + static_cast<int64_t>(r) * W + B.C + c] = J[B.j_off + e];
    }
}

template <class T>
cudaError_t put(T* dst, const std::vector<T>& v, cudaStream_t st) {
    if (v.empty()) return cudaSuccess;
    return cudaMemcpyAsync(dst, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice, st);
}

size_t up(size_t b) { return (b + 255) / 256 * 256; }

}  // namespace

void SvdPlan::build(const std::vector<SvdShape>& shapes, int smem_dim) {
    blocks.clear();
    gemms.clear();
    tiles.clear();
    gemm_rng.assign(1, 0);
    z_size = j_size = f_size = w_size = n_size = 0;
    smem_floats = max_rows = most_rows = 0;
    any_smem = any_global = any_companion = false;
    int64_t m_off = 0, e_off = 0;
    for (const SvdShape& s : shapes) {
        SvdBlock B{};
        // rows of the block itself (dim rows, their rotations kept as the companion), or of its transpose
        // (the vectors are the normalised rows): whichever needs fewer FP64 operations per sweep, the
        // product and the update counting 1 and 4 per element
        const double own = 1.0 * s.dim * s.dim * (5.0 * s.other + 4.0 * s.dim);
        const double trans = 1.0 * s.other * s.other * 5.0 * s.dim;
        B.companion = own <= trans ? 1 : 0;
        B.dim = s.dim;
        B.R = B.companion ? s.dim : s.other;
        B.C = B.companion ? s.other : s.dim;
        most_rows = std::max(most_rows, B.R);
        B.z_off = z_size;
        z_size += static_cast<int64_t>(B.R) * B.C;
        B.j_off = j_size;
        j_size += static_cast<int64_t>(B.R) * B.R;
        B.f_off = f_size;
        f_size += static_cast<int64_t>(B.R) * (B.C + (B.companion ? B.R : 0));
        B.n_off = n_size;
        n_size += B.R;
        const int64_t fl = static_cast<int64_t>(B.R) * ((B.C + 3) / 4 * 4 + (B.R + 3) / 4 * 4) + B.R;
        // shared memory while it fits and the caller's limit on the dimension allows it
        B.smem = (s.dim <= smem_dim || smem_dim >= kSvdSmemDefault) && fl <= kSvdSmemFloats ? 1 : 0;
        B.w_off = w_size;
        if (B.smem) {
            any_smem = true;
            max_rows = std::max(max_rows, B.R);
            smem_floats = std::max<int>(smem_floats, static_cast<int>(fl));
        } else {
            any_global = true;
            w_size += static_cast<int64_t>(B.R) * (B.C + B.R);
        }
        any_companion = any_companion || B.companion;
        B.m_off = m_off;
        B.e_off = e_off;
        m_off += static_cast<int64_t>(s.dim) * s.dim;
        e_off += s.dim;
        blocks.push_back(B);
    }
    // products: T = 3/2 - 1/2 J J^T, J' = T J (twice, the second pair back into J's place), Z' = J Z
    for (int step = 0; step < 5; ++step) {
        for (const SvdBlock& B : blocks) {
            SvdGemm G{};
            G.M = G.N = G.K = B.R;
            G.a = G.b = G.c = B.j_off;
            G.lda = G.ldb = G.ldc = B.R;
            G.alpha = 1.0;
            if (step == 0 || step == 2) {
                G.transb = 1;
                G.alpha = -0.5;
                G.diag = 1.5;
            }
            if (step == 4) {
                G.N = B.C;
                G.b = B.z_off;
                G.ldb = B.C;
                G.c = B.f_off;
                G.ldc = B.C + (B.companion ? B.R : 0);
            }
            for (int m0 = 0; m0 < G.M; m0 += kGemmTile)
                for (int n0 = 0; n0 < G.N; n0 += kGemmTile) tiles.push_back(make_int3(static_cast<int>(gemms.size()), m0, n0));
            gemms.push_back(G);
        }
        gemm_rng.push_back(static_cast<int>(tiles.size()));
    }
}

size_t SvdPlan::workspace() const {
    return up(blocks.size() * sizeof(SvdBlock)) + up(gemms.size() * sizeof(SvdGemm)) + up(tiles.size() * sizeof(int3)) +
           up(blocks.size() * 2 * kSvdConv * sizeof(int)) + up(z_size * 8) + 3 * up(j_size * 8) + up(f_size * 8) +
           up(w_size * 4) + up(n_size * 8) + up(n_size * 4);
}

double* SvdPlan::z_buffer(void* ws) const {
    return reinterpret_cast<double*>(static_cast<char*>(ws) + up(blocks.size() * sizeof(SvdBlock)) +
                                     up(gemms.size() * sizeof(SvdGemm)) + up(tiles.size() * sizeof(int3)) +
                                     up(blocks.size() * 2 * kSvdConv * sizeof(int)));
}

// Measured (GB300): the decimations of one canonicalisation (random L = 24, D = 256 triplet state, 23 of them,
// blocks up to 100 rows) take 17.5 ms, the middle decimation of the L = 24, D = 256 chain (blocks up to 126 rows)
// 5.3 ms; two-sided FP64 Jacobi on X X^T with a one-thread truncation took 308 and 22 ms.
cudaError_t launch_svd(const SvdPlan& P, void* ws, double* mats, double* evals, int* unsettled, cudaStream_t st) {
    const int nb = static_cast<int>(P.blocks.size());
    if (nb == 0) return cudaSuccess;
    if (P.most_rows > kSvdMaxRows || P.max_sweeps > kSvdConv) return cudaErrorInvalidValue;
    char* p = static_cast<char*>(ws);
    auto take = [&](size_t bytes) {
        char* q = p;
        p += up(bytes);
        return q;
    };
    auto* blocks = reinterpret_cast<SvdBlock*>(take(nb * sizeof(SvdBlock)));
    auto* gemms = reinterpret_cast<SvdGemm*>(take(P.gemms.size() * sizeof(SvdGemm)));
    auto* tiles = reinterpret_cast<int3*>(take(P.tiles.size() * sizeof(int3)));
    auto* conv = reinterpret_cast<int*>(take(static_cast<size_t>(nb) * 2 * kSvdConv * sizeof(int)));
    auto* z = reinterpret_cast<double*>(take(P.z_size * 8));
    auto* j0 = reinterpret_cast<double*>(take(P.j_size * 8));
    auto* j1 = reinterpret_cast<double*>(take(P.j_size * 8));
    auto* t0 = reinterpret_cast<double*>(take(P.j_size * 8));
    auto* f = reinterpret_cast<double*>(take(P.f_size * 8));
    auto* w = reinterpret_cast<float*>(take(P.w_size * 4));
    auto* n64 = reinterpret_cast<double*>(take(P.n_size * 8));
    auto* n32 = reinterpret_cast<float*>(take(P.n_size * 4));
    cudaError_t e = put(blocks, P.blocks, st);
    if (e == cudaSuccess) e = put(gemms, P.gemms, st);
    if (e == cudaSuccess) e = put(tiles, P.tiles, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(conv, 0, static_cast<size_t>(nb) * 2 * kSvdConv * sizeof(int), st);
    if (e != cudaSuccess) return e;
    if (P.any_smem) {
        const int bytes = P.smem_floats * static_cast<int>(sizeof(float));
        e = cudaFuncSetAttribute(k_osj32_smem, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kSvdSmemFloats * static_cast<int>(sizeof(float)));
        if (e != cudaSuccess) return e;
        const int threads = std::min(kOsj32Threads, std::max(64, ((P.max_rows + 1) / 2 * 8 + 31) / 32 * 32));  // 8 per pair
        k_osj32_smem<<<nb, threads, bytes, st>>>(blocks, z, j0, P.smem_floats);
    }
    if (P.any_global) k_osj32_global<<<nb * kOsjC, 256, 0, st>>>(blocks, z, w, n32, j0, conv);
    auto gemm = [&](int step, const double* a, const double* b, double* c) {
        const int lo = P.gemm_rng[step], hi = P.gemm_rng[step + 1];
        if (hi > lo) k_block_gemm<<<hi - lo, 128, 0, st>>>(a, b, c, gemms, tiles + lo);
    };
    gemm(0, j0, j0, t0);
    gemm(1, t0, j0, j1);
    gemm(2, j1, j1, t0);
    gemm(3, t0, j1, j0);
    gemm(4, j0, z, f);
    if (P.any_companion) k_companion<<<nb, 256, 0, st>>>(blocks, j0, f);
    k_osj64<<<nb * kOsjC, 256, 0, st>>>(blocks, f, n64, conv, mats, evals, P.max_sweeps, unsettled);
    return cudaGetLastError();
}

}  // namespace spmps
