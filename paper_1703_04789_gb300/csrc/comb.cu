// Phase B of the contraction plans on unrotated operators (see comb.h): host lists and kernels.
#include "comb.h"

#include <map>

namespace spmps {

namespace {

// Local states of a particle number m, ascending: one leg {0}, {b, a}, {ab}; two legs s = 4 s1 + s2.
__host__ __device__ constexpr int state_count(int legs, int m) {
    return legs == 1 ? (m == 1 ? 2 : 1) : (m == 0 || m == 4 ? 1 : (m == 2 ? 6 : 4));
}

// The states a state is joined to by the rotation of its legs, as a bit mask.
uint32_t rotation_mask(int legs, int t) {
    auto one = [](int x) -> uint32_t { return x == 1 || x == 2 ? 0x6u : 1u << x; };
    if (legs == 1) return one(t);
    uint32_t out = 0;
    for (int a = 0; a < 4; ++a)
        for (int b = 0; b < 4; ++b)
            if ((one(t >> 2) >> a & 1u) && (one(t & 3) >> b & 1u)) out |= 1u << (4 * a + b);
    return out;
}

// Above this many inputs a class no longer fits the fused kernel's shared memory at a useful occupancy
// (48 inputs x 128 elements x 8 bytes = 48 KB: four CTAs per SM).  A nearest-neighbour chain has at most 28
// inputs per class, a ten-orbital active space hundreds.
constexpr int kFusedInputs = 48;
constexpr int kFusedThreads = 128;

// Ket legs of one element rotated in place: (b, a) -> (c b + s a, -s b + c a) by three shears with
// t = tan(theta / 2), |t| < 1 (three FMA instead of four operations: the FP64 pipe bounds this phase).
__device__ __forceinline__ void shear(double& b, double& a, double t, double s) {
    b = fma(t, a, b);
    a = fma(-s, b, a);
    b = fma(t, a, b);
}
template <int LEGS>
__device__ __forceinline__ void rotate(double* v, int m, double t, double s) {
    if constexpr (LEGS == 1) {
        if (m == 1) shear(v[0], v[1], t, s);
    } else {
        if (m == 1 || m == 3) {
            shear(v[0], v[1], t, s);
            shear(v[2], v[3], t, s);
        } else if (m == 2) {  // (0,ab), (b,b), (b,a), (a,b), (a,a), (ab,0)
            shear(v[1], v[2], t, s);
            shear(v[3], v[4], t, s);
            shear(v[1], v[3], t, s);
            shear(v[2], v[4], t, s);
        }
    }
}

// Fused form for classes of few inputs: one thread per element of a (row group, column group) pair reads
// each of its inputs once (asynchronous copies into its own column of shared memory, all in flight at
// once), rotates them there and forms all outputs.  T1 is read once and T3 written once.  The FP64 pipe
// (2 FMA per clock and SM) is the first bound: three FMA per rotated pair of states, one per
// coefficient other than a leading 1; the pair's records are staged in shared memory so that no chain of
// global loads stands in front of them.  Measured (GB300, middle action of the L = 24, D = 256, n_beta = 8
// chain, 12 M elements read and written): 109 us; the form with rotated coefficients, one CTA per output
// block and every term read from L2, took 162 us after a zero fill of T1 of 23 us.
constexpr int kStageIns = kFusedInputs, kStageDsts = 64, kStageCoefs = 128;

template <int LEGS>
__global__ void __launch_bounds__(kFusedThreads) k_comb_pair(const __grid_constant__ Slots S, const __grid_constant__ CombDev D, int unit0, int g0, int shared) {
    extern __shared__ double vin[];
    __shared__ CombIn sins[kStageIns];
    __shared__ CombSet ssets[kStageIns];
    __shared__ CombDst sdsts[kStageDsts];
    __shared__ CombCoef scoefs[kStageCoefs];
    const int2 U = D.units[unit0 + blockIdx.x];
    const CombPair P = D.pairs[U.x];
    const int g = g0 + blockIdx.y, tid = threadIdx.x;
    const int nmore = shared ? P.nmore : 0, nd = P.ndst + nmore;
    const bool staged = nd <= kStageDsts && P.ncoef <= kStageCoefs;
    for (int i = tid; i < P.nin; i += kFusedThreads) sins[i] = D.ins[P.in0 + i];
    for (int i = tid; i < P.nset; i += kFusedThreads) ssets[i] = D.sets[P.set0 + i];
    if (staged) {
        for (int i = tid; i < nd; i += kFusedThreads) sdsts[i] = D.dsts[i < P.ndst ? P.dst0 + i : P.more0 + i - P.ndst];
        for (int i = tid; i < P.ncoef; i += kFusedThreads) scoefs[i] = D.coefs[P.coef0 + i];
    }
    __syncthreads();
    const int e = U.y + tid;
    if (e >= P.rows * P.cols) return;
    const int r = e / P.cols, c = e - r * P.cols;
    const double* __restrict__ T1 = S.p[3] + g * D.stride.t1[P.op];
    const int lab = D.lab[P.lab0 + c];
    const double rt = D.rot[2 * g], rs = D.rot[2 * g + 1];
    double* v = vin + tid;
#pragma unroll 4
    for (int i = 0; i < P.nin; ++i) {
        const bool ok = sins[i].off >= 0 && (sins[i].mask >> lab & 1ull);
        const uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(v + i * kFusedThreads));
        if (ok)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst),
                         "l"(T1 + sins[i].off + r * sins[i].ld + c));
        else
            v[i * kFusedThreads] = 0.0;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    for (int i = 0; i < P.nset; ++i) {  // only this thread's column: no barrier
        const int m = ssets[i].m;
        if (m == 0 || m == 2 * LEGS || sins[ssets[i].in].off < 0) continue;
        double* w = v + ssets[i].in * kFusedThreads;
        double x[LEGS == 1 ? 2 : 6];
        const int n = state_count(LEGS, m);
#pragma unroll
        for (int q = 0; q < (LEGS == 1 ? 2 : 6); ++q) x[q] = q < n ? w[q * kFusedThreads] : 0.0;
        rotate<LEGS>(x, m, rt, rs);
#pragma unroll
        for (int q = 0; q < (LEGS == 1 ? 2 : 6); ++q)
            if (q < n) w[q * kFusedThreads] = x[q];
    }
#pragma unroll 2
    for (int o = 0; o < nd; ++o) {
        const CombDst& d = staged ? sdsts[o] : D.dsts[o < P.ndst ? P.dst0 + o : P.more0 + o - P.ndst];
        const CombCoef* k = staged ? scoefs + (d.term0 - P.coef0) : D.coefs + d.term0;
        if (r < d.row0 || r >= d.row0 + d.rows) continue;
        double acc = 0.0;
        for (int t = 0; t < d.nterm; ++t) {
            const double x = v[k[t].in * kFusedThreads];
            if (t == 0)
                acc = k[t].unit ? x : k[t].coef * x;
            else
                acc = fma(k[t].coef, x, acc);
        }
        (S.p[4] + g * D.stride.t3[d.op])[d.off + static_cast<int64_t>(r) * d.ld + c] = acc;
    }
}

// Separate rotation of T1 in place for classes of many inputs: one CTA per (pair, channel).
template <int LEGS>
__global__ void __launch_bounds__(256) k_comb_rotate(const __grid_constant__ Slots S, const __grid_constant__ CombDev D, int rot0, int g0) {
    const int2 U = D.rots[rot0 + blockIdx.x];
    const CombPair P = D.pairs[U.x];
    const CombSet st = D.sets[P.set0 + U.y];
    const CombIn* in = D.ins + P.in0 + st.in;
    const int g = g0 + blockIdx.y, n = state_count(LEGS, st.m), total = P.rows * P.cols;
    double* T1 = S.p[3] + g * D.stride.t1[P.op];
    const double rt = D.rot[2 * g], rs = D.rot[2 * g + 1];
    for (int e = threadIdx.x; e < total; e += blockDim.x) {
        const int r = e / P.cols, c = e - r * P.cols;
        const int lab = D.lab[P.lab0 + c];
        double v[LEGS == 1 ? 2 : 6];
#pragma unroll
        for (int q = 0; q < (LEGS == 1 ? 2 : 6); ++q)
            v[q] = q < n && (in[q].mask >> lab & 1ull) ? T1[in[q].off + static_cast<int64_t>(r) * in[q].ld + c] : 0.0;
        rotate<LEGS>(v, st.m, rt, rs);
#pragma unroll
        for (int q = 0; q < (LEGS == 1 ? 2 : 6); ++q)
            if (q < n) T1[in[q].off + static_cast<int64_t>(r) * in[q].ld + c] = v[q];
    }
}

// Separate combination: one CTA per output block and beta point, four elements per thread, so that a
// term's record is read once per four FMA.  Bound by the FP64 pipe (84 % of its cycles active; 121 terms
// per output on average at K = 20); the inputs of a beta point come from L2.  Measured (K = 20, D = 100,
// n_beta = 12, middle action): 25.2 ms for the phase, 95.7 ms with rotated coefficients (2.2 times the
// nonzeros) and without leaving out the rows that phase C does not read.
__global__ void __launch_bounds__(128) k_comb_list(const __grid_constant__ Slots S, const __grid_constant__ CombDev D, int out0, int n_out, int g0) {
    constexpr int E = 4;
    const int ob = blockIdx.x;  // operator 0's (or 1's) blocks, then operator 1's on operator 0's T1
    const CombDst d = D.dsts[D.outs[ob < n_out ? out0 + ob : D.shared0 + ob - n_out]];
    const CombPair P = D.pairs[d.pair];
    const int g = g0 + blockIdx.y, total = d.rows * P.cols;
    const double* __restrict__ T1 = S.p[3] + g * D.stride.t1[P.op];
    double* __restrict__ T3 = S.p[4] + g * D.stride.t3[d.op] + d.off;
    const CombIn* __restrict__ ins = D.ins + P.in0;
    const CombCoef* __restrict__ coefs = D.coefs + d.term0;
    for (int base = threadIdx.x; base - (threadIdx.x & 31) < total; base += 128 * E) {
        int row[E], col[E];
        double acc[E];
        int live = 0;  // elements of this warp, uniform over it
#pragma unroll
        for (int i = 0; i < E; ++i) {
            const int e = base + 128 * i;
            live += e - (static_cast<int>(threadIdx.x) & 31) < total ? 1 : 0;
            const int ee = e < total ? e : 0;
            row[i] = d.row0 + ee / P.cols;
            col[i] = ee - (row[i] - d.row0) * P.cols;
            acc[i] = 0.0;
        }
#pragma unroll 2
        for (int t = 0; t < d.nterm; ++t) {
            const CombCoef k = coefs[t];
            const int64_t off = ins[k.in].off;
            const int ld = ins[k.in].ld;
            if (off < 0) continue;
            const double* p = T1 + off;
#pragma unroll
            for (int i = 0; i < E; ++i)
                if (i < live) acc[i] = fma(k.coef, __ldg(p + row[i] * ld + col[i]), acc[i]);
        }
#pragma unroll
        for (int i = 0; i < E; ++i)
            if (base + 128 * i < total) T3[static_cast<int64_t>(row[i]) * d.ld + col[i]] = acc[i];
    }
}

}  // namespace

double comb_add(CombChan& C, const CombSpec& sp) {
    const int ns = sp.legs == 1 ? 4 : 16, mmax = 2 * sp.legs;
    const int nrow = static_cast<int>(sp.row->groups.size()), ncol = static_cast<int>(sp.col->groups.size());
    const std::vector<int>&cin = *sp.cn_in, &cout = *sp.cn_out;
    const int nw = static_cast<int>(cin.size()), nu = static_cast<int>(cout.size());
    C.legs = sp.legs;
    if (C.unit_rng.empty()) {
        C.unit_rng.assign(1, 0);
        C.rot_rng.assign(1, 0);
        C.out_rng.assign(1, 0);
        C.lab.assign(sp.col->D, 0);
        for (const Group& G : sp.col->groups) C.zero_t1 = C.zero_t1 || G.count > 63;
        for (const Group& G : sp.col->groups)
            for (int j = 0; j < G.count; ++j) {
                const Label& L = sp.col->labels[G.first + j];
                for (int i = 0; i < L.dim; ++i) C.lab[L.off + i] = static_cast<uint8_t>(std::min(j, 63));
            }
    }
    std::vector<std::vector<int>> states(mmax + 1);
    for (int t = 0; t < ns; ++t) states[qn_n(ns, t)].push_back(t);
    struct Out {
        int u, s, term0, nterm;
        std::vector<std::pair<int, int>> rotated;  // (set, nonzeros of the rotated operator)
    };
    struct Class {
        std::vector<CombSet> sets;
        std::vector<Out> outs;
        int nin = 0, coef0 = 0, ncoef = 0, share_in = -1;
    };
    std::map<int, Class> classes;
    double flops = 0.0;
    const int pair0 = static_cast<int>(C.pairs.size());
    int widest = 0;
    for (int ga = 0; ga < nrow; ++ga)
        for (int gb = 0; gb < ncol; ++gb) {
            // n(t) - sign * charge = d
            const int d = sp.sign > 0 ? sp.col->groups[gb].n - sp.row->groups[ga].n
                                      : sp.row->groups[ga].n - sp.col->groups[gb].n;
            auto it = classes.find(d);
            if (it == classes.end()) {
                it = classes.emplace(d, Class()).first;
                Class& K = it->second;
                K.coef0 = static_cast<int>(C.coefs.size());
                std::vector<int> first(nw, -1), set_of(nw, -1);
                for (int w = 0; w < nw; ++w) {
                    const int m = d + sp.sign * cin[w];
                    if (m < 0 || m > mmax) continue;
                    set_of[w] = static_cast<int>(K.sets.size());
                    first[w] = K.nin;
                    K.sets.push_back({w, m, K.nin});
                    K.nin += static_cast<int>(states[m].size());
                }
                std::vector<int> place(ns, 0);
                for (int m = 0; m <= mmax; ++m)
                    for (size_t q = 0; q < states[m].size(); ++q) place[states[m][q]] = static_cast<int>(q);
                for (int u = 0; u < nu; ++u) {
                    const int m = d + sp.sign * cout[u];
                    if (m < 0 || m > mmax) continue;
                    for (int s : states[m]) {
                        Out o{u, s, static_cast<int>(C.coefs.size()), 0, {}};
                        uint32_t bits = 0;
                        int lastw = -1;
                        auto flush = [&]() {
                            if (lastw >= 0 && bits) o.rotated.push_back({set_of[lastw], __builtin_popcount(bits)});
                            bits = 0;
                        };
                        for (const ChanEntry& e : (*sp.entries)[u]) {
                            if (e.s != s || e.coef == 0.0 || first[e.w] < 0) continue;
                            if (e.w != lastw) {
                                flush();
                                lastw = e.w;
                            }
                            bits |= rotation_mask(sp.legs, e.t);
                            C.coefs.push_back({e.coef, first[e.w] + place[e.t], e.coef == 1.0 ? 1 : 0});
                        }
                        flush();
                        o.nterm = static_cast<int>(C.coefs.size()) - o.term0;
                        K.outs.push_back(std::move(o));
                    }
                }
                if (sp.share >= 0 && first[sp.share] >= 0) {  // operator 1's outputs: copies of that channel
                    K.share_in = static_cast<int>(C.coefs.size());
                    for (int q = 0; q < static_cast<int>(states[d + sp.sign * cin[sp.share]].size()); ++q)
                        C.coefs.push_back({1.0, first[sp.share] + q, 1});
                }
                K.ncoef = static_cast<int>(C.coefs.size()) - K.coef0;
            }
            const Class& K = it->second;
            if (K.outs.empty() && K.share_in < 0) continue;  // operator 1 may have outputs where this one has none
            CombPair P{};
            P.op = sp.op;
            P.rows = sp.row->groups[ga].dim;
            P.cols = sp.col->groups[gb].dim;
            P.lab0 = sp.col->groups[gb].off;
            P.in0 = static_cast<int>(C.ins.size());
            P.nin = K.nin;
            P.set0 = static_cast<int>(C.sets.size());
            P.nset = static_cast<int>(K.sets.size());
            P.dst0 = static_cast<int>(C.dsts.size());
            std::vector<char> present(K.sets.size(), 0);
            const Group& GB = sp.col->groups[gb];
            const Group& GA = sp.row->groups[ga];
            for (size_t i = 0; i < K.sets.size(); ++i) {
                const CombSet& st = K.sets[i];
                const int64_t o1 = (*sp.o1)[static_cast<size_t>(st.w) * nrow + ga];
                const ColLayout& L = (*sp.c1)[static_cast<size_t>(st.w) * nrow + ga];
                present[i] = o1 >= 0;
                for (int t : states[st.m]) {
                    CombIn in{};
                    in.off = -1;
                    if (o1 >= 0) {
                        in.off = o1 + L.col[t];
                        in.ld = L.width;
                        for (int j = 0; j < GB.count; ++j) {
                            const Label& B = sp.col->labels[GB.first + j];
                            if (j >= 63)
                                in.mask |= 1ull << 63;  // one bit for the rest: T1 starts at zero then
                            else if (sp.ket->find(B.n - sp.sign * qn_n(ns, t), B.tm - sp.sign * qn_m(ns, t)) >= 0)
                                in.mask |= 1ull << j;
                        }
                    }
                    C.ins.push_back(in);
                }
                C.sets.push_back(st);
            }
            for (const Out& o : K.outs) {
                const int64_t o2 = (*sp.o2)[static_cast<size_t>(o.u) * nrow + ga];
                if (o2 < 0) continue;
                const ColLayout& L = (*sp.c2)[static_cast<size_t>(o.u) * nrow + ga];
                for (const auto& rz : o.rotated)
                    if (present[rz.first]) flops += 2.0 * P.rows * P.cols * rz.second;
                int lo = -1, hi = -1;  // rows from the first to the last label that phase C reads
                for (int j = 0; j < GA.count; ++j)
                    if (sp.needed(GA.first + j, o.s)) {
                        if (lo < 0) lo = sp.row->labels[GA.first + j].off - GA.off;
                        hi = sp.row->labels[GA.first + j].off - GA.off + sp.row->labels[GA.first + j].dim;
                    }
                if (lo < 0) continue;
                CombDst D{};
                D.off = o2 + L.col[o.s];
                D.ld = L.width;
                D.row0 = lo;
                D.rows = hi - lo;
                D.term0 = o.term0;
                D.nterm = o.nterm;
                D.pair = static_cast<int>(C.pairs.size());
                D.op = sp.op;
                C.dsts.push_back(D);
            }
            P.ndst = static_cast<int>(C.dsts.size()) - P.dst0;
            P.more0 = static_cast<int>(C.dsts.size());
            P.coef0 = K.coef0;
            P.ncoef = K.ncoef;
            const int64_t so = sp.share >= 0 && K.share_in >= 0 ? (*sp.share_o2)[ga] : -1;
            if (so >= 0 && (*sp.o1)[static_cast<size_t>(sp.share) * nrow + ga] >= 0) {
                const std::vector<int>& st = states[d + sp.sign * cin[sp.share]];
                for (size_t q = 0; q < st.size(); ++q) {
                    int lo = -1, hi = -1;
                    for (int j = 0; j < GA.count; ++j)
                        if (sp.needed(GA.first + j, st[q])) {
                            if (lo < 0) lo = sp.row->labels[GA.first + j].off - GA.off;
                            hi = sp.row->labels[GA.first + j].off - GA.off + sp.row->labels[GA.first + j].dim;
                        }
                    if (lo < 0) continue;
                    CombDst D{};
                    D.off = so + (*sp.share_c2)[ga].col[st[q]];
                    D.ld = (*sp.share_c2)[ga].width;
                    D.row0 = lo;
                    D.rows = hi - lo;
                    D.term0 = K.share_in + static_cast<int>(q);
                    D.nterm = 1;
                    D.pair = static_cast<int>(C.pairs.size());
                    D.op = 1;
                    C.dsts.push_back(D);
                }
            }
            P.nmore = static_cast<int>(C.dsts.size()) - P.more0;
            if (P.ndst + P.nmore == 0) {
                C.ins.resize(P.in0);
                C.sets.resize(P.set0);
                continue;
            }
            widest = std::max(widest, P.nin);
            C.pairs.push_back(P);
        }
    const bool fused = widest <= kFusedInputs;
    for (int p = pair0; p < static_cast<int>(C.pairs.size()); ++p) {
        const CombPair& P = C.pairs[p];
        if (fused) {
            for (int e = 0; e < P.rows * P.cols; e += kFusedThreads) C.units.push_back(make_int2(p, e));
            continue;
        }
        for (int i = 0; i < P.nset; ++i) {
            const CombSet& st = C.sets[P.set0 + i];
            const CombIn* in = &C.ins[P.in0 + st.in];
            if (in[0].off < 0) continue;
            // columns of the pair: every label of its column group
            uint64_t labels = 0;
            for (int c = 0; c < P.cols; ++c) labels |= 1ull << C.lab[P.lab0 + c];
            bool whole = true;
            for (int q = 0; q < state_count(sp.legs, st.m); ++q) whole = whole && (in[q].mask & labels) == labels;
            const bool still = st.m == 0 || st.m == mmax;  // nothing to rotate
            if (!still || !whole) C.rots.push_back(make_int2(p, i));
        }
        for (int o = 0; o < P.ndst; ++o) C.outs.push_back(P.dst0 + o);
        for (int o = 0; o < P.nmore; ++o) C.shared_outs.push_back(P.more0 + o);
    }
    if (sp.share >= 0) C.shares = true;
    if (fused) C.max_nin = std::max(C.max_nin, widest);
    C.unit_rng.push_back(static_cast<int>(C.units.size()));
    C.rot_rng.push_back(static_cast<int>(C.rots.size()));
    C.out_rng.push_back(static_cast<int>(C.outs.size()));
    return flops;
}

bool comb_check(const CombChan& C, int G, int64_t t1, int64_t t3, std::string* why) {
    auto bad = [&](const char* m) {
        *why = m;
        return false;
    };
    for (const CombPair& P : C.pairs) {
        if (P.rows <= 0 || P.cols <= 0 || P.op < 0 || P.op > 1) return bad("bad combination pair");
        if (P.lab0 < 0 || P.lab0 + P.cols > static_cast<int>(C.lab.size())) return bad("combination columns out of range");
        if (P.in0 < 0 || P.in0 + P.nin > static_cast<int>(C.ins.size())) return bad("combination inputs out of range");
        for (int i = 0; i < P.nset; ++i) {
            const CombSet& st = C.sets[P.set0 + i];
            if (st.m < 0 || st.m > 2 * C.legs || st.in < 0 || st.in + state_count(C.legs, st.m) > P.nin)
                return bad("bad combination set");
        }
        for (int i = 0; i < P.nin; ++i) {
            const CombIn& in = C.ins[P.in0 + i];
            if (in.off < 0) continue;
            if (in.off + (G - 1) * C.stride.t1[P.op] + static_cast<int64_t>(P.rows - 1) * in.ld + P.cols - 1 >= t1 || in.ld < P.cols)
                return bad("combination input out of range");
        }
        for (int o = 0; o < P.ndst + P.nmore; ++o) {
            const CombDst& d = C.dsts[o < P.ndst ? P.dst0 + o : P.more0 + o - P.ndst];
            if (d.op < 0 || d.op > 1 || d.term0 < P.coef0 || d.term0 + d.nterm > P.coef0 + P.ncoef ||
                P.coef0 + P.ncoef > static_cast<int>(C.coefs.size()))
                return bad("bad combination output");
            if (d.row0 < 0 || d.rows <= 0 || d.row0 + d.rows > P.rows || d.ld < P.cols || d.off < 0 ||
                d.off + (G - 1) * C.stride.t3[d.op] + static_cast<int64_t>(d.row0 + d.rows - 1) * d.ld + P.cols - 1 >= t3)
                return bad("combination output out of range");
            for (int t = 0; t < d.nterm; ++t)
                if (C.coefs[d.term0 + t].in < 0 || C.coefs[d.term0 + t].in >= P.nin) return bad("combination term out of range");
        }
    }
    return true;
}

cudaError_t launch_comb_chan(const Slots& slots, const CombChan& C, const CombDev& D, int op0, int op1, int g0, int ng,
                             bool shared, int64_t* launches, cudaStream_t st) {
    const int last = shared ? op0 + 1 : op1;  // operators whose own T1 is read
    const int u0 = C.unit_rng[op0], u1 = C.unit_rng[last];
    if (u1 > u0) {
        const int smem = C.max_nin * kFusedThreads * static_cast<int>(sizeof(double));
        const dim3 grid(u1 - u0, ng);
        static int attr_device = -1;  // static and dynamic shared memory together pass 48 KB
        int dev = 0;
        cudaGetDevice(&dev);
        if (attr_device != dev) {
            constexpr int most = kFusedInputs * kFusedThreads * static_cast<int>(sizeof(double));
            cudaError_t e = cudaFuncSetAttribute(k_comb_pair<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
            if (e == cudaSuccess) e = cudaFuncSetAttribute(k_comb_pair<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
            if (e != cudaSuccess) return e;
            attr_device = dev;
        }
        if (C.legs == 1)
            k_comb_pair<1><<<grid, kFusedThreads, smem, st>>>(slots, D, u0, g0, shared ? 1 : 0);
        else
            k_comb_pair<2><<<grid, kFusedThreads, smem, st>>>(slots, D, u0, g0, shared ? 1 : 0);
        ++*launches;
    }
    const int r0 = C.rot_rng[op0], r1 = C.rot_rng[last];
    if (r1 > r0) {
        if (C.legs == 1)
            k_comb_rotate<1><<<dim3(r1 - r0, ng), 256, 0, st>>>(slots, D, r0, g0);
        else
            k_comb_rotate<2><<<dim3(r1 - r0, ng), 256, 0, st>>>(slots, D, r0, g0);
        ++*launches;
    }
    const int o0 = C.out_rng[op0], n = C.out_rng[last] - o0;
    const int more = shared ? static_cast<int>(C.shared_outs.size()) : 0;
    if (n + more > 0) {
        k_comb_list<<<dim3(n + more, ng), 128, 0, st>>>(slots, D, o0, n, g0);
        ++*launches;
    }
    return cudaGetLastError();
}

}  // namespace spmps
