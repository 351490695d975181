// The MPO-leg combination of the contraction plans (phase B), on unrotated operators (comb.cu).
//
// The rotation exp(-i beta S_y) multiplies the ket leg of every MPO site (Eq. expSy), so phase B is a
// rotation of the ket legs of T1, which mixes only the singly occupied states, followed by the unrotated
// operator.  The operator's coefficients depend on neither the beta point nor the bra group: for a
// row group of n particles and a column group of n + d, the inputs are the (channel w, local state t) with
// n(t) - charge(w) = d, the outputs the (u, s) with n(s) - charge(u) = d, and one sparse matrix per d joins
// them for every pair of groups with that d and every beta point.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <functional>
#include <string>
#include <vector>

#include "core.h"

namespace spmps {

// W[w, u, s, t] of one site, or of two sites contracted over their bond (s = 4 s1 + s2).
struct ChanEntry {
    int w, s, t;
    double coef;
};

struct CombIn {
    int64_t off;    // first element (row 0, column 0) of the input in T1 for beta point 0; -1: absent (zero)
    uint64_t mask;  // bit j: phase A writes the columns of label j of the column group (else they are zero)
    int ld, pad;
};
struct CombSet {
    int w, m, in;   // channel, particle number of its local states, first input of the class
};
struct CombDst {
    int64_t off;    // row 0 of the row group, first column, in T3 for beta point 0
    int ld, row0, rows;  // only the rows that phase C reads
    int term0, nterm, pair, op, pad;
};
struct CombCoef {
    double coef;
    int in, unit;   // unit 1: the coefficient is 1 (a copy or an addition needs no multiplication)
};
struct CombPair {
    int in0, nin, set0, nset;
    int dst0, ndst;       // its operator's outputs
    int more0, nmore;     // outputs of operator 1 that read operator 0's T1 (CombSpec::share)
    int coef0, ncoef;     // the coefficients of the class
    int rows, cols, lab0, op;
};
struct CombOpStride {
    int64_t t1[2], t3[2];  // elements between consecutive beta points, per operator
};

struct CombChan {
    std::vector<CombIn> ins;
    std::vector<CombSet> sets;
    std::vector<CombDst> dsts;
    std::vector<CombCoef> coefs;
    std::vector<CombPair> pairs;
    std::vector<uint8_t> lab;    // label index inside its group, per column of the column bond
    std::vector<int2> units;     // (pair, first element) of the fused form
    std::vector<int2> rots;      // (pair, set) of the separate rotation
    std::vector<int> outs;       // destination of each block of the separate combination
    std::vector<int> unit_rng, rot_rng, out_rng;  // per operator
    std::vector<int> shared_outs;  // blocks of operator 1 on operator 0's T1, after outs
    bool shares = false;         // operator 1 may read operator 0's T1 (both wanted: its phase A is not run)
    CombOpStride stride{};
    int legs = 0, max_nin = 0;
    bool zero_t1 = false;        // a column group has more labels than a mask has bits
    void clear() { *this = CombChan(); }
};

// What phase B of one operator reads and writes (offsets for beta point 0).
struct CombSpec {
    int op = 0, legs = 1, sign = 1;  // column group of (block, t): n(row) - charge + sign n(t) (sign +1), or
                                     // n(row) - charge - n(t) (sign -1)
    const Bond *row = nullptr, *col = nullptr;
    const Bond* ket = nullptr;       // bond of the label that phase A contracted
    const std::vector<int>*cn_in = nullptr, *cn_out = nullptr;
    const std::vector<int64_t>*o1 = nullptr, *o2 = nullptr;  // [channel * groups + row group], -1 absent
    const std::vector<ColLayout>*c1 = nullptr, *c2 = nullptr;
    const std::vector<std::vector<ChanEntry>>* entries = nullptr;  // per output channel, by (w, s, t)
    std::function<bool(int label, int s)> needed;                  // whether phase C reads row label, state s
    // operator 0 only: channel whose T1 is operator 1's (-1: none), and operator 1's T3 blocks per row group
    int share = -1;
    const std::vector<int64_t>* share_o2 = nullptr;
    const std::vector<ColLayout>* share_c2 = nullptr;
};

// Appends one operator's phase B; returns its algorithmic flops for one beta point (2 per element and
// nonzero of the rotated operator, all rows of every block).
double comb_add(CombChan& C, const CombSpec& spec);
// Every element lies inside T1 (size t1) and T3 (size t3) for all G beta points.
bool comb_check(const CombChan& C, int G, int64_t t1, int64_t t3, std::string* why);

struct CombDev {
    const CombIn* ins;
    const CombSet* sets;
    const CombDst* dsts;
    const CombCoef* coefs;
    const CombPair* pairs;
    const uint8_t* lab;
    const int2* units;
    const int2* rots;
    const int* outs;
    int shared0;        // first of operator 1's blocks on operator 0's T1 in outs
    const double* rot;  // per beta point tan(beta / 4), sin(beta / 2)
    CombOpStride stride;
};

// Phase B of operators [op0, op1) and beta points [g0, g0 + ng); with `shared` operator 1's outputs are
// formed from operator 0's T1 (op0 = 0, op1 = 2).  *launches counts the kernels.
cudaError_t launch_comb_chan(const Slots& slots, const CombChan& C, const CombDev& D, int op0, int op1, int g0, int ng,
                             bool shared, int64_t* launches, cudaStream_t st);

}  // namespace spmps
