// Shared by the kernels of the joint generating functions (k_bin2d.cu,
// k_gf2d_tc.cu): the grid, the slots of the chunk's union window, the
// per-trajectory constants.
#pragma once

#include "dfloat.cuh"
#include "gbs_internal.cuh"

namespace gbs {
namespace bin2d {

// Shape of one launch over the grid (passed by value).
struct GridD {
    int d;                   // bins
    int K[kMaxBins];         // points per dimension
    int Koff[kMaxBins];      // offsets of each dimension's tables
    int tile[kMaxBins + 1];  // bin b = GEMM tiles [tile[b], tile[b + 1])
};

__device__ __forceinline__ int slots_of(int K, int W1, int W2) {
    const int half = K >> 1;
    const int n1 = W1 >= half ? K : 2 * W1 + 1;
    const int n2 = W2 < 0 ? 0 : (W2 >= half ? K : 2 * W2 + 1);
    return n1 + n2 >= K ? K : n1 + n2;
}

// k of slot i of one dimension: the window around 0 (k = -W1..W1), then the
// one around K/2; the whole range when they cover it.
__device__ __forceinline__ int slot_k(int i, int K, int W1, int W2) {
    const int half = K >> 1;
    const int n1 = W1 >= half ? K : 2 * W1 + 1;
    const int n2 = W2 < 0 ? 0 : (W2 >= half ? K : 2 * W2 + 1);
    if (n1 + n2 >= K) return i;
    if (i < n1) {
        const int k = i - W1;
        return k < 0 ? k + K : k;
    }
    return half - W2 + (i - n1);
}

// Slots of the union window per dimension.
struct Slots {
    int S[kMaxBins];
    int W1[kMaxBins], W2[kMaxBins];
};

__device__ __forceinline__ Slots slots_of_grid(const GridD &g, const int *wmax) {
    Slots s;
#pragma unroll
    for (int b = 0; b < kMaxBins; ++b) {
        s.W1[b] = wmax[b];
        s.W2[b] = wmax[kMaxBins + b];
        s.S[b] = b < g.d ? slots_of(g.K[b], s.W1[b], s.W2[b]) : 1;
    }
    return s;
}

// Dimensions [0, nb) of the flattened slot index idx (last of them fastest)
// -> k_b; returns the row-major grid index over those dimensions.
__device__ __forceinline__ int64_t slot_ks(const GridD &g, const Slots &s, int nb, int64_t idx,
                                           int (&k)[kMaxBins]) {
    int64_t rem = idx;
#pragma unroll
    for (int b = kMaxBins - 1; b >= 0; --b) {
        if (b >= nb) continue;
        const int sb = (int)(rem % s.S[b]);
        rem /= s.S[b];
        k[b] = slot_k(sb, g.K[b], s.W1[b], s.W2[b]);
    }
    int64_t o = 0;
#pragma unroll
    for (int b = 0; b < kMaxBins; ++b)
        if (b < nb) o = o * g.K[b] + k[b];
    return o;
}

// Per-trajectory constants of the factorised evaluation (one pass per chunk):
// the bins' n_S and the exponent offsets, V = df (BF16 networks) or double.
template <typename V>
struct __align__(16) SepTrajT {
    V x[kMaxBins], y[kMaxBins];  // n_Sb
    V m2, mp2;          // M_B, M'_B (offsets of the second factors)
    V o1a, o1b;         // offsets of the first factors: +M_B, +M'_B + c2 + log inv
    V rA;               // inv e^{c1} (<= 1)
    int flags;          // kSep... below
    float top;          // bound of the log of the first factor's magnitude
};
using SepTraj = SepTrajT<df>;
using SepTraj64 = SepTrajT<double>;
static_assert(sizeof(SepTraj) == sizeof(SepTraj64), "k_sep_lists reads flags and top of either");
constexpr int kSepPoint = 2;   // per-point FP64 route
constexpr int kSepB = 4;       // B term used
constexpr int kSepOne = 8;     // rA == 1
constexpr int kSepNone = 16;   // no trajectory
// log of the largest first factor that k_gf2d_tc's fixed-point factors take:
// their resolution is 2^-55 of the sub-ensemble's largest one, 2^-47 with this
// bound, the double-float factors' own relative error
constexpr float kSepTcTop = 5.5f;
// the same for FP64 factors, whose exponents and phases, |n_Sb| of order 1 and more,
// carry 2^-53 of themselves: below 2^3, rounded by at most 2^-53
constexpr float kSepTcTop64 = 2.0f;

// A sub-ensemble's lists of trajectories (k_sep_lists, for the digit-product
// kernels): a = contracted A terms, x = B terms and (rA - 1) A terms
// (kSepRest set), g = trajectories left to the outer-product kernel; f: 2^f
// above every contracted first factor.
struct SepMeta {
    int a, x, g, f;
};
constexpr int kSepRest = 1 << 30;

}  // namespace bin2d

// The tensor-core kernels of the joint generating functions (k_gf2d_tc.cu):
// whether they take `count` trajectories of this grid; a piece's bytes of work
// space; one piece (list of the trajectories left over and their counts
// returned for the outer-product kernel).
bool gf2d_tc_takes(bool fp64, int n_sub, int64_t KA, int KB, int64_t count);
int64_t gf2d_tc_piece(int n_sub, int64_t KA, int KB, int64_t count, size_t *bytes);
template <typename V>
int launch_gf2d_tc(gbs_net *net, const bin2d::GridD &g, const bin2d::SepTrajT<V> *sep, int64_t count,
                   uint64_t e0, const DfConsts &K, const int **rest, const bin2d::SepMeta **meta,
                   int *rest_ld);

}  // namespace gbs
