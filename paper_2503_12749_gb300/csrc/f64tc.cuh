// Operand layout and digit arithmetic of the FP64 tensor-core GEMM
// (k_gemm_f64tc.cu), shared with the sampler that writes its trajectory
// operand.
#pragma once

#include <cuda_fp16.h>

#include <cstdint>

namespace gbs {
namespace f64tc {

constexpr int kDigits = 7;        // balanced base-256 digits of a 56-bit fixed-point number
constexpr int kTrajTile = 32;     // trajectories per tile, two sub-tiles of 16
// one K step of 16 input modes: digit q of a 128-row A tile, of a 32-row
// (16 alpha, 16 beta) B sub-tile
constexpr int kASlice = 128 * 32;
constexpr int kAStage = kDigits * kASlice;
constexpr int kBSlice = 32 * 32;
constexpr int kBSub = kDigits * kBSlice;
constexpr int kBStage = 2 * kBSub;
// The trajectory operand of the GEMM has kTrajBits more bits than T, all of them
// in its leading digit (|b_0| <= 2^10, an FP16 number too): its scale is that of
// the largest possible draw, 8.67 standard deviations rounded up to a power of
// two, so that with 55 bits a typical amplitude kept 50 or 51 of its 53.
constexpr int kTrajBits = 3;
// scales beyond 2^+-kExpRange are left to the SIMT kernel
constexpr int kExpRange = 400;
constexpr int kExpNone = -(1 << 20);
constexpr int kExpVacuum = -kExpRange - 1;  // an input mode in the vacuum state

// Byte offset of (row, k) within a slice of one 16-wide K step: 8-row groups
// of 256 bytes, each two core matrices of 8 rows x 16 bytes.
__host__ __device__ __forceinline__ int core_offset(int row, int k) {
    return (row >> 3) * 256 + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2;
}

// v 2^s rounded to an integer, to nearest and halves to even, for |v 2^s| <= 2^58 and
// a normal v; 0 below one half.  (Where a few bits are dropped many values are
// halves: with 55 bits, rounding those away from zero biased n_S by 0.7 2^-53.)
__device__ __forceinline__ int64_t to_fixed(double v, int s) {
    const int64_t bits = __double_as_longlong(v);
    const int ex = (int)((bits >> 52) & 0x7ff) - 1075 + s;  // |v| 2^s = m 2^ex
    const int64_t m = (bits & 0xfffffffffffffll) | 0x10000000000000ll;
    int64_t x;
    if (ex >= 0) {
        x = m << ex;
    } else if (ex < -54) {
        x = 0;
    } else {
        const int64_t t = m >> (-ex - 1);  // floor of twice the value
        const bool up = (t << (-ex - 1)) != m || (t & 2);
        x = (t + (up ? 1 : 0)) >> 1;
    }
    return bits < 0 ? -x : x;
}

// The seven balanced digits of x0 and x1 as pairs of FP16 numbers (x0's in the low
// half), most significant first: bytes of x + 128 (1 + 256 + ...), less 128.  FP16
// rather than BF16 because a byte below 1024 is exact in it, so both digits of a
// pair take one byte permutation, one logic instruction and one packed
// subtraction.  The leading digit has 9 bits (0..256) for |x| <= 2^55; kWide (|x|
// <= 2^(55 + kTrajBits)) converts it, up to +-1024 here, one by one.
template <bool kWide = false>
__device__ __forceinline__ void digit_pairs(int64_t x0, int64_t x1, uint32_t (&d)[kDigits]) {
    const uint64_t y0 = (uint64_t)x0 + 0x80808080808080ull, y1 = (uint64_t)x1 + 0x80808080808080ull;
    const __half2 bias = __float2half2_rn(1152.0f);  // 1024 + 128
    auto less = [&](uint32_t v) {
        const __half2 h = __hsub2(*reinterpret_cast<const __half2 *>(&v), bias);
        return *reinterpret_cast<const uint32_t *>(&h);
    };
    const uint32_t h0 = (uint32_t)(y0 >> 32), h1 = (uint32_t)(y1 >> 32);
    if (kWide) {
        const __half2 h = __halves2half2(__short2half_rn((short)((int)h0 >> 16)),
                                         __short2half_rn((short)((int)h1 >> 16)));
        const __half2 top = __hsub2(h, __float2half2_rn(128.0f));
        d[0] = *reinterpret_cast<const uint32_t *>(&top);
    } else {
        d[0] = less(__byte_perm(h0, h1, 0x7632) + 0x64006400u);
    }
#pragma unroll
    for (int q = 1; q < kDigits; ++q) {
        const int byte = kDigits - 1 - q;
        const uint32_t v = byte >= 4 ? __byte_perm(h0, h1, (byte - 4) | byte << 8)
                                     : __byte_perm((uint32_t)y0, (uint32_t)y1, byte | (byte + 4) << 8);
        d[q] = less((v & 0x00ff00ffu) | 0x64006400u);
    }
}

}  // namespace f64tc

inline int f64tc_kblocks(int N) { return (N + 15) / 16; }

}  // namespace gbs
