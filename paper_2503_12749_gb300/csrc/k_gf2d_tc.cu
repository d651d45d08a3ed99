// The joint generating functions of d = 2..4 output bins as exact integer
// contractions on the tensor cores.
//
// With the factorisation of k_bin2d.cu a sub-ensemble's sums are contractions
// over its trajectories,
//   sum G_+P = sum_e A_1 A_2,   sum G_mP = sum G_+P + sum_e [B_1 B_2 + (rA - 1) A_1 A_2],
// of complex vectors on the first bins' flattened slots and the last bin's.
// The factors are evaluated once per (trajectory, slot) in double-float (BF16
// networks; the outer-product kernel evaluates them once per tile of 32 x 32
// slots) or FP64 (the others; k_gf2d evaluates every grid point), written
// as 56-bit fixed-point numbers of seven balanced 8-bit digits, and the digit
// products are contracted without rounding by the pipeline of the FP64 GEMM
// (f64tc_pipe.cuh): rows are (slot of the first factor, Re / Im), columns the
// second factor's slots, and each trajectory is two steps of the contraction,
//   Re row: (A_1r, -A_1i), Im row: (A_1i, A_1r) against (A_2r, A_2i).
// The second factors are at most 1, the first ones of a sub-ensemble below 2^f
// of their largest: resolutions 2^-56 and 2^(f - 56), against 2^-46 relative of
// the double-float factors (FP64 ones have f <= 3, 2^-53 of exponents and phases, and
// sums that were rounded at every term).  Trajectories whose first factor may exceed e^kSepTcTop
// (e^kSepTcTop64), or whose phase or exponent is beyond the double-float functions,
// are listed for the general kernels (k_gf2d_df, k_gf2d).  The integer sums do not depend on
// their order, so the lists are compacted.
// Root mean square error over the grid of the mean sums of 160 trajectories against
// 113-bit arithmetic from the same n and n_Sb (matrix-P, +P; general kernels -> here):
// FP64, 8 modes 1.2e-16, 4.8e-16 -> 5.0e-17, 3.3e-16; 40 4.6e-17, 3.6e-17 -> 3.7e-17,
// 2.2e-17; 200 lossless (9 networks) 1.6e-16, 2.2e-17 -> 1.5e-16, 1.5e-17; BF16, 8
// modes 1.6e-14, 1.0e-14 -> 2.8e-15, 5.5e-15; 200 lossy 3.0e-16, 3.0e-16 -> 1.5e-16, 1.5e-16.
//
// Why: the double-float outer products are 2 x 16 packed FP32 instructions per
// grid point and trajectory on the FP32 pipe; as digits they are 34 tensor-core
// multiply-adds of 4096 per SM and clock.  Measured (200 lossless modes, K1 = K2 =
// 128, 1.2e6 trajectories): generating functions 63 -> 18 ms, whole call 67.5 ->
// 23.1 ms; of 131072 trajectories the factors' digits 1.00 ms, the contraction
// 0.90 ms (its products at 0.67 of the measured BF16 rate: 400 tiles make 2.6 waves,
// and the drain of the sums is not fully covered, f64tc_pipe.cuh).
// FP64 networks, 100 sub-ensembles, 20000 trajectories: 200 lossless modes on 128 x
// 128 50.1 -> 2.00 ms; 50 and 10000, 60 modes on 32 x 32 x 32 51.3 -> 6.37 ms; 40 and
// 20000, 8 modes (some trajectories too wide) 48.0 -> 6.76 ms.
#include "bin2d.cuh"
#include "f64tc_pipe.cuh"
#include "gf64.cuh"

#include <algorithm>
#include <type_traits>

namespace gbs {
namespace {

using namespace bin2d;
using namespace f64tc;

constexpr int kListThreads = 256;
constexpr int kDigThreads = 256;
constexpr int kQuads = 8;           // groups of four trajectories staged at a time
constexpr int kTrajWords = sizeof(SepTraj) / 16;
static_assert(sizeof(SepTraj) % 16 == 0, "trajectories copied in 16-byte words");
constexpr int kSepOff = 1 << 29;
constexpr int kSlotTile = 64;       // slots of either factor per tile
constexpr int kEntryBlock = 8;      // trajectories per K block of 16
// Work space of the operands: pieces of about 65,000 trajectories at K1 = K2 =
// 128, whose 400 tiles (100 sub-ensembles) fill 152 SMs 2.6 times.
constexpr size_t kWorkBytes = (size_t)2 << 30;
// Trajectories per sub-ensemble and launch from which the contraction is used,
// for grids whose last bin has more than 32 points and for those with 32 (half
// of a tile's columns are padding).  Whole gbs_sample_nd calls, outer products ->
// contraction (us): 100 sub-ensembles on 64 x 64 of 16 trajectories 151 -> 164, 32
// 158 -> 157, 64 271 -> 220; 128 x 128 of 32 324 -> 256, 512 2913 -> 1038; 32 x 32 of
// 32 139 -> 164, 10 of 2000 2463 -> 848; 50 of 1000 on 32 x 32 x 32 9658 -> 5641.  FP64
// networks, whose general kernel is ten times slower: 100 of 8 on 32 x 32 345 -> 200.
constexpr int64_t kMinPerSub = 32, kMinPerSub32 = 128, kMinPerSub64 = 8;

// Offsets of the work space for `q` (a multiple of 8) trajectories per
// sub-ensemble: K blocks r cap + [0, q / 8) hold the A terms, the next 2 q / 8
// the B terms and the (rA - 1) A terms.
struct Work {
    int q, cap;
    size_t img_b, lists, meta, bytes;

    Work(int n_sub, int64_t KA, int KB, int64_t per_sub) {
        q = (int)((per_sub + kEntryBlock - 1) / kEntryBlock * kEntryBlock);
        cap = 3 * (q / kEntryBlock);
        const size_t blocks = (size_t)n_sub * cap;
        const size_t mt = (size_t)((KA + kSlotTile - 1) / kSlotTile);
        const size_t ct = (size_t)((KB + kSlotTile - 1) / kSlotTile);
        img_b = blocks * mt * kAStage;
        lists = img_b + blocks * ct * kBStage;
        meta = lists + sizeof(int) * (size_t)n_sub * 4 * q;
        bytes = meta + sizeof(SepMeta) * (size_t)n_sub;
    }
};

// One block per sub-ensemble: its lists [A: q][X: 2 q][rest: q], in order.
template <typename V>
__global__ void __launch_bounds__(kListThreads)
    k_sep_lists(const SepTrajT<V> *__restrict__ sep, float most, int64_t count, uint64_t e0, int n_sub,
                int q, int *__restrict__ lists, SepMeta *__restrict__ meta, int64_t *__restrict__ counts) {
    __shared__ int s_sum[kListThreads / 32];
    __shared__ unsigned s_top[kListThreads / 32];
    const int r = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t first = (int64_t)(((uint64_t)r + (uint64_t)n_sub - e0 % (uint64_t)n_sub) %
                                    (uint64_t)n_sub);
    const int64_t cnt_r = first < count ? (count - 1 - first) / n_sub + 1 : 0;
    int *la = lists + (size_t)r * 4 * q, *lx = la + q, *lg = lx + 2 * q;
    int a = 0, x = 0, g = 0;  // entries so far
    float top = 0.0f;
    for (int64_t base = 0; base < cnt_r; base += kListThreads) {
        const int64_t t = base + threadIdx.x;
        const int64_t i = first + t * n_sub;
        int flags = 0;
        bool in = false, left = false;
        if (t < cnt_r) {
            flags = sep[i].flags;
            const float b = sep[i].top;
            in = !(flags & kSepPoint) && b <= most;
            left = !in;
            if (in) top = fmaxf(top, b);
        }
        const int nb = in && (flags & kSepB) ? 1 : 0, nq = in && !(flags & kSepOne) ? 1 : 0;
        // the three counts side by side, 10 bits each (at most 512 per pass)
        const int own = (in ? 1 : 0) | (nb + nq) << 10 | (left ? 1 : 0) << 20;
        int inc = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += v;
        }
        if (lane == 31) s_sum[warp] = inc;
        __syncthreads();
        int before = inc - own, all = 0;
#pragma unroll
        for (int w = 0; w < kListThreads / 32; ++w) {
            if (w < warp) before += s_sum[w];
            all += s_sum[w];
        }
        if (in) la[a + (before & 1023)] = (int)i;
        int o = x + (before >> 10 & 1023);
        if (nb) lx[o++] = (int)i;
        if (nq) lx[o] = (int)i | kSepRest;
        if (left) lg[g + (before >> 20)] = (int)i;
        a += all & 1023;
        x += all >> 10 & 1023;
        g += all >> 20;
        __syncthreads();
    }
    const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(top));
    if (lane == 0) s_top[warp] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned b = 0;
        for (int w = 0; w < kListThreads / 32; ++w) b = max(b, s_top[w]);
        const int f = (int)floorf(__uint_as_float(b) * 1.44269504f + 0.01f) + 1;
        meta[r] = SepMeta{a, x, g, f};
        counts[r] += cnt_r;
    }
}

// (hi + lo) 2^32 scale rounded to an integer, |.| <= 2^55: 32-bit conversions,
// the 64-bit one has an eighth of their rate.
__device__ __forceinline__ int64_t df_fixed(float hi, float lo, float scale) {
    const float h = hi * scale;                     // below 2^23
    const int top = __float2int_rn(h);
    const float rest = (h - (float)top) * 0x1p32f;  // exact, |.| <= 2^31
    return ((int64_t)top << 32) + __float2int_rn(rest) + __float2int_rn(lo * scale * 0x1p32f);
}

// v 2^s rounded to an integer, |v 2^s| <= 2^55 (to_fixed takes normal numbers).
__device__ __forceinline__ int64_t to_fixed_any(double v, int s) {
    return fabs(v) < 0x1p-60 ? 0 : to_fixed(v, s);
}

// Digits (re, im) of four trajectories of slot `slot` (0..63) of a tile: rows
// (re, -im) and (im, re), or a column (re, im); `half` of the K block.
__device__ __forceinline__ void store_row(uint8_t *tile, int slot, int half, const uint32_t (&w)[kDigits][4]) {
    uint8_t *o = tile + core_offset(2 * slot, 8 * half);
    constexpr uint32_t neg = 0x80000000u;
#pragma unroll
    for (int p = 0; p < kDigits; ++p) {
        *reinterpret_cast<uint4 *>(o + p * kASlice) =
            make_uint4(w[p][0] ^ neg, w[p][1] ^ neg, w[p][2] ^ neg, w[p][3] ^ neg);
        *reinterpret_cast<uint4 *>(o + p * kASlice + 16) =
            make_uint4(__byte_perm(w[p][0], 0u, 0x1032), __byte_perm(w[p][1], 0u, 0x1032),
                       __byte_perm(w[p][2], 0u, 0x1032), __byte_perm(w[p][3], 0u, 0x1032));
    }
}
__device__ __forceinline__ void store_col(uint8_t *tile, int slot, int half, const uint32_t (&w)[kDigits][4]) {
    uint8_t *o = tile + (slot >> 5) * kBSub + core_offset(slot & 31, 8 * half);
#pragma unroll
    for (int p = 0; p < kDigits; ++p)
        *reinterpret_cast<uint4 *>(o + p * kBSlice) = make_uint4(w[p][0], w[p][1], w[p][2], w[p][3]);
}

// The operands' digits: a thread holds one slot of either factor and takes four
// trajectories of a list at a time (8 steps of the contraction, 16 bytes per
// digit and row).  Bound by the double-float functions' instructions; the stores
// (21 KB per trajectory at K1 = K2 = 128 with a B term) are at a third of DRAM's
// rate.  131072 trajectories there: 1.72 ms with scalar double-float functions and
// 64-bit conversions, 1.35 with two trajectories on packed instructions, 1.00 with
// the trajectories' constants staged in shared memory and three blocks per SM.
template <int D>
__global__ void __launch_bounds__(kDigThreads, 3)
    k_sep_digits(const SepTraj *__restrict__ sep, const SepMeta *__restrict__ meta,
                 const int *__restrict__ lists, int q, const int *__restrict__ wmax, const GridD g,
                 const double2 *__restrict__ tw, const DfConsts K, uint8_t *__restrict__ imgA,
                 uint8_t *__restrict__ imgB) {
    __shared__ DfTables s_tab;
    __shared__ SepTraj s_tr[4 * kQuads];
    __shared__ int s_en[4 * kQuads];  // list entries, kSepOff beyond the list's end
    const int tid = threadIdx.x, r = blockIdx.y;
    if (tid < 64) s_tab.exp2[tid] = df{K.exp2_hi[tid], K.exp2_lo[tid]};
    if (tid < 33) {
        s_tab.sn[tid] = df{K.sin_hi[tid], K.sin_lo[tid]};
        s_tab.cs[tid] = df{K.cos_hi[tid], K.cos_lo[tid]};
    }
    __syncthreads();
    constexpr int d = D;
    const Slots sl = slots_of_grid(g, wmax);
    int Sa = 1;
    for (int b = 0; b < d - 1; ++b) Sa *= sl.S[b];
    const int Sb = sl.S[d - 1];
    const int mt = (Sa + kSlotTile - 1) / kSlotTile, ct = (Sb + kSlotTile - 1) / kSlotTile;
    const int Ra = (Sa + 31) / 32 * 32;  // a warp holds slots of one factor
    const SepMeta mr = meta[r];
    const int qa = 2 * ((mr.a + kEntryBlock - 1) / kEntryBlock);
    const int qx = 2 * ((mr.x + kEntryBlock - 1) / kEntryBlock);
    const int *la = lists + (size_t)r * 4 * q;
    const size_t kb_a = (size_t)r * 3 * (q / kEntryBlock), kb_x = kb_a + q / kEntryBlock;
    for (int pass = 0; pass < Ra + Sb; pass += kDigThreads) {
        const int s = pass + tid;
        const bool row = s < Ra, live = row ? s < Sa : s < Ra + Sb;
        const int slot = !live ? 0 : row ? s : s - Ra;
        df cm[d - 1], sn[d - 1];  // a row's bins, or a column's one
        {
            int k[kMaxBins] = {0, 0, 0, 0};
            if (row) slot_ks(g, sl, d - 1, slot, k);
            else k[0] = slot_k(slot, g.K[d - 1], sl.W1[d - 1], sl.W2[d - 1]);
#pragma unroll
            for (int b = 0; b < d - 1; ++b) {
                const double2 t = tw[row ? g.Koff[b] + k[b] : g.Koff[d - 1] + k[0]];
                cm[b] = df_from_double(t.x);
                sn[b] = df_from_double(t.y);
            }
        }
        // first factors below 2^f, second factors at most 1; df_fixed multiplies
        // by 2^32
        const float scale = __uint_as_float((uint32_t)(127 - 32 + 55 - (row ? mr.f : 0)) << 23);
        for (int u0 = blockIdx.x * kQuads; u0 < qa + qx; u0 += gridDim.x * kQuads) {
            __syncthreads();
            for (int j = tid; j < 4 * kQuads * kTrajWords; j += kDigThreads) {
                const int e = j / kTrajWords, part = j % kTrajWords, u = u0 + (e >> 2);
                if (u >= qa + qx) continue;
                const bool isx = u >= qa;
                const int n = isx ? mr.x : mr.a, i = 4 * (isx ? u - qa : u) + (e & 3);
                const int entry = (isx ? la + q : la)[min(i, n - 1)];
                reinterpret_cast<uint4 *>(&s_tr[e])[part] =
                    reinterpret_cast<const uint4 *>(&sep[entry & (kSepOff - 1)])[part];
                if (part == 0) s_en[e] = i < n ? entry : entry | kSepOff;
            }
            __syncthreads();
            for (int u = u0; live && u < min(u0 + kQuads, qa + qx); ++u) {
                const bool isx = u >= qa;
                const int quad = isx ? u - qa : u;
                const int e0 = 4 * (u - u0);
                uint32_t w[kDigits][4];  // (re, im) of each trajectory
                // two trajectories side by side on the packed FP32x2 instructions
#pragma unroll
                for (int t = 0; t < 4; t += 2) {
                    const int en[2] = {s_en[e0 + t], s_en[e0 + t + 1]};
                    const SepTraj &s0 = s_tr[e0 + t], &s1 = s_tr[e0 + t + 1];
                    const bool r0 = (en[0] & kSepRest) != 0, r1 = (en[1] & kSepRest) != 0;
                    const bool b0 = isx && !r0, b1 = isx && !r1;
                    df2 l, ph;
                    if (row) {
#pragma unroll
                        for (int b = 0; b < d - 1; ++b) {
                            const df2 c2 = df2_make(cm[b], cm[b]), n2 = df2_make(sn[b], sn[b]);
                            const df2 x = df2_make(s0.x[b], s1.x[b]), y = df2_make(s0.y[b], s1.y[b]);
                            const df2 lb = df2_add(df2_mul(c2, x), df2_neg(df2_mul(n2, y)));
                            const df2 pb = df2_add(df2_mul(n2, x), df2_mul(c2, y));
                            l = b == 0 ? lb : df2_add(l, lb);
                            ph = b == 0 ? pb : df2_add(ph, pb);
                        }
                    } else {
                        const df2 c2 = df2_make(cm[0], cm[0]), n2 = df2_make(sn[0], sn[0]);
                        const df2 x = df2_make(s0.x[d - 1], s1.x[d - 1]), y = df2_make(s0.y[d - 1], s1.y[d - 1]);
                        l = df2_add(df2_mul(c2, x), df2_neg(df2_mul(n2, y)));
                        ph = df2_add(df2_mul(n2, x), df2_mul(c2, y));
                    }
                    // l + M_B, -l + M'_B + c2 + log inv; l - M_B, -l - M'_B; the phase
                    // has the exponent's sign
                    const float2 sg = f2(b0 ? -1.0f : 1.0f, b1 ? -1.0f : 1.0f);
                    const df o0 = row ? (b0 ? s0.o1b : s0.o1a) : df_neg(b0 ? s0.mp2 : s0.m2);
                    const df o1 = row ? (b1 ? s1.o1b : s1.o1a) : df_neg(b1 ? s1.mp2 : s1.m2);
                    df2 ex = df2_add(df2{f2_mul(l.hi, sg), f2_mul(l.lo, sg)}, df2_make(o0, o1));
                    // below FP32's normal range (or no trajectory): zero
                    const float2 on = f2(ex.hi.x >= -87.0f && !(en[0] & kSepOff) ? 1.0f : 0.0f,
                                         ex.hi.y >= -87.0f && !(en[1] & kSepOff) ? 1.0f : 0.0f);
                    ex.hi = f2(fmaxf(ex.hi.x, -87.0f), fmaxf(ex.hi.y, -87.0f));
                    df2 sp, cp;
                    df2_sincos_tab(ph, s_tab, K, sp, cp);
                    df2 e = df2_exp_tab(ex, s_tab, K);
                    e = {f2_mul(e.hi, on), f2_mul(e.lo, on)};
                    const df one = {1.0f, 0.0f};
                    if (row && (r0 || r1))
                        e = df2_mul(e, df2_make(r0 ? df_add_f(s0.rA, -1.0f) : one,
                                                r1 ? df_add_f(s1.rA, -1.0f) : one));
                    const df2 re = df2_mul(e, cp);
                    df2 im = df2_mul(e, sp);
                    im = {f2_mul(im.hi, sg), f2_mul(im.lo, sg)};
                    uint32_t dg[kDigits];
                    digit_pairs(df_fixed(re.hi.x, re.lo.x, scale), df_fixed(im.hi.x, im.lo.x, scale), dg);
#pragma unroll
                    for (int p = 0; p < kDigits; ++p) w[p][t] = dg[p];
                    digit_pairs(df_fixed(re.hi.y, re.lo.y, scale), df_fixed(im.hi.y, im.lo.y, scale), dg);
#pragma unroll
                    for (int p = 0; p < kDigits; ++p) w[p][t + 1] = dg[p];
                }
                const size_t kb = (isx ? kb_x : kb_a) + (quad >> 1);
                if (row) store_row(imgA + (kb * mt + (slot >> 6)) * kAStage, slot & 63, quad & 1, w);
                else store_col(imgB + (kb * ct + (slot >> 6)) * kBStage, slot & 63, quad & 1, w);
            }
        }
    }
}

// The same from FP64 factors (FP64 and FP32 networks): bound by the FP64 pipe's
// exponentials, sines and cosines.
template <int D>
__global__ void __launch_bounds__(kDigThreads)
    k_sep_digits64(const SepTraj64 *__restrict__ sep, const SepMeta *__restrict__ meta,
                   const int *__restrict__ lists, int q, const int *__restrict__ wmax, const GridD g,
                   const double2 *__restrict__ tw, const Gf64Tables tabs,
                   uint8_t *__restrict__ imgA, uint8_t *__restrict__ imgB) {
    __shared__ Gf64Tables s_tab;
    constexpr int d = D;
    const int tid = threadIdx.x, r = blockIdx.y;
    if (tid < 64) s_tab.exp2[tid] = tabs.exp2[tid];
    for (int t = tid; t < 256; t += kDigThreads) {
        s_tab.sn[t] = tabs.sn[t];
        s_tab.cs[t] = tabs.cs[t];
    }
    __syncthreads();
    const Slots sl = slots_of_grid(g, wmax);
    int Sa = 1;
    for (int b = 0; b < d - 1; ++b) Sa *= sl.S[b];
    const int Sb = sl.S[d - 1];
    const int mt = (Sa + kSlotTile - 1) / kSlotTile, ct = (Sb + kSlotTile - 1) / kSlotTile;
    const int Ra = (Sa + 31) / 32 * 32;
    const SepMeta mr = meta[r];
    const int qa = 2 * ((mr.a + kEntryBlock - 1) / kEntryBlock);
    const int qx = 2 * ((mr.x + kEntryBlock - 1) / kEntryBlock);
    const int *la = lists + (size_t)r * 4 * q;
    const size_t kb_a = (size_t)r * 3 * (q / kEntryBlock), kb_x = kb_a + q / kEntryBlock;
    for (int s = tid; s < Ra + Sb; s += kDigThreads) {
        const bool row = s < Ra;
        const int slot = row ? s : s - Ra;
        if (row && slot >= Sa) continue;
        double cm[d - 1], sn[d - 1];
        {
            int k[kMaxBins] = {0, 0, 0, 0};
            if (row) slot_ks(g, sl, d - 1, slot, k);
            else k[0] = slot_k(slot, g.K[d - 1], sl.W1[d - 1], sl.W2[d - 1]);
#pragma unroll
            for (int b = 0; b < d - 1; ++b) {
                const double2 t = tw[row ? g.Koff[b] + k[b] : g.Koff[d - 1] + k[0]];
                cm[b] = t.x;
                sn[b] = t.y;
            }
        }
        const int shift = 55 - (row ? mr.f : 0);
        for (int u = blockIdx.x; u < qa + qx; u += gridDim.x) {
            const bool isx = u >= qa;
            const int quad = isx ? u - qa : u;
            const int *list = (isx ? la + q : la) + 4 * quad;
            const int left = (isx ? mr.x : mr.a) - 4 * quad;
            uint32_t w[kDigits][4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                int64_t xr = 0, xi = 0;
                if (t < left) {
                    const int entry = list[t];
                    const SepTraj64 &st = sep[entry & (kSepRest - 1)];
                    const bool rest = (entry & kSepRest) != 0, isb = isx && !rest;
                    double l = 0.0, ph = 0.0;
                    if (row) {
#pragma unroll
                        for (int b = 0; b < d - 1; ++b) {
                            l += cm[b] * st.x[b] - sn[b] * st.y[b];
                            ph += sn[b] * st.x[b] + cm[b] * st.y[b];
                        }
                    } else {
                        l = cm[0] * st.x[d - 1] - sn[0] * st.y[d - 1];
                        ph = sn[0] * st.x[d - 1] + cm[0] * st.y[d - 1];
                    }
                    const double ofs = row ? (isb ? st.o1b : st.o1a) : -(isb ? st.mp2 : st.m2);
                    double si, co, e = exp_tab64((isb ? -l : l) + ofs, s_tab);
                    sincos_tab64(ph, s_tab, si, co);
                    if (row && rest) e *= st.rA - 1.0;
                    xr = to_fixed_any(e * co, shift);
                    xi = to_fixed_any(e * (isb ? -si : si), shift);
                }
                uint32_t dg[kDigits];
                digit_pairs(xr, xi, dg);
#pragma unroll
                for (int p = 0; p < kDigits; ++p) w[p][t] = dg[p];
            }
            const size_t kb = (isx ? kb_x : kb_a) + (quad >> 1);
            if (row) store_row(imgA + (kb * mt + (slot >> 6)) * kAStage, slot & 63, quad & 1, w);
            else store_col(imgB + (kb * ct + (slot >> 6)) * kBStage, slot & 63, quad & 1, w);
        }
    }
}

// Tiles of 64 x 64 slots of one sub-ensemble, persistent CTAs.  A tile is two
// contractions into the same 64-bit sums: the A terms (the +P sum, added to
// acc), then the others (the matrix-P sum).
__global__ void __launch_bounds__(kThreads, 1)
    k_gf2d_tc(const uint8_t *__restrict__ imgA, const uint8_t *__restrict__ imgB,
              const SepMeta *__restrict__ meta, int q, const int *__restrict__ wmax, const GridD g,
              int n_sub, double *__restrict__ acc, uint64_t wait_ns, unsigned long long *err_ptr) {
    extern __shared__ uint8_t smem_raw[];
    Pipe pipe(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile unsigned long long *err = err_ptr;
    int Sa = 1, Sb;
    {
        const Slots sl = slots_of_grid(g, wmax);
        for (int b = 0; b < g.d - 1; ++b) Sa *= sl.S[b];
        Sb = sl.S[g.d - 1];
    }
    const int KB = g.K[g.d - 1];
    const int mt = (Sa + kSlotTile - 1) / kSlotTile, ct = (Sb + kSlotTile - 1) / kSlotTile;
    const int ntiles = n_sub * mt * ct;
    const uint32_t tmem = pipe.open();
    auto job = [&](int i, Contraction &c) {
        const int64_t t = blockIdx.x + (int64_t)(i >> 1) * gridDim.x;
        if (t >= ntiles) return false;
        const int r = (int)t / (mt * ct), rem = (int)t % (mt * ct);
        const size_t kb = (size_t)r * 3 * (q / kEntryBlock) + ((i & 1) ? q / kEntryBlock : 0);
        c.sa = (size_t)mt * kAStage;
        c.sb = (size_t)ct * kBStage;
        c.a = imgA + kb * c.sa + (size_t)(rem / ct) * kAStage;
        c.b = imgB + kb * c.sb + (size_t)(rem % ct) * kBStage;
        c.KB = (((i & 1) ? meta[r].x : meta[r].a) + kEntryBlock - 1) / kEntryBlock;
        return true;
    };
    if (warp == 0) {
        if (lane == 0) pipe.load(job, err, wait_ns);
    } else if (warp == 1) {
        if (lane == 0) pipe.multiply(job, tmem, err, wait_ns);
    } else {
        const int quarter = warp & 3, sub = (warp - 2) >> 2;
        const int row = quarter * 32 + lane;
        const uint32_t tb = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)sub * 256u;
        uint32_t ck = 0;
        for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
            const int r = t / (mt * ct);
            int64_t hi[32], lo[32];
#pragma unroll
            for (int c = 0; c < 32; ++c) hi[c] = lo[c] = 0;
            for (int part = 0; part < 2; ++part) {
                const int blocks = ((part ? meta[r].x : meta[r].a) + kEntryBlock - 1) / kEntryBlock;
                for (int n = (blocks + kChunkKB - 1) / kChunkKB; n > 0; --n, ++ck)
                    pipe.add_chunk(ck, sub, tb, hi, lo, err, wait_ns);
                // everything else is formed here: the sums leave it no registers
                const int rem = t - r * mt * ct;
                const int slot = rem / ct * kSlotTile + (row >> 1);
                const int slot0 = rem % ct * kSlotTile + sub * 32;
                if (slot >= Sa) continue;
                const Slots sl = slots_of_grid(g, wmax);
                const int W1 = sl.W1[g.d - 1], W2 = sl.W2[g.d - 1];
                int64_t grid = 1;
                for (int b = 0; b < g.d; ++b) grid *= g.K[b];
                int k[kMaxBins] = {0, 0, 0, 0};
                const int64_t oA = slot_ks(g, sl, g.d - 1, slot, k);
                const int f = meta[r].f - 70;
                double *o = acc + 2 * ((size_t)(part ? r : n_sub + r) * grid + (size_t)oA * KB) + (row & 1);
                // (one addition per element and launch: the sums stay reproducible;
                // reductions at L2, since a load, an addition and a store each wait
                // for the one before)
#pragma unroll
                for (int c = 0; c < 32; ++c)
                    if (slot0 + c < Sb)
                        atomicAdd(o + 2 * slot_k(slot0 + c, KB, W1, W2), fixed_to_double(hi[c], lo[c], f));
            }
        }
    }
    pipe.close(tmem);
}

}  // namespace

// (rows, 128 a tile, are 64 slots of the first factor)
bool gf2d_tc_takes(bool fp64, int n_sub, int64_t KA, int KB, int64_t count) {
    if (KA < 32 || KB < 32 || KA > (1 << 20)) return false;
    if (count / n_sub < (fp64 ? kMinPerSub64 : KB > 32 ? kMinPerSub : kMinPerSub32)) return false;
    return Work(n_sub, KA, KB, kMinPerSub).bytes <= kWorkBytes;
}

int64_t gf2d_tc_piece(int n_sub, int64_t KA, int KB, int64_t count, size_t *bytes) {
    const size_t per = Work(n_sub, KA, KB, kEntryBlock).bytes;  // of 8 per sub-ensemble
    const int64_t most = (int64_t)(kWorkBytes / per) * kEntryBlock * n_sub;
    const int64_t pieces = (count + most - 1) / most;
    const int64_t step = (int64_t)kEntryBlock * n_sub;
    const int64_t piece = ((count + pieces - 1) / pieces + step - 1) / step * step;
    if (bytes) *bytes = Work(n_sub, KA, KB, piece / n_sub).bytes;
    return piece;
}

template <typename V>
int launch_gf2d_tc(gbs_net *net, const GridD &g, const SepTrajT<V> *sep, int64_t count, uint64_t e0,
                   const DfConsts &K, const int **rest, const SepMeta **meta, int *rest_ld) {
    const int n_sub = net->n_sub2, KB = g.K[g.d - 1];
    const int64_t KA = net->grid2 / KB;
    const Work w(n_sub, KA, KB, (count + n_sub - 1) / n_sub);
    if (w.bytes > net->gf2_bytes) return set_error(GBS_EINVAL, "joint generating functions: work space");
    uint8_t *base = static_cast<uint8_t *>(net->d_gf2);
    int *lists = reinterpret_cast<int *>(base + w.lists);
    SepMeta *m = reinterpret_cast<SepMeta *>(base + w.meta);
    constexpr bool fp64 = std::is_same<V, double>::value;
    k_sep_lists<<<n_sub, kListThreads, 0, net->stream>>>(sep, fp64 ? kSepTcTop64 : kSepTcTop, count, e0,
                                                         n_sub, w.q, lists, m, net->d_counts2);
    GBS_LAUNCH_CHECK();
    // about five blocks per block slot of the chip
    const int groups = (2 * w.cap + kQuads - 1) / kQuads;
    const int per = std::max(1, std::min(groups, 16 * net->sm_count / n_sub));
    const dim3 grid((unsigned)per, (unsigned)n_sub);
    if constexpr (fp64) {
        static const Gf64Tables T = make_gf64_tables();
        auto digits = g.d == 2 ? k_sep_digits64<2> : g.d == 3 ? k_sep_digits64<3> : k_sep_digits64<4>;
        digits<<<grid, kDigThreads, 0, net->stream>>>(sep, m, lists, w.q, net->d_wmax2, g, net->d_tw2,
                                                      T, base, base + w.img_b);
    } else {
        auto digits = g.d == 2 ? k_sep_digits<2> : g.d == 3 ? k_sep_digits<3> : k_sep_digits<4>;
        digits<<<grid, kDigThreads, 0, net->stream>>>(sep, m, lists, w.q, net->d_wmax2, g, net->d_tw2, K,
                                                      base, base + w.img_b);
    }
    GBS_LAUNCH_CHECK();
    GBS_CUDA_TRY(cudaFuncSetAttribute(k_gf2d_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kPipeBytes));
    const int64_t tiles = (int64_t)n_sub * ((KA + kSlotTile - 1) / kSlotTile) *
                          ((KB + kSlotTile - 1) / kSlotTile);
    k_gf2d_tc<<<(unsigned)std::min<int64_t>(tiles, net->sm_count), kThreads, kPipeBytes, net->stream>>>(
        base, base + w.img_b, m, w.q, net->d_wmax2, g, n_sub, reinterpret_cast<double *>(net->d_acc2),
        net->wait_ns, net->d_flags + 1);
    GBS_LAUNCH_CHECK();
    *rest = lists + 3 * (size_t)w.q;
    *meta = m;
    *rest_ld = 4 * w.q;
    return GBS_OK;
}

template int launch_gf2d_tc(gbs_net *, const GridD &, const SepTrajT<df> *, int64_t, uint64_t,
                            const DfConsts &, const int **, const SepMeta **, int *);
template int launch_gf2d_tc(gbs_net *, const GridD &, const SepTrajT<double> *, int64_t, uint64_t,
                            const DfConsts &, const int **, const SepMeta **, int *);

}  // namespace gbs
