// The joint generating functions of d = 2..4 output bins as exact integer
// contractions on the tensor cores (BF16 networks).
//
// With the factorisation of k_bin2d.cu a sub-ensemble's sums are contractions
// over its trajectories,
//   sum G_+P = sum_e A_1 A_2,   sum G_mP = sum G_+P + sum_e [B_1 B_2 + (rA - 1) A_1 A_2],
// of complex vectors on the first bins' flattened slots and the last bin's.
// The factors are evaluated once per (trajectory, slot) in double-float (the
// outer-product kernel evaluates them once per tile of 32 x 32 slots), written
// as 56-bit fixed-point numbers of seven balanced 8-bit digits, and the digit
// products are contracted without rounding by the pipeline of the FP64 GEMM
// (f64tc_pipe.cuh): rows are (slot of the first factor, Re / Im), columns the
// second factor's slots, and each trajectory is two steps of the contraction,
//   Re row: (A_1r, -A_1i), Im row: (A_1i, A_1r) against (A_2r, A_2i).
// The second factors are at most 1, the first ones of a sub-ensemble below 2^f
// of their largest: resolutions 2^-56 and 2^(f - 56), against 2^-46 relative of
// the double-float factors.  Trajectories whose first factor may exceed
// e^kSepTcTop, or whose phase or exponent is beyond the double-float functions,
// are listed for the outer-product kernel.  The integer sums do not depend on
// their order, so the lists are compacted.
//
// Why: the double-float outer products are 2 x 16 packed FP32 instructions per
// grid point and trajectory on the FP32 pipe; as digits they are 34 tensor-core
// multiply-adds of 4096 per SM and clock.
#include "bin2d.cuh"
#include "f64tc_pipe.cuh"

#include <algorithm>

namespace gbs {
namespace {

using namespace bin2d;
using namespace f64tc;

constexpr int kListThreads = 256;
constexpr int kDigThreads = 256;
constexpr int kSlotTile = 64;       // slots of either factor per tile
constexpr int kEntryBlock = 8;      // trajectories per K block of 16
// Work space of the operands: pieces of about 65,000 trajectories at K1 = K2 =
// 128, whose 400 tiles (100 sub-ensembles) fill 152 SMs 2.6 times.
constexpr size_t kWorkBytes = (size_t)2 << 30;
// Trajectories per sub-ensemble and launch from which the contraction is used.
constexpr int64_t kMinPerSub = 64;

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
__global__ void __launch_bounds__(kListThreads)
    k_sep_lists(const SepTraj *__restrict__ sep, int64_t count, uint64_t e0, int n_sub, int q,
                int *__restrict__ lists, SepMeta *__restrict__ meta, int64_t *__restrict__ counts) {
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
            in = !(flags & kSepPoint) && b <= kSepTcTop;
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

// v scale rounded to an integer; |v scale| <= 2^55.
__device__ __forceinline__ int64_t df_fixed(df v, float scale) {
    return __float2ll_rn(v.hi * scale) + __float2ll_rn(v.lo * scale);
}

// The operands' digits: a thread holds one slot of either factor and takes four
// trajectories of a list at a time (8 steps of the contraction, 16 bytes per
// digit and row).  Bound by the double-float functions' instructions and the
// stores (21 KB per trajectory at K1 = K2 = 128 with a B term).
template <int D>
__global__ void __launch_bounds__(kDigThreads, 2)
    k_sep_digits(const SepTraj *__restrict__ sep, const SepMeta *__restrict__ meta,
                 const int *__restrict__ lists, int q, const int *__restrict__ wmax, const GridD g,
                 const double2 *__restrict__ tw, const DfConsts K, uint8_t *__restrict__ imgA,
                 uint8_t *__restrict__ imgB) {
    __shared__ DfTables s_tab;
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
    for (int s = tid; s < Ra + Sb; s += kDigThreads) {
        const bool row = s < Ra;
        const int slot = row ? s : s - Ra;
        if (row && slot >= Sa) continue;
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
        // first factors below 2^f, second factors at most 1 (2^54: room for
        // their rounding)
        const float scale = __uint_as_float((uint32_t)(127 + (row ? 55 - mr.f : 54)) << 23);
        const uint32_t off = row ? (uint32_t)core_offset(2 * (slot & 63), 0)
                                 : (uint32_t)(((slot >> 5) & 1) * kBSub + core_offset(slot & 31, 0));
        for (int u = blockIdx.x; u < qa + qx; u += gridDim.x) {
            const bool isx = u >= qa;
            const int quad = isx ? u - qa : u;
            const int *list = (isx ? la + q : la) + 4 * quad;
            const int left = (isx ? mr.x : mr.a) - 4 * quad;  // entries from here on
            uint32_t w[kDigits][4], v[kDigits][4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
#pragma unroll
                for (int p = 0; p < kDigits; ++p) w[p][t] = v[p][t] = 0u;
                if (t < left) {
                    const int entry = list[t];
                    const SepTraj &st = sep[entry & (kSepRest - 1)];
                    const bool rest = (entry & kSepRest) != 0, isb = isx && !rest;
                    df l, ph;
                    if (row) {
#pragma unroll
                        for (int b = 0; b < d - 1; ++b) {
                            const df lb = df_sub(df_mul(cm[b], st.x[b]), df_mul(sn[b], st.y[b]));
                            const df pb = df_add(df_mul(sn[b], st.x[b]), df_mul(cm[b], st.y[b]));
                            l = b == 0 ? lb : df_add(l, lb);
                            ph = b == 0 ? pb : df_add(ph, pb);
                        }
                    } else {
                        l = df_sub(df_mul(cm[0], st.x[d - 1]), df_mul(sn[0], st.y[d - 1]));
                        ph = df_add(df_mul(sn[0], st.x[d - 1]), df_mul(cm[0], st.y[d - 1]));
                    }
                    // l + M_B, -l + M'_B + c2 + log inv; l - M_B, -l - M'_B
                    const df ofs = row ? (isb ? st.o1b : st.o1a) : df_neg(isb ? st.mp2 : st.m2);
                    const df ex = df_add(isb ? df_neg(l) : l, ofs);
                    if (ex.hi >= -87.0f) {
                        df sp, cp;
                        df_sincos_tab(ph, s_tab, K, sp, cp);
                        df e = df_exp_tab(ex, s_tab, K);
                        if (row && rest) e = df_mul(e, df_add_f(st.rA, -1.0f));
                        const df re = df_mul(e, cp);
                        df im = df_mul(e, sp);
                        if (isb) im = df_neg(im);
                        uint16_t xr[kDigits], xi[kDigits];
                        digits_bf16(df_fixed(re, scale), xr);
                        digits_bf16(df_fixed(im, scale), xi);
#pragma unroll
                        for (int p = 0; p < kDigits; ++p) {
                            const uint32_t a = xr[p], b = xi[p];
                            // Re row (re, -im), Im row (im, re); column (re, im)
                            w[p][t] = a | (row ? b ^ 0x8000u : b) << 16;
                            v[p][t] = b | a << 16;
                        }
                    }
                }
            }
            const size_t kb = (isx ? kb_x : kb_a) + (quad >> 1);
            const uint32_t half = (quad & 1) * 128;
            if (row) {
                uint8_t *o = imgA + (kb * mt + (slot >> 6)) * kAStage + off + half;
#pragma unroll
                for (int p = 0; p < kDigits; ++p) {
                    *reinterpret_cast<uint4 *>(o + p * kASlice) =
                        make_uint4(w[p][0], w[p][1], w[p][2], w[p][3]);
                    *reinterpret_cast<uint4 *>(o + p * kASlice + 16) =
                        make_uint4(v[p][0], v[p][1], v[p][2], v[p][3]);
                }
            } else {
                uint8_t *o = imgB + (kb * ct + (slot >> 6)) * kBStage + off + half;
#pragma unroll
                for (int p = 0; p < kDigits; ++p)
                    *reinterpret_cast<uint4 *>(o + p * kBSlice) =
                        make_uint4(w[p][0], w[p][1], w[p][2], w[p][3]);
            }
        }
    }
}

// Tiles of 64 x 64 slots of one sub-ensemble, persistent CTAs.  A tile is two
// contractions into the same 64-bit sums: the A terms (the +P sum, added to
// acc), then the others (the matrix-P sum).
__global__ void __launch_bounds__(kThreads, 1)
    k_gf2d_tc(const uint8_t *__restrict__ imgA, const uint8_t *__restrict__ imgB,
              const SepMeta *__restrict__ meta, int q, const int *__restrict__ wmax, const GridD g,
              int n_sub, double *__restrict__ acc, unsigned long long *err_ptr) {
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
        if (lane == 0) pipe.load(job, err, kWaitNs);
    } else if (warp == 1) {
        if (lane == 0) pipe.multiply(job, tmem, err, kWaitNs);
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
                    pipe.add_chunk(ck, sub, tb, hi, lo, err, kWaitNs);
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
                const int f = meta[r].f + 1 - 70;
                double *o = acc + 2 * ((size_t)(part ? r : n_sub + r) * grid + (size_t)oA * KB) + (row & 1);
#pragma unroll
                for (int c = 0; c < 32; ++c)
                    if (slot0 + c < Sb)
                        o[2 * slot_k(slot0 + c, KB, W1, W2)] += fixed_to_double(hi[c], lo[c], f);
            }
        }
    }
    pipe.close(tmem);
}

}  // namespace

// Columns are padded to 64 slots, so grids whose last bin has 32 points or
// fewer would spend half of the products on padding.
bool gf2d_tc_takes(int n_sub, int64_t KA, int KB, int64_t count) {
    if (KA <= 32 || KB <= 32 || KA > (1 << 20)) return false;
    if (count / n_sub < kMinPerSub) return false;
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

int launch_gf2d_tc(gbs_net *net, const GridD &g, const SepTraj *sep, int64_t count, uint64_t e0,
                   const DfConsts &K, const int **rest, const SepMeta **meta, int *rest_ld) {
    const int n_sub = net->n_sub2, KB = g.K[g.d - 1];
    const int64_t KA = net->grid2 / KB;
    const Work w(n_sub, KA, KB, (count + n_sub - 1) / n_sub);
    if (w.bytes > net->gf2_bytes) return set_error(GBS_EINVAL, "joint generating functions: work space");
    uint8_t *base = static_cast<uint8_t *>(net->d_gf2);
    int *lists = reinterpret_cast<int *>(base + w.lists);
    SepMeta *m = reinterpret_cast<SepMeta *>(base + w.meta);
    k_sep_lists<<<n_sub, kListThreads, 0, net->stream>>>(sep, count, e0, n_sub, w.q, lists, m,
                                                         net->d_counts2);
    GBS_LAUNCH_CHECK();
    // about four blocks per block slot of the chip, each on many trajectories
    const int per = std::max(1, std::min(w.cap, 8 * net->sm_count / n_sub));
    auto digits = g.d == 2 ? k_sep_digits<2> : g.d == 3 ? k_sep_digits<3> : k_sep_digits<4>;
    digits<<<dim3((unsigned)per, (unsigned)n_sub), kDigThreads, 0, net->stream>>>(
        sep, m, lists, w.q, net->d_wmax2, g, net->d_tw2, K, base, base + w.img_b);
    GBS_LAUNCH_CHECK();
    GBS_CUDA_TRY(cudaFuncSetAttribute(k_gf2d_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kPipeBytes));
    const int64_t tiles = (int64_t)n_sub * ((KA + kSlotTile - 1) / kSlotTile) *
                          ((KB + kSlotTile - 1) / kSlotTile);
    k_gf2d_tc<<<(unsigned)std::min<int64_t>(tiles, net->sm_count), kThreads, kPipeBytes, net->stream>>>(
        base, base + w.img_b, m, w.q, net->d_wmax2, g, n_sub, reinterpret_cast<double *>(net->d_acc2),
        net->d_flags + 1);
    GBS_LAUNCH_CHECK();
    *rest = lists + 3 * (size_t)w.q;
    *meta = m;
    *rest_ld = 4 * w.q;
    return GBS_OK;
}

}  // namespace gbs
