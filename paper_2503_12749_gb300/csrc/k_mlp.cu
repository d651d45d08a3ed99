// The surrogate's multilayer perceptron on the tcgen05 tensor cores:
// forward (GEMM + bias + silu), backward (data and weight GEMMs with the
// silu derivative fused), loss, bias gradients and Adam (Kingma & Ba 2015,
// Algorithm 1).  Not part of the paper: it learns the distribution the
// matrix-P ensemble computes.
//
// Every product is C = A B^T with both operands K-major BF16 in global
// memory, loaded by TMA in 64-wide K boxes (128-byte swizzle) into a 4-stage
// shared-memory ring, multiplied by one thread with tcgen05.mma M=128 N=64
// K=16 into a 64-column TMEM accumulator, and read back by eight epilogue
// warps with tcgen05.ld.  Weights enter as one BF16 plane (their rounding
// of the FP32 master copy); activations and gradients as two planes hi + lo
// (hi = bf16(x), lo = bf16(x - hi)), so each product of an activation plane
// pair with the weights gives ~16 significant bits:
//   forward          Y_l    = H_{l-1} W_l^T            A = H (2 planes), B = W (1)
//   backward, data   dH_{l-1} = dY_l W_l               A = dY (2), B = W^T (1)
//   backward, weight dW_l   = dY_l^T H_{l-1}           A = dY^T (2), B = H^T (2)
// The forward and backward epilogues write their results both row-major
// (the next layer's A operand) and transposed (the weight GEMM's operands),
// and the Adam kernel writes W and W^T, so that no operand needs a transpose
// inside a GEMM.  The weight GEMMs of all layers are one launch and split their
// K (the batch); the Adam kernel sums the split partials in a fixed order, so a
// training step is deterministic.
//
// The layers are small (1800 x 512 x 512: 2.8 GFLOP with two planes, 1.5 us of
// the tensor pipe), so a launch is bound by the latency of its loads and its
// epilogue, and a training step by the number of launches: tiles of 64 columns
// put 120 CTAs on the chip where 256 put 30, with an epilogue a quarter as long;
// the epilogue turns its rows through shared memory so that every store
// instruction writes whole lines (a row per lane touched 32 lines); loss, loss
// gradient and the column sums for the bias gradients are epilogues of the
// GEMMs that produce their inputs; and each launch starts its prologue under its
// predecessor (programmatic dependent launch).  One Adam step at 1800 rows,
// 10-512-512-512-512: 105 us in 9 launches, 557 before (15 launches of 256-column
// tiles, a graph a step); a layer is then 1.2 us from its predecessor's end, 1.1
// to its first data, 3.3 for its 8 stages and 5 for the epilogue.
#include "gbs_internal.cuh"
#include "gbs_surrogate.h"
#include "tc_ptx.cuh"

#include <algorithm>
#include <cmath>
#include <new>
#include <vector>

namespace gbs {
namespace {

constexpr int kBM = 128;   // rows of A per tile (TMEM lanes)
constexpr int kBN = 64;    // rows of B per tile (TMEM columns): layers, one job a launch
constexpr int kBNGrad = 128;  // weight gradients, all layers in one launch
constexpr int kBK = 64;            // K elements per stage
constexpr int kAPlane = kBM * 2 * kBK;  // bytes of one A plane of a stage
constexpr int kEpiWarps = 8;
// A warp's 32 x 32 block, lane = row (v[i]: column i), turned through the
// warp's shared buffer tb (rows of 33 floats) so that global rows are read and
// written as whole lines.
constexpr int kTurnRow = 33;
constexpr int kTurnBytes = 32 * kTurnRow * 4;
template <int BN>
struct Ring {
    static constexpr int kNB = BN == kBN ? 1 : 2;  // B planes: weights one, activations two
    static constexpr int kBPlane = BN * 2 * kBK;
    static constexpr int kStageBytes = 2 * kAPlane + kNB * kBPlane;
    static constexpr int kStages = BN == kBN ? 4 : 3;
    // the layers' turn buffers hold their second input before the ring is free;
    // the weight gradients use the ring
    static constexpr int kTurnOffset = BN == kBN ? kStages * kStageBytes : 0;
    static constexpr int kBarOffset =
        kStages * kStageBytes + (BN == kBN ? kEpiWarps * kTurnBytes : 0);
    static constexpr int kSmem = 1024 + kBarOffset + 256;
    static_assert(kSmem <= 227 * 1024, "shared memory of the MLP GEMM");
    // accumulators side by side: the tensor core truncates its FP32 accumulator at
    // every product, about 2^-24 of it, so a weight gradient's K (the batch) is
    // summed in kAccs parts per CTA, which the epilogue adds.  Median error of a last
    // layer's gradient, width 512, 1800 rows (3 splits): 6.7e-6 with one accumulator,
    // 5.4e-6 with four (8 splits of one: 5.7e-6); 1024, 32768 rows: 1.1e-4 and 2.3e-5
    // (2.3e-5).  10 Adam steps of 1800 rows 1473 -> 1488 us.
    static constexpr int kAccs = BN == kBN ? 1 : 4;
};
constexpr int kThreads = 64 + 32 * kEpiWarps;  // warp 0 TMA, warp 1 MMA, then the epilogue
constexpr int kMaxLayers = 8;
constexpr int kInPad = 32;     // input features padded (a stage reads zeros beyond them)
constexpr int kMaxSplit = 4;   // splits of a weight gradient's K

enum Epi { kEpiHidden = 0, kEpiOut = 1, kEpiBwd = 2, kEpiGrad = 3, kEpiLoss = 4 };

struct MlpGemm {
    CUtensorMap a[2];  // A planes [rows][K], box 64 x 128
    CUtensorMap b[2];  // B planes [rows][K], box 64 x 64
    int na, nb;        // planes of A and B (products: every pair with ia + ib <= 1)
    int kb_total;      // 64-wide K blocks
    int kb_split;      // K blocks per split
    int mt, nt;        // tiles of rows and columns
    int mode;
    int rows_valid;    // A rows that carry data (batch rows); others are written as 0
    int cols_valid;    // B rows (output columns) written by kEpiGrad
    const float *bias;             // [N] (kEpiHidden, kEpiOut, kEpiLoss)
    const float *aux;              // pre-activations (kEpiBwd) or targets (kEpiLoss), [M][ld_aux]
    int ld_aux;
    float *out;                    // FP32 result [M][ld_out] (+ split * split_stride)
    int ld_out;
    int64_t split_stride;
    __nv_bfloat16 *hi, *lo;        // row-major planes [M][ld_bf]
    int ld_bf;
    __nv_bfloat16 *thi, *tlo;      // transposed planes [N][ld_t]
    int ld_t;
    float *bpart;                  // kEpiBwd, kEpiLoss: column sums per 32 rows [M / 32][ld_bf]
    // kEpiLoss: dL/dy = scale (y - t); squared errors per warp; step counters
    // and Adam bias corrections advanced when count_step
    float scale;
    double *part;
    int count_step;
    long long *step;
    float *corr;
    unsigned long long *err;
};

// The GEMMs of one launch: job j takes blockIdx.z in [z0[j], z0[j + 1]), its
// splits; CTAs beyond a job's tiles return.
template <int kJobs>
struct MlpSet {
    MlpGemm g[kJobs];
    int z0[kJobs + 1];
    int n;
};

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ float silu_f(float y) { return y / (1.0f + expf(-y)); }

__device__ __forceinline__ float silu_grad_f(float y) {
    const float s = 1.0f / (1.0f + expf(-y));
    return s * (1.0f + y * (1.0f - s));
}

__device__ __forceinline__ void split_bf16(float x, __nv_bfloat16 &h, __nv_bfloat16 &l) {
    h = __float2bfloat16_rn(x);
    l = __float2bfloat16_rn(x - __bfloat162float(h));
}

__device__ __forceinline__ void turn_put(float *tb, int lane, const float (&v)[32]) {
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 32; ++i) tb[lane * kTurnRow + i] = v[i];
    __syncwarp();
}

__device__ __forceinline__ void store_block_f32(float *dst, int ld, const float *tb, int lane) {
    dst += lane;
#pragma unroll
    for (int r = 0; r < 32; ++r) dst[(size_t)r * ld] = tb[r * kTurnRow + lane];
}

// Rows: half a warp a row, two columns a lane.
__device__ __forceinline__ void store_block_planes(__nv_bfloat16 *hi, __nv_bfloat16 *lo, int ld,
                                                   const float *tb, int lane) {
    const int c = (lane & 15) * 2, r0 = lane >> 4;
    hi += (size_t)r0 * ld + c;
    lo += (size_t)r0 * ld + c;
#pragma unroll
    for (int r = 0; r < 32; r += 2) {
        __nv_bfloat162 h, l;
        split_bf16(tb[(r + r0) * kTurnRow + c], h.x, l.x);
        split_bf16(tb[(r + r0) * kTurnRow + c + 1], h.y, l.y);
        *reinterpret_cast<__nv_bfloat162 *>(hi + (size_t)r * ld) = h;
        *reinterpret_cast<__nv_bfloat162 *>(lo + (size_t)r * ld) = l;
    }
}

// Columns of the block as rows of the transposed planes: half a warp a
// column, two rows a lane.
__device__ __forceinline__ void store_block_turned(__nv_bfloat16 *thi, __nv_bfloat16 *tlo, int ld_t,
                                                   const float *tb, int lane) {
    const int r = (lane & 15) * 2, c0 = lane >> 4;
    thi += (size_t)c0 * ld_t + r;
    tlo += (size_t)c0 * ld_t + r;
#pragma unroll
    for (int c = 0; c < 32; c += 2) {
        __nv_bfloat162 h, l;
        split_bf16(tb[r * kTurnRow + c + c0], h.x, l.x);
        split_bf16(tb[(r + 1) * kTurnRow + c + c0], h.y, l.y);
        *reinterpret_cast<__nv_bfloat162 *>(thi + (size_t)c * ld_t) = h;
        *reinterpret_cast<__nv_bfloat162 *>(tlo + (size_t)c * ld_t) = l;
    }
}

template <int kJobs, int BN>
__global__ void __launch_bounds__(kThreads, 1)
    k_mlp_gemm(const __grid_constant__ MlpSet<kJobs> set) {
    int job = 0;
    if (kJobs > 1)
        while (job + 1 < set.n && (int)blockIdx.z >= set.z0[job + 1]) ++job;
    const MlpGemm &p = set.g[job];
    const int split = blockIdx.z - set.z0[job];
    if ((int)blockIdx.x >= p.mt || (int)blockIdx.y >= p.nt) return;
    using R = Ring<BN>;
    constexpr int kStages = R::kStages, kStageBytes = R::kStageBytes, kBPlane = R::kBPlane;
    constexpr uint32_t kIdesc = ptx::idesc_bf16_f32(kBM, BN);
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    auto a_tile = [&](int s, int q) { return smem + s * kStageBytes + q * kAPlane; };
    auto b_tile = [&](int s, int q) { return smem + s * kStageBytes + 2 * kAPlane + q * kBPlane; };
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + R::kBarOffset);
    uint64_t *full = bars;
    uint64_t *empty = bars + kStages;
    uint64_t *tfull = bars + 2 * kStages;
    uint64_t *drain = tfull + 1;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(drain + 1);

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    volatile unsigned long long *err = p.err;
    const int kb0 = split * p.kb_split;
    const int nkb = min(p.kb_total, kb0 + p.kb_split) - kb0;  // >= 1 (host)
    // 32-wide K blocks per accumulator
    const int acc_blocks = (nkb * (kBK / 32) + R::kAccs - 1) / R::kAccs;
    const int m0 = blockIdx.x * kBM;
    const int n0 = blockIdx.y * BN;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            ptx::mbar_init(ptx::smem_u32(&full[s]), 1);
            ptx::mbar_init(ptx::smem_u32(&empty[s]), 1);
        }
        ptx::mbar_init(ptx::smem_u32(tfull), 1);
        ptx::mbar_init(ptx::smem_u32(drain), 1);
        ptx::fence_barrier_init();
    }
    if (warp == 1) {
        ptx::tmem_alloc(ptx::smem_u32(tmem_slot), R::kAccs * BN);
        ptx::tmem_relinquish();
    }
    if (threadIdx.x == 0) {
        for (int q = 0; q < p.na; ++q) ptx::prefetch_tmap(&p.a[q]);
        for (int q = 0; q < p.nb; ++q) ptx::prefetch_tmap(&p.b[q]);
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    // everything before this ran beside the previous launch; from here on its
    // results are read and its inputs overwritten
    pdl_wait();
    pdl_launch();

    if (warp == 0) {
        if (lane == 0) {
            // ------------------------------------------------------ TMA producer
            const uint32_t bytes = (uint32_t)(p.na * kAPlane + p.nb * kBPlane);
            int stage = 0;
            uint32_t phase = 0, used = 0, last_phase = 0;
            for (int kb = 0; kb < nkb; ++kb) {
                if (!ptx::mbar_wait(ptx::smem_u32(&empty[stage]), phase ^ 1u, err)) break;
                const uint32_t fb = ptx::smem_u32(&full[stage]);
                ptx::mbar_arrive_expect_tx(fb, bytes);
                const int kx = (kb0 + kb) * kBK;
                for (int q = 0; q < p.na; ++q)
                    ptx::tma_load_2d(ptx::smem_u32(a_tile(stage, q)), &p.a[q], fb, kx, m0);
                for (int q = 0; q < p.nb; ++q)
                    ptx::tma_load_2d(ptx::smem_u32(b_tile(stage, q)), &p.b[q], fb, kx, n0);
                used |= 1u << stage;
                last_phase = (last_phase & ~(1u << stage)) | (phase << stage);
                if (++stage == kStages) {
                    stage = 0;
                    phase ^= 1u;
                }
            }
            // every load issued here has landed before the CTA may exit
            for (int s = 0; s < kStages; ++s)
                if (used & (1u << s))
                    ptx::mbar_wait(ptx::smem_u32(&full[s]), (last_phase >> s) & 1u, err,
                                   200000000ull);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // ------------------------------------------------------ MMA issuer
            // products with ia + ib <= 1, the main product A0 B0 last
            int pa[3], pb[3], np = 0;
            if (p.na > 1) { pa[np] = 1; pb[np] = 0; ++np; }
            if (p.nb > 1) { pa[np] = 0; pb[np] = 1; ++np; }
            pa[np] = 0;
            pb[np] = 0;
            ++np;
            int stage = 0;
            uint32_t phase = 0, acc = 0;
            for (int kb = 0; kb < nkb; ++kb) {
                if (!ptx::mbar_wait(ptx::smem_u32(&full[stage]), phase, err)) break;
                ptx::tc_fence_after();
                // per 32 K the correction products first, A0 B0 last
#pragma unroll
                for (int h = 0; h < kBK / 32; ++h) {
                    uint32_t d = tmem_base;
                    if (R::kAccs > 1) {
                        const int block = kb * (kBK / 32) + h;
                        d += (uint32_t)(block / acc_blocks * BN);
                        if (block % acc_blocks == 0) acc = 0u;
                    }
                    for (int pr = 0; pr < np; ++pr) {
                        const uint32_t a0 = ptx::smem_u32(a_tile(stage, pa[pr])) + h * 64;
                        const uint32_t b0 = ptx::smem_u32(b_tile(stage, pb[pr])) + h * 64;
#pragma unroll
                        for (int kk = 0; kk < 2; ++kk) {
                            ptx::mma_bf16(d, ptx::desc_k_sw128(a0 + kk * 32),
                                          ptx::desc_k_sw128(b0 + kk * 32), kIdesc, acc);
                            acc = 1u;
                        }
                    }
                }
                ptx::mma_commit(ptx::smem_u32(&empty[stage]));
                if (++stage == kStages) {
                    stage = 0;
                    phase ^= 1u;
                }
            }
            ptx::mma_commit(ptx::smem_u32(tfull));
            ptx::mma_commit(ptx::smem_u32(drain));
            ptx::mbar_wait(ptx::smem_u32(drain), 0u, err, 200000000ull);
        }
    } else {
        // ---------------------------------------------------------- epilogue
        const int quarter = warp & 3;
        const int row0 = m0 + quarter * 32;
        float *tb = reinterpret_cast<float *>(smem + R::kTurnOffset + (warp - 2) * kTurnBytes);
        const int half = ((warp - 2) >> 2) * 32;
        const uint32_t tl = tmem_base + ((uint32_t)(quarter * 32) << 16);
        if constexpr (BN == kBNGrad) {
            // (every MMA has completed, so every load of the ring has been read)
            ptx::mbar_wait(ptx::smem_u32(tfull), 0u, err);
            __syncwarp();  // the TMEM loads are the whole warp's
            ptx::tc_fence_after();
            for (int c0 = half; c0 < BN && n0 + c0 < p.cols_valid; c0 += 64) {
                float v[32];
                ptx::tmem_ld32(tl + (uint32_t)c0, v);
                ptx::tmem_ld_wait();
                for (int b = acc_blocks, a = 1; b < nkb * (kBK / 32); b += acc_blocks, ++a) {
                    float u[32];
                    ptx::tmem_ld32(tl + (uint32_t)(a * BN + c0), u);
                    ptx::tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 32; ++i) v[i] += u[i];
                }
                turn_put(tb, lane, v);
                store_block_f32(p.out + split * p.split_stride + (size_t)row0 * p.ld_out + n0 + c0,
                                p.ld_out, tb, lane);
            }
        } else {
            const int col0 = n0 + half;
            const bool live = row0 + lane < p.rows_valid;
            // the second input, while the products run: the bias (column i in
            // lane i), and pre-activations or targets (which have rows_valid
            // rows only), every row's load in flight at once
            const float bias = p.bias ? p.bias[col0 + lane] : 0.0f;
            if (p.mode == kEpiBwd || p.mode == kEpiLoss) {
                const float *src = p.aux + (size_t)row0 * p.ld_aux + col0 + lane;
                const int nr = p.mode == kEpiBwd ? 32 : p.rows_valid - row0;
                float a[32];
#pragma unroll
                for (int r = 0; r < 32; ++r) a[r] = r < nr ? __ldg(src + (size_t)r * p.ld_aux) : 0.0f;
#pragma unroll
                for (int r = 0; r < 32; ++r) tb[r * kTurnRow + lane] = a[r];
                __syncwarp();
            }
            ptx::mbar_wait(ptx::smem_u32(tfull), 0u, err);
            __syncwarp();  // the TMEM loads are the whole warp's
            ptx::tc_fence_after();
            float v[32];
            ptx::tmem_ld32(tl + (uint32_t)half, v);
            ptx::tmem_ld_wait();
            if (p.mode == kEpiBwd) {
#pragma unroll
                for (int i = 0; i < 32; ++i)
                    v[i] = live ? v[i] * silu_grad_f(tb[lane * kTurnRow + i]) : 0.0f;
            } else {
#pragma unroll
                for (int i = 0; i < 32; ++i) v[i] += __shfl_sync(0xffffffffu, bias, i);
            }
            if (p.mode == kEpiHidden) {
#pragma unroll
                for (int i = 0; i < 32; ++i) v[i] = live ? v[i] : 0.0f;
                turn_put(tb, lane, v);
                store_block_f32(p.out + (size_t)row0 * p.ld_out + col0, p.ld_out, tb, lane);
#pragma unroll
                for (int i = 0; i < 32; ++i) v[i] = live ? silu_f(v[i]) : 0.0f;
            } else if (p.mode == kEpiLoss) {
                // the row's 32 squared errors summed in a tree (a chain of 32 FP32
                // additions errs by several times as much)
                float sq[32];
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    const float e = live ? v[i] - tb[lane * kTurnRow + i] : 0.0f;
                    sq[i] = e * e;
                    v[i] = p.scale * e;
                }
#pragma unroll
                for (int w = 16; w > 0; w >>= 1)
#pragma unroll
                    for (int i = 0; i < w; ++i) sq[i] += sq[i + w];
                double s = (double)sq[0];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                if (lane == 0)
                    p.part[((size_t)blockIdx.x * p.nt + blockIdx.y) * kEpiWarps + (warp - 2)] = s;
                if (p.count_step && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 64) {
                    const long long t = p.step[0] + 1;
                    p.step[0] = t;
                    p.step[1] += 1;  // steps of the current training call
                    p.corr[0] = (float)(1.0 - pow(0.9, (double)t));
                    p.corr[1] = (float)(1.0 - pow(0.999, (double)t));
                }
            }
            turn_put(tb, lane, v);
            if (p.mode == kEpiOut) {
                store_block_f32(p.out + (size_t)row0 * p.ld_out + col0, p.ld_out, tb, lane);
            } else {
                store_block_planes(p.hi + (size_t)row0 * p.ld_bf + col0,
                                   p.lo + (size_t)row0 * p.ld_bf + col0, p.ld_bf, tb, lane);
                store_block_turned(p.thi + (size_t)col0 * p.ld_t + row0,
                                   p.tlo + (size_t)col0 * p.ld_t + row0, p.ld_t, tb, lane);
                if (p.mode != kEpiHidden) {
                    float s = 0.0f;
#pragma unroll
                    for (int r = 0; r < 32; ++r) s += tb[r * kTurnRow + lane];
                    p.bpart[(size_t)(row0 >> 5) * p.ld_bf + col0 + lane] = s;
                }
            }
        }
    }

    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem_base, R::kAccs * BN);
    }
}

// Inputs X [B][in_dim] FP32 -> planes [B_pad][32] and transposed [32][ld_t];
// padding rows and columns are 0.
__global__ void k_mlp_input(const float *__restrict__ X, int B, int in_dim, int B_pad,
                            __nv_bfloat16 *hi, __nv_bfloat16 *lo, __nv_bfloat16 *thi,
                            __nv_bfloat16 *tlo, int ld_t) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= B_pad * kInPad) return;
    const int row = idx / kInPad;
    const int c = idx % kInPad;
    const float x = (row < B && c < in_dim) ? X[(size_t)row * in_dim + c] : 0.0f;
    __nv_bfloat16 h, l;
    split_bf16(x, h, l);
    hi[idx] = h;
    lo[idx] = l;
    thi[(size_t)c * ld_t + row] = h;
    tlo[(size_t)c * ld_t + row] = l;
}

struct Layout {
    int L;
    int n_out[kMaxLayers], k_pad[kMaxLayers];
    int64_t off_W[kMaxLayers], off_b[kMaxLayers], end[kMaxLayers];  // master layout
    const float *dw[kMaxLayers];  // [S][n_out][k_pad] partials
    const float *db[kMaxLayers];  // [SB][n_out] column sums
    int S[kMaxLayers];
    int SB;
    __nv_bfloat16 *wbf[kMaxLayers], *wtbf[kMaxLayers];
};

// Adam on every master element; refreshes the BF16 W and W^T copies.  With
// grad_out != NULL only writes the gradient (no update).  Gradients are the
// fixed-order sums of the split partials.  One block (32 x 8) per 32 x 32 tile
// of a weight matrix, W^T written through shared memory as rows of 64 bytes;
// tile column k_pad / 32 of a layer stands for its biases.  The last block sums
// the nloss squared errors into the loss (out[step] and *out64).
__global__ void __launch_bounds__(256)
    k_mlp_adam(Layout lay, float *__restrict__ master, float *__restrict__ mom1,
               float *__restrict__ mom2, const float *__restrict__ lr_tab, const long long *step,
               const float *corr, float *__restrict__ grad_out, const double *__restrict__ part,
               int nloss, double elements, float *__restrict__ hist, double *__restrict__ out64) {
    __shared__ __nv_bfloat16 turn[32][34];
    __shared__ double red[256];
    pdl_wait();
    if (blockIdx.x == gridDim.x - 1) {
        double s = 0.0;
        for (int i = threadIdx.x; i < nloss; i += 256) s += part[i];
        red[threadIdx.x] = s;
        __syncthreads();
        for (int w = 128; w > 0; w >>= 1) {
            if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            const double loss = red[0] / elements;
            if (hist) hist[step[1] - 1] = (float)loss;
            *out64 = loss;
        }
        return;
    }
    int l = 0, t = blockIdx.x;
    for (;; ++l) {
        const int nt = (lay.k_pad[l] / 32 + 1) * (lay.n_out[l] / 32);
        if (t < nt) break;
        t -= nt;
    }
    const int kt = lay.k_pad[l] / 32 + 1;
    const int n0 = (t / kt) * 32, k0 = (t % kt) * 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const bool is_w = k0 < lay.k_pad[l];
    const int kp = lay.k_pad[l];
    const float lr = grad_out ? 0.0f : lr_tab[step[1] - 1];
    const float c0 = grad_out ? 1.0f : corr[0], c1 = grad_out ? 1.0f : corr[1];
    auto update = [&](float &w, float &m1, float &m2, float g) {
        m1 = 0.9f * m1 + 0.1f * g;
        m2 = 0.999f * m2 + 0.001f * g * g;
        w = w - lr * (m1 / c0) / (sqrtf(m2 / c1) + 1e-8f);
    };
    if (!is_w) {
        float *sums = reinterpret_cast<float *>(red);  // [8][32]
        float b = 0.0f;
#pragma unroll 4
        for (int q = ty; q < lay.SB; q += 8) b += lay.db[l][(size_t)q * lay.n_out[l] + n0 + tx];
        sums[threadIdx.x] = b;
        __syncthreads();
        if (ty == 0) {
#pragma unroll
            for (int q = 1; q < 8; ++q) b += sums[q * 32 + tx];
            const int64_t i = lay.off_b[l] + n0 + tx;
            if (grad_out) grad_out[i] = b;
            else update(master[i], mom1[i], mom2[i], b);
        }
        return;
    }
    // four consecutive inputs k of one output n per thread, every load in flight
    const int n = threadIdx.x >> 3, k = (threadIdx.x & 7) * 4;
    const int64_t plane = (int64_t)lay.n_out[l] * kp;
    const int64_t j = (int64_t)(n0 + n) * kp + k0 + k, i = lay.off_W[l] + j;
    float4 part_g[kMaxSplit];
#pragma unroll
    for (int z = 0; z < kMaxSplit; ++z)
        if (z < lay.S[l]) part_g[z] = *reinterpret_cast<const float4 *>(lay.dw[l] + z * plane + j);
    float4 w, m1, m2;
    if (!grad_out) {
        w = *reinterpret_cast<const float4 *>(master + i);
        m1 = *reinterpret_cast<const float4 *>(mom1 + i);
        m2 = *reinterpret_cast<const float4 *>(mom2 + i);
    }
    float4 g = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
    for (int z = 0; z < kMaxSplit; ++z)
        if (z < lay.S[l]) {
            g.x += part_g[z].x;
            g.y += part_g[z].y;
            g.z += part_g[z].z;
            g.w += part_g[z].w;
        }
    if (grad_out) {
        *reinterpret_cast<float4 *>(grad_out + i) = g;
        return;
    }
    update(w.x, m1.x, m2.x, g.x);
    update(w.y, m1.y, m2.y, g.y);
    update(w.z, m1.z, m2.z, g.z);
    update(w.w, m1.w, m2.w, g.w);
    *reinterpret_cast<float4 *>(master + i) = w;
    *reinterpret_cast<float4 *>(mom1 + i) = m1;
    *reinterpret_cast<float4 *>(mom2 + i) = m2;
    __nv_bfloat16 b[4] = {__float2bfloat16_rn(w.x), __float2bfloat16_rn(w.y),
                          __float2bfloat16_rn(w.z), __float2bfloat16_rn(w.w)};
    __nv_bfloat162 *wb = reinterpret_cast<__nv_bfloat162 *>(lay.wbf[l] + j);
    wb[0] = __nv_bfloat162(b[0], b[1]);
    wb[1] = __nv_bfloat162(b[2], b[3]);
    if (!lay.wtbf[l]) return;
#pragma unroll
    for (int q = 0; q < 4; ++q) turn[k + q][n] = b[q];
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int kk = ty + 8 * q;
        lay.wtbf[l][(size_t)(k0 + kk) * lay.n_out[l] + n0 + tx] = turn[kk][tx];
    }
}

// BF16 copies of the master weights (after gbs_mlp_set_params).
__global__ void k_mlp_refresh(Layout lay, int64_t total, const float *__restrict__ master) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    int l = 0;
    while (l + 1 < lay.L && i >= lay.end[l]) ++l;
    if (i >= lay.off_b[l]) return;
    const int64_t j = i - lay.off_W[l];
    const int n = (int)(j / lay.k_pad[l]);
    const int k = (int)(j % lay.k_pad[l]);
    const __nv_bfloat16 wb = __float2bfloat16_rn(master[i]);
    lay.wbf[l][j] = wb;
    if (lay.wtbf[l]) lay.wtbf[l][(size_t)k * lay.n_out[l] + n] = wb;
}

template <typename T>
int mlp_alloc(T **p, size_t count, std::vector<void *> &owned) {
    *p = nullptr;
    if (count == 0) return GBS_OK;
    cudaError_t e = cudaMalloc(reinterpret_cast<void **>(p), count * sizeof(T));
    if (e != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return set_error(GBS_ENOMEM, "cudaMalloc(%zu bytes) for the MLP failed: %s",
                         count * sizeof(T), cudaGetErrorString(e));
    }
    owned.push_back(*p);
    e = cudaMemset(*p, 0, count * sizeof(T));
    if (e != cudaSuccess) return set_error(GBS_ECUDA, "cudaMemset failed: %s", cudaGetErrorString(e));
    return GBS_OK;
}

bool g_attr_done[64] = {};

}  // namespace
}  // namespace gbs

using namespace gbs;

struct gbs_mlp {
    int in_dim = 0, width = 0, out_dim = 0, L = 0, max_batch = 0, Bmax = 0;  // Bmax: padded
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int device = 0;
    std::vector<void *> owned;
    Layout lay = {};
    int64_t nmaster = 0, nparams = 0;
    float *master = nullptr, *m1 = nullptr, *m2 = nullptr, *grad = nullptr;
    __nv_bfloat16 *xp = nullptr, *xtp = nullptr;           // 2 planes each
    float *pre[kMaxLayers] = {};                            // hidden layers
    __nv_bfloat16 *hp[kMaxLayers] = {}, *htp[kMaxLayers] = {};
    float *y = nullptr;
    __nv_bfloat16 *dyp[kMaxLayers] = {}, *dytp[kMaxLayers] = {};
    float *dw[kMaxLayers] = {}, *db[kMaxLayers] = {};
    double *part = nullptr;     // squared errors per epilogue warp
    int nloss = 0;
    long long *step = nullptr;  // [2]: Adam steps, steps of the current training call
    float *corr = nullptr;      // [2]: 1 - beta1^t, 1 - beta2^t
    float *lr = nullptr;
    int lr_cap = 0;
    float *loss_hist = nullptr;
    double *loss64 = nullptr;
    unsigned long long *err = nullptr;
};

namespace {

size_t plane_elems(int rows, int cols) { return (size_t)rows * cols; }

// Tensor map of a BF16 plane [rows][inner] in boxes of kBK x box_rows with the
// 128-byte swizzle; reads beyond its ends are zeros.
int encode_plane(CUtensorMap *map, void *base, uint64_t inner, uint64_t rows, uint32_t box_rows) {
    return encode_2d(map, base, inner, rows, inner * 2, kBK, box_rows, CU_TENSOR_MAP_SWIZZLE_128B);
}

int make_gemm(gbs_mlp *m, MlpGemm &p, int BN, int mode, __nv_bfloat16 *a0, __nv_bfloat16 *a1,
              int a_rows, int a_ld, __nv_bfloat16 *b0, __nv_bfloat16 *b1, int b_rows, int b_ld,
              int K, int M, int N, int split) {
    p = MlpGemm{};
    int rc;
    if ((rc = encode_plane(&p.a[0], a0, (uint64_t)a_ld, (uint64_t)a_rows, kBM))) return rc;
    p.na = 1;
    if (a1) {
        if ((rc = encode_plane(&p.a[1], a1, (uint64_t)a_ld, (uint64_t)a_rows, kBM))) return rc;
        p.na = 2;
    }
    if ((rc = encode_plane(&p.b[0], b0, (uint64_t)b_ld, (uint64_t)b_rows, (uint32_t)BN))) return rc;
    p.nb = 1;
    if (b1) {
        if ((rc = encode_plane(&p.b[1], b1, (uint64_t)b_ld, (uint64_t)b_rows, (uint32_t)BN))) return rc;
        p.nb = 2;
    }
    p.kb_total = (K + kBK - 1) / kBK;
    const int S = std::max(1, std::min(split, p.kb_total));
    p.kb_split = (p.kb_total + S - 1) / S;
    p.mt = M / kBM;
    p.nt = (N + BN - 1) / BN;
    p.mode = mode;
    p.err = m->err;
    return GBS_OK;
}

int splits_of(const MlpGemm &p) { return (p.kb_total + p.kb_split - 1) / p.kb_split; }

// A kernel of the step, its prologue overlapping the launch before it.
template <typename... P, typename... A>
int launch_pdl(gbs_mlp *m, void (*kern)(P...), dim3 grid, int threads, size_t smem, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = m->stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    GBS_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, args...));
    return GBS_OK;
}

template <int kJobs, int BN>
int launch(gbs_mlp *m, const MlpSet<kJobs> &s) {
    dim3 grid(0, 0, (unsigned)s.z0[s.n]);
    for (int j = 0; j < s.n; ++j) {
        grid.x = std::max(grid.x, (unsigned)s.g[j].mt);
        grid.y = std::max(grid.y, (unsigned)s.g[j].nt);
    }
    return launch_pdl(m, k_mlp_gemm<kJobs, BN>, grid, kThreads, Ring<BN>::kSmem, s);
}

// The launches of one pass, built once per call.
struct Plan {
    std::vector<MlpSet<1>> layers;  // forward, then data gradients
    MlpSet<kMaxLayers> grad;        // weight gradients
};

int ensure_attr() {
    int dev = 0;
    GBS_CUDA_TRY(cudaGetDevice(&dev));
    if (dev >= 0 && dev < 64 && g_attr_done[dev]) return GBS_OK;
    GBS_CUDA_TRY(cudaFuncSetAttribute(k_mlp_gemm<1, kBN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      Ring<kBN>::kSmem));
    GBS_CUDA_TRY(cudaFuncSetAttribute(k_mlp_gemm<kMaxLayers, kBNGrad>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      Ring<kBNGrad>::kSmem));
    if (dev >= 0 && dev < 64) g_attr_done[dev] = true;
    return GBS_OK;
}

// Forward of `batch` rows (B_pad = batch rounded up to 128); input planes
// must be written already.  Output into m->y, or (targets T given) the loss
// gradient into the last layer's planes and the squared errors into m->part.
int plan_forward(gbs_mlp *m, Plan &plan, int batch, const float *T = nullptr, int count_step = 0) {
    const int Bp = (batch + kBM - 1) / kBM * kBM;
    int rc;
    for (int l = 0; l < m->L; ++l) {
        MlpGemm g;
        const bool last = l == m->L - 1;
        __nv_bfloat16 *a0 = l == 0 ? m->xp : m->hp[l - 1];
        __nv_bfloat16 *a1 = a0 + (size_t)m->Bmax * (l == 0 ? kInPad : m->width);
        const int k = m->lay.k_pad[l];
        const int n = m->lay.n_out[l];
        if ((rc = make_gemm(m, g, kBN, !last ? kEpiHidden : T ? kEpiLoss : kEpiOut, a0, a1, m->Bmax, k,
                            m->lay.wbf[l], nullptr, n, k, k, Bp, n, 1)))
            return rc;
        g.rows_valid = batch;
        g.bias = m->master + m->lay.off_b[l];
        __nv_bfloat16 *rows = last ? m->dyp[l] : m->hp[l], *cols = last ? m->dytp[l] : m->htp[l];
        g.out = last ? m->y : m->pre[l];
        g.ld_out = n;
        g.hi = rows;
        g.lo = rows + (size_t)m->Bmax * n;
        g.ld_bf = n;
        g.thi = cols;
        g.tlo = cols + (size_t)n * m->Bmax;
        g.ld_t = m->Bmax;
        if (last && T) {
            g.aux = T;
            g.ld_aux = n;
            g.bpart = m->db[l];
            g.scale = 2.0f / ((float)batch * (float)n);
            g.part = m->part;
            g.count_step = count_step;
            g.step = m->step;
            g.corr = m->corr;
            m->nloss = g.mt * g.nt * kEpiWarps;
        }
        plan.layers.push_back(MlpSet<1>{{g}, {0, 1}, 1});
    }
    return GBS_OK;
}

int run_input(gbs_mlp *m, const float *X, int batch) {
    const int Bp = (batch + kBM - 1) / kBM * kBM;
    const int total = Bp * kInPad;
    k_mlp_input<<<(total + 255) / 256, 256, 0, m->stream>>>(
        X, batch, m->in_dim, Bp, m->xp, m->xp + (size_t)m->Bmax * kInPad, m->xtp,
        m->xtp + (size_t)kInPad * m->Bmax, m->Bmax);
    GBS_LAUNCH_CHECK();
    return GBS_OK;
}

// Backward and the gradient partials of one batch (after a forward with
// targets).
int plan_backward(gbs_mlp *m, Plan &plan, int batch) {
    const int Bp = (batch + kBM - 1) / kBM * kBM;
    const int L = m->L;
    int rc;
    // data gradients, layer L-1 .. 1 (0-based l: dY_{l-1} from dY_l)
    for (int l = L - 1; l >= 1; --l) {
        const int n = m->lay.n_out[l];
        const int k = m->lay.k_pad[l];  // = width
        MlpGemm g;
        if ((rc = make_gemm(m, g, kBN, kEpiBwd, m->dyp[l], m->dyp[l] + (size_t)m->Bmax * n, m->Bmax, n,
                            m->lay.wtbf[l], nullptr, k, n, n, Bp, k, 1)))
            return rc;
        g.rows_valid = batch;
        g.aux = m->pre[l - 1];
        g.ld_aux = k;
        g.hi = m->dyp[l - 1];
        g.lo = m->dyp[l - 1] + (size_t)m->Bmax * k;
        g.ld_bf = k;
        g.thi = m->dytp[l - 1];
        g.tlo = m->dytp[l - 1] + (size_t)k * m->Bmax;
        g.ld_t = m->Bmax;
        g.bpart = m->db[l - 1];
        plan.layers.push_back(MlpSet<1>{{g}, {0, 1}, 1});
    }
    // weight gradients: dW_l = dY_l^T H_{l-1}, K = the batch, split so that the
    // launch is one wave: the hidden and output layers alike, the first (one
    // column tile) from what they leave; two splits at least, which with their
    // accumulators sum the batch in eight parts, 32 rows being the smallest
    int sms = 0, tiles = 0;
    GBS_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, m->device));
    for (int l = 1; l < L; ++l)
        tiles += (m->lay.n_out[l] / kBM) * ((m->lay.k_pad[l] + kBNGrad - 1) / kBNGrad);
    const int S = std::max(2, std::min(kMaxSplit, sms / tiles));
    const int S0 = std::max(2, std::min(kMaxSplit, (sms - S * tiles) / (m->lay.n_out[0] / kBM)));
    plan.grad.n = L;
    plan.grad.z0[0] = 0;
    for (int l = 0; l < L; ++l) {
        const int n = m->lay.n_out[l];
        const int k = m->lay.k_pad[l];
        __nv_bfloat16 *b0 = l == 0 ? m->xtp : m->htp[l - 1];
        __nv_bfloat16 *b1 = b0 + (size_t)k * m->Bmax;
        MlpGemm &g = plan.grad.g[l];
        if ((rc = make_gemm(m, g, kBNGrad, kEpiGrad, m->dytp[l], m->dytp[l] + (size_t)n * m->Bmax, n,
                            m->Bmax, b0, b1, k, m->Bmax, Bp, n, k, l ? S : S0)))
            return rc;
        g.cols_valid = k;
        g.out = m->dw[l];
        g.ld_out = k;
        g.split_stride = (int64_t)n * k;
        m->lay.S[l] = splits_of(g);
        plan.grad.z0[l + 1] = plan.grad.z0[l] + m->lay.S[l];
    }
    m->lay.SB = Bp / 32;
    return GBS_OK;
}

int run_layers(gbs_mlp *m, const Plan &plan) {
    int rc;
    for (const MlpSet<1> &s : plan.layers)
        if ((rc = launch<1, kBN>(m, s))) return rc;
    return GBS_OK;
}

// Adam (or, with grad_out, the gradient alone) and the loss.
int run_adam(gbs_mlp *m, int batch, float *hist, float *grad_out) {
    unsigned tiles = 0;
    for (int l = 0; l < m->L; ++l) {
        m->lay.dw[l] = m->dw[l];
        m->lay.db[l] = m->db[l];
        tiles += (unsigned)((m->lay.k_pad[l] / 32 + 1) * (m->lay.n_out[l] / 32));
    }
    return launch_pdl(m, k_mlp_adam, dim3(tiles + 1), 256, 0, m->lay, m->master, m->m1, m->m2,
                      (const float *)m->lr, (const long long *)m->step, (const float *)m->corr,
                      grad_out, (const double *)m->part, m->nloss,
                      (double)batch * (double)m->out_dim, hist, m->loss64);
}

int check_err(gbs_mlp *m) {
    unsigned long long h = 0;
    GBS_CUDA_TRY(cudaMemcpyAsync(&h, m->err, sizeof(h), cudaMemcpyDeviceToHost, m->stream));
    GBS_CUDA_TRY(cudaStreamSynchronize(m->stream));
    if (h) {
        cudaMemsetAsync(m->err, 0, sizeof(unsigned long long), m->stream);
        return set_error(GBS_ETIMEOUT, "an MLP GEMM gave up waiting on its pipeline");
    }
    return GBS_OK;
}

int check_batch(gbs_mlp *m, int batch) {
    if (batch < 1 || batch > m->max_batch)
        return set_error(GBS_EINVAL, "batch %d outside [1, %d]", batch, m->max_batch);
    return GBS_OK;
}

// Whether every value is finite: the largest magnitude's bit pattern (written
// to vectorise).
__attribute__((optimize("O3"))) bool all_finite(const float *v, int64_t n) {
    const uint32_t *b = reinterpret_cast<const uint32_t *>(v);
    uint32_t top = 0;
    for (int64_t i = 0; i < n; ++i) top = std::max(top, b[i] & 0x7fffffffu);
    return top < 0x7f800000u;
}

// Packed (user) parameters <-> master layout: the first layer's weights have
// padded rows, everything after them is the same in both.
int copy_params(gbs_mlp *m, float *master, float *packed, bool to_device) {
    const size_t w0 = (size_t)m->width * m->in_dim;
    const size_t rest = (size_t)(m->nmaster - m->lay.off_b[0]);
    const cudaMemcpyKind kind = to_device ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToHost;
    const size_t pu = sizeof(float) * m->in_dim, pm = sizeof(float) * kInPad;
    GBS_CUDA_TRY(cudaMemcpy2DAsync(to_device ? master : packed, to_device ? pm : pu,
                                   to_device ? packed : master, to_device ? pu : pm, pu,
                                   (size_t)m->width, kind, m->stream));
    float *a = master + m->lay.off_b[0], *b = packed + w0;
    GBS_CUDA_TRY(cudaMemcpyAsync(to_device ? a : b, to_device ? b : a, sizeof(float) * rest, kind,
                                 m->stream));
    return GBS_OK;
}

void destroy(gbs_mlp *m) {
    if (!m) return;
    for (void *p : m->owned) cudaFree(p);
    if (m->own_stream && m->stream) cudaStreamDestroy(m->stream);
    delete m;
}

}  // namespace

extern "C" {

int gbs_mlp_create(int in_dim, int width, int out_dim, int layers, int max_batch, void *stream,
                   gbs_mlp_t *out) {
    if (!out) return set_error(GBS_EINVAL, "out is NULL");
    *out = nullptr;
    if (in_dim < 1 || in_dim > kInPad) return set_error(GBS_EINVAL, "in_dim must be in [1, 32]");
    if (width < 256 || width > 4096 || width % 256 || out_dim < 256 || out_dim > 4096 ||
        out_dim % 256)
        return set_error(GBS_EINVAL, "width and out_dim must be multiples of 256 in [256, 4096]");
    if (layers < 2 || layers > kMaxLayers)
        return set_error(GBS_EINVAL, "layers must be in [2, %d]", kMaxLayers);
    if (max_batch < 1 || max_batch > 65536) return set_error(GBS_EINVAL, "max_batch must be in [1, 65536]");
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return set_error(GBS_ECUDA, "no usable CUDA device");
    }
    if (!device_has_tcgen05(dev)) return set_error(GBS_ENOTSUP, "this library is built for sm_103a (GB300) only");
    int rc;
    if ((rc = ensure_attr())) return rc;
    gbs_mlp *m = new (std::nothrow) gbs_mlp();
    if (!m) return set_error(GBS_ENOMEM, "host allocation failed");
    m->in_dim = in_dim;
    m->width = width;
    m->out_dim = out_dim;
    m->L = layers;
    m->max_batch = max_batch;
    m->Bmax = (max_batch + kBM - 1) / kBM * kBM;
    m->device = dev;
    if (stream) {
        m->stream = static_cast<cudaStream_t>(stream);
    } else {
        if (cudaStreamCreateWithFlags(&m->stream, cudaStreamNonBlocking) != cudaSuccess) {
            delete m;
            return set_error(GBS_ECUDA, "cudaStreamCreate failed");
        }
        m->own_stream = true;
    }
    auto fail = [&](int code) {
        destroy(m);
        return code;
    };
    Layout &lay = m->lay;
    lay.L = layers;
    int64_t off = 0;
    m->nparams = 0;
    for (int l = 0; l < layers; ++l) {
        lay.n_out[l] = l == layers - 1 ? out_dim : width;
        lay.k_pad[l] = l == 0 ? kInPad : width;
        lay.off_W[l] = off;
        off += (int64_t)lay.n_out[l] * lay.k_pad[l];
        lay.off_b[l] = off;
        off += lay.n_out[l];
        lay.end[l] = off;
        m->nparams += (int64_t)lay.n_out[l] * (l == 0 ? in_dim : width) + lay.n_out[l];
    }
    m->nmaster = off;
    const int B = m->Bmax;
    if ((rc = mlp_alloc(&m->master, (size_t)off, m->owned)) ||
        (rc = mlp_alloc(&m->m1, (size_t)off, m->owned)) ||
        (rc = mlp_alloc(&m->m2, (size_t)off, m->owned)) ||
        (rc = mlp_alloc(&m->grad, (size_t)off, m->owned)) ||
        (rc = mlp_alloc(&m->xp, 2 * plane_elems(B, kInPad), m->owned)) ||
        (rc = mlp_alloc(&m->xtp, 2 * plane_elems(kInPad, B), m->owned)) ||
        (rc = mlp_alloc(&m->y, plane_elems(B, out_dim), m->owned)) ||
        (rc = mlp_alloc(&m->part, (size_t)(B / kBM) * (out_dim / kBN) * kEpiWarps, m->owned)) ||
        (rc = mlp_alloc(&m->step, 2, m->owned)) || (rc = mlp_alloc(&m->corr, 2, m->owned)) ||
        (rc = mlp_alloc(&m->loss64, 1, m->owned)) || (rc = mlp_alloc(&m->err, 1, m->owned)))
        return fail(rc);
    for (int l = 0; l < layers; ++l) {
        const int n = lay.n_out[l], k = lay.k_pad[l];
        if ((rc = mlp_alloc(&lay.wbf[l], plane_elems(n, k), m->owned)) ||
            (l > 0 && (rc = mlp_alloc(&lay.wtbf[l], plane_elems(k, n), m->owned))) ||
            (rc = mlp_alloc(&m->dyp[l], 2 * plane_elems(B, n), m->owned)) ||
            (rc = mlp_alloc(&m->dytp[l], 2 * plane_elems(n, B), m->owned)) ||
            (rc = mlp_alloc(&m->dw[l], (size_t)kMaxSplit * plane_elems(n, k), m->owned)) ||
            (rc = mlp_alloc(&m->db[l], plane_elems(B / 32, n), m->owned)))
            return fail(rc);
        if (l < layers - 1) {
            if ((rc = mlp_alloc(&m->pre[l], plane_elems(B, n), m->owned)) ||
                (rc = mlp_alloc(&m->hp[l], 2 * plane_elems(B, n), m->owned)) ||
                (rc = mlp_alloc(&m->htp[l], 2 * plane_elems(n, B), m->owned)))
                return fail(rc);
        }
    }
    *out = m;
    return GBS_OK;
}

int gbs_mlp_param_count(gbs_mlp_t m, int64_t *count) {
    if (!m || !count) return set_error(GBS_EINVAL, "NULL argument");
    *count = m->nparams;
    return GBS_OK;
}

int gbs_mlp_set_params(gbs_mlp_t m, const float *params) {
    if (!m || !params) return set_error(GBS_EINVAL, "NULL argument");
    if (!all_finite(params, m->nparams))
        for (int64_t i = 0; i < m->nparams; ++i)
            if (!std::isfinite(params[i])) return set_error(GBS_EINVAL, "parameter %lld is not finite", (long long)i);
    int rc;
    const size_t bytes = sizeof(float) * (size_t)m->nmaster;
    GBS_CUDA_TRY(cudaMemsetAsync(m->master, 0, sizeof(float) * (size_t)m->lay.off_b[0], m->stream));
    if ((rc = copy_params(m, m->master, const_cast<float *>(params), true))) return rc;
    GBS_CUDA_TRY(cudaMemsetAsync(m->m1, 0, bytes, m->stream));
    GBS_CUDA_TRY(cudaMemsetAsync(m->m2, 0, bytes, m->stream));
    GBS_CUDA_TRY(cudaMemsetAsync(m->step, 0, 2 * sizeof(long long), m->stream));
    k_mlp_refresh<<<(unsigned)((m->nmaster + 255) / 256), 256, 0, m->stream>>>(m->lay, m->nmaster,
                                                                                m->master);
    GBS_LAUNCH_CHECK();
    GBS_CUDA_TRY(cudaStreamSynchronize(m->stream));
    return GBS_OK;
}

static int copy_packed(gbs_mlp_t m, const float *src_dev, float *dst) {
    int rc;
    if ((rc = copy_params(m, const_cast<float *>(src_dev), dst, false))) return rc;
    GBS_CUDA_TRY(cudaStreamSynchronize(m->stream));
    return GBS_OK;
}

int gbs_mlp_get_params(gbs_mlp_t m, float *params) {
    if (!m || !params) return set_error(GBS_EINVAL, "NULL argument");
    return copy_packed(m, m->master, params);
}

int gbs_mlp_get_adam_state(gbs_mlp_t m, float *mom1, float *mom2, int64_t *step) {
    if (!m) return set_error(GBS_EINVAL, "NULL argument");
    int rc;
    if (mom1 && (rc = copy_packed(m, m->m1, mom1))) return rc;
    if (mom2 && (rc = copy_packed(m, m->m2, mom2))) return rc;
    if (step) {
        long long h[2] = {0, 0};
        GBS_CUDA_TRY(cudaMemcpyAsync(h, m->step, sizeof(h), cudaMemcpyDeviceToHost, m->stream));
        GBS_CUDA_TRY(cudaStreamSynchronize(m->stream));
        *step = h[0];
    }
    return GBS_OK;
}

int gbs_mlp_forward(gbs_mlp_t m, const float *X_dev, int batch, float *Y_dev) {
    if (!m || !X_dev || !Y_dev) return set_error(GBS_EINVAL, "NULL argument");
    int rc;
    if ((rc = check_batch(m, batch))) return rc;
    Plan plan;
    if ((rc = plan_forward(m, plan, batch)) || (rc = run_input(m, X_dev, batch)) ||
        (rc = run_layers(m, plan)))
        return rc;
    GBS_CUDA_TRY(cudaMemcpyAsync(Y_dev, m->y, sizeof(float) * (size_t)batch * m->out_dim,
                                 cudaMemcpyDeviceToDevice, m->stream));
    return GBS_OK;
}

int gbs_mlp_gradients(gbs_mlp_t m, const float *X_dev, const float *T_dev, int batch, double *loss,
                      float *grad) {
    if (!m || !X_dev || !T_dev) return set_error(GBS_EINVAL, "NULL argument");
    int rc;
    if ((rc = check_batch(m, batch))) return rc;
    Plan plan;
    if ((rc = plan_forward(m, plan, batch, T_dev)) || (rc = plan_backward(m, plan, batch)) ||
        (rc = run_input(m, X_dev, batch)) || (rc = run_layers(m, plan)) ||
        (rc = launch<kMaxLayers, kBNGrad>(m, plan.grad)) ||
        (rc = run_adam(m, batch, nullptr, m->grad)))
        return rc;
    if ((rc = check_err(m))) return rc;
    if (loss) {
        GBS_CUDA_TRY(cudaMemcpyAsync(loss, m->loss64, sizeof(double), cudaMemcpyDeviceToHost, m->stream));
        GBS_CUDA_TRY(cudaStreamSynchronize(m->stream));
    }
    if (grad && (rc = copy_packed(m, m->grad, grad))) return rc;
    return GBS_OK;
}

int gbs_mlp_train(gbs_mlp_t m, const float *X_dev, const float *T_dev, int batch, int steps,
                  const float *lr, float *loss_hist) {
    if (!m || !X_dev || !T_dev || !lr) return set_error(GBS_EINVAL, "NULL argument");
    if (steps < 0) return set_error(GBS_EINVAL, "steps must be >= 0");
    int rc;
    if ((rc = check_batch(m, batch))) return rc;
    if (steps == 0) return GBS_OK;
    for (int i = 0; i < steps; ++i)
        if (!std::isfinite(lr[i]) || lr[i] < 0.0f) return set_error(GBS_EINVAL, "lr[%d] invalid", i);
    if (steps > m->lr_cap) {
        float *p = nullptr;
        if ((rc = mlp_alloc(&p, (size_t)steps, m->owned))) return rc;
        m->lr = p;
        m->lr_cap = steps;
        float *h = nullptr;
        if ((rc = mlp_alloc(&h, (size_t)steps, m->owned))) return rc;
        m->loss_hist = h;
    }
    GBS_CUDA_TRY(cudaMemcpyAsync(m->lr, lr, sizeof(float) * steps, cudaMemcpyHostToDevice, m->stream));
    GBS_CUDA_TRY(cudaMemsetAsync(m->step + 1, 0, sizeof(long long), m->stream));
    if ((rc = run_input(m, X_dev, batch))) return rc;
    // direct launches, not a graph: a step is 9 launches that the host issues
    // in a third of the time they run, and each overlaps the one before it
    // across steps too
    Plan plan;
    if ((rc = plan_forward(m, plan, batch, T_dev, 1)) || (rc = plan_backward(m, plan, batch)))
        return rc;
    for (int i = 0; i < steps; ++i)
        if ((rc = run_layers(m, plan)) || (rc = launch<kMaxLayers, kBNGrad>(m, plan.grad)) ||
            (rc = run_adam(m, batch, m->loss_hist, nullptr)))
            return rc;
    if ((rc = check_err(m))) return rc;
    if (loss_hist)
        GBS_CUDA_TRY(cudaMemcpyAsync(loss_hist, m->loss_hist, sizeof(float) * steps,
                                     cudaMemcpyDeviceToHost, m->stream));
    GBS_CUDA_TRY(cudaStreamSynchronize(m->stream));
    return GBS_OK;
}

void gbs_mlp_free(gbs_mlp_t m) { destroy(m); }

}  // extern "C"
