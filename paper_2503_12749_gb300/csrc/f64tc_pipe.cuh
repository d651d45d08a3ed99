// The pipeline of the exact digit-product contractions (f64tc.cuh): bulk copies
// of operand stages, the products of the digits into eight sums D_d per
// sub-tile, and the barriers between them and the epilogue warps.  Used by the
// FP64 GEMM (k_gemm_f64tc.cu) and the joint generating functions
// (k_gf2d_tc.cu), which differ in what their operands are and where the sums go.
#pragma once

#include "f64tc.cuh"
#include "tc_ptx.cuh"

namespace gbs {
namespace f64tc {

constexpr int kStageBytes = kAStage + kBStage;
constexpr int kStages = 5;    // 210 KB of the 227 KB
constexpr int kBurst = 4;     // stages per sub-tile turn
constexpr int kChunkKB = 8;   // K blocks (of 16) per exact accumulation: 128 modes
constexpr int kEpiWarps = 8;  // 4 lane quarters x 2 sub-tiles
constexpr int kThreads = 64 + 32 * kEpiWarps;  // warp 0 loads, warp 1 issues the products
constexpr int kBarBytes = 256;
constexpr int kPipeBytes = 1024 + kStages * kStageBytes + kBarBytes;  // (the base is aligned to 1024)
static_assert(kChunkKB == 2 * kBurst, "a chunk is two turns of each sub-tile");

// K-major operand without swizzle: core matrices of 8 rows x 16 bytes; the
// two of a 16-wide K step 128 bytes apart (leading offset), 8-row groups 256
// bytes apart (stride offset); descriptor version 1 (bit 46).
__device__ __forceinline__ uint64_t desc_k_plain(uint32_t saddr) {
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | (uint64_t)(128u >> 4) << 16 |
           (uint64_t)(256u >> 4) << 32 | (uint64_t)1u << 46;
}

// (hi 2^32 + lo) 2^e as a double, rounded to nearest (integer instructions:
// the FP64 pipe converts at 2 lanes per clock).
__device__ __forceinline__ double fixed_to_double(int64_t hi, int64_t lo, int e) {
    hi += lo >> 32;
    uint32_t l = (uint32_t)lo;
    const bool neg = hi < 0;
    uint64_t h = (uint64_t)hi;
    if (neg) {
        l = 0u - l;
        h = ~h + (l == 0u ? 1u : 0u);
    }
    if (h == 0) {
        if (l == 0u) return 0.0;
        h = l;
        l = 0u;
        e -= 32;
    }
    const int s = __clzll((long long)h);
    const uint64_t m = (h << s) | ((((uint64_t)l << 32) >> 1) >> (63 - s));
    const uint64_t r = (m >> 11) + ((m >> 10) & 1u);  // 53 bits, the top one set
    // m 2^(e + 32 - s): its leading bit weighs 2^(63 + 32 - s + e)
    const int64_t expo = (int64_t)(63 + 32 - s + e + 1023 - 1);
    const int64_t bits = (expo << 52) + (int64_t)r;
    return __longlong_as_double(bits | (neg ? (int64_t)0x8000000000000000ull : 0));
}

// One contraction of a CTA: stages at a + kb sa and b + kb sb, kb = 0..KB - 1.
struct Contraction {
    const uint8_t *a, *b;
    size_t sa, sb;
    int KB;
};

// Shared memory: the stages, the barriers, then what the caller wants.  Kept as
// one 32-bit address: the epilogue has no registers to spare.
struct Pipe {
    uint32_t base;

    __device__ __forceinline__ explicit Pipe(const uint8_t *raw) : base((ptx::smem_u32(raw) + 1023u) & ~1023u) {}
    // the generic address of what lies behind the barriers
    __device__ __forceinline__ uint8_t *rest(uint8_t *raw) const {
        return raw + (base - ptx::smem_u32(raw)) + kStages * kStageBytes + kBarBytes;
    }
    __device__ __forceinline__ uint32_t bar(int i) const {
        return base + (uint32_t)(kStages * kStageBytes + 8 * i);
    }
    __device__ __forceinline__ uint32_t full(int s) const { return bar(s); }
    __device__ __forceinline__ uint32_t empty(int s) const { return bar(kStages + s); }
    __device__ __forceinline__ uint32_t tfull(int sub) const { return bar(2 * kStages + sub); }
    __device__ __forceinline__ uint32_t tempty(int sub) const { return bar(2 * kStages + 2 + sub); }
    __device__ __forceinline__ uint32_t drain() const { return bar(2 * kStages + 4); }
    __device__ __forceinline__ uint32_t never() const { return bar(2 * kStages + 5); }
    __device__ __forceinline__ uint32_t tmem_slot() const { return bar(2 * kStages + 6); }

    // Barriers and TMEM; all threads; returns the TMEM base.
    __device__ __forceinline__ uint32_t open() {
        if (threadIdx.x == 0) {
            for (int s = 0; s < kStages; ++s) {
                ptx::mbar_init(full(s), 1);
                ptx::mbar_init(empty(s), 1);
            }
            for (int b = 0; b < 2; ++b) {
                ptx::mbar_init(tfull(b), 1);
                ptx::mbar_init(tempty(b), kEpiWarps / 2);
            }
            ptx::mbar_init(drain(), 1);
            ptx::mbar_init(never(), 1);  // nothing arrives on it
            ptx::fence_barrier_init();
        }
        if (threadIdx.x >> 5 == 1) {
            ptx::tmem_alloc<1>(tmem_slot(), 512);
            ptx::tmem_relinquish<1>();
        }
        ptx::tc_fence_before();
        __syncthreads();
        ptx::tc_fence_after();
        uint32_t tmem;
        asm volatile("ld.shared.b32 %0, [%1];" : "=r"(tmem) : "r"(tmem_slot()));
        return tmem;
    }

    __device__ __forceinline__ void close(uint32_t tmem) {
        ptx::tc_fence_before();
        __syncthreads();
        ptx::tc_fence_after();
        if (threadIdx.x >> 5 == 1) ptx::tmem_dealloc<1>(tmem, 512);
    }

    // Waits are bounded by wait_ns (the network's, gbs_set_wait_limit); one that
    // gives up raises *err and every role stops waiting.
    // One thread: the stages of contractions job(0, c), job(1, c), .. (false: no
    // more).
    template <typename Job>
    __device__ __forceinline__ void load(const Job &job, volatile unsigned long long *err,
                                         uint64_t wait_ns) const {
        int stage = 0;
        uint32_t phase = 0, used = 0, last = 0;
        bool ok = true;
        Contraction c;
        for (int i = 0; ok && job(i, c); ++i) {
            for (int kb = 0; kb < c.KB; ++kb) {
                if (!ptx::mbar_wait(empty(stage), phase ^ 1u, err, wait_ns)) {
                    ok = false;
                    break;
                }
                const uint32_t fb = full(stage);
                const uint32_t s = base + (uint32_t)(stage * kStageBytes);
                ptx::mbar_arrive_expect_tx(fb, kStageBytes);
                ptx::bulk_load(s, c.a + (size_t)kb * c.sa, kAStage, fb);
                ptx::bulk_load(s + kAStage, c.b + (size_t)kb * c.sb, kBStage, fb);
                used |= 1u << stage;
                last = (last & ~(1u << stage)) | (phase << stage);
                if (++stage == kStages) {
                    stage = 0;
                    phase ^= 1u;
                }
            }
        }
        // every load issued here has landed before the CTA exits
        for (int s = 0; s < kStages; ++s)
            if (used & (1u << s))
                ptx::mbar_wait(full(s), (last >> s) & 1u, err, 200000000ull,
                               false);
    }

    // One thread: their products, chunk by chunk (kChunkKB stages) into the two
    // sub-tiles' accumulators.
    template <typename Job>
    __device__ __forceinline__ void multiply(const Job &job, uint32_t tmem,
                                             volatile unsigned long long *err,
                                             uint64_t wait_ns) const {
            int base = 0;         // ring stage of the turn's first K block
            uint32_t base_ph = 0; // its phase
            uint32_t ck = 0;      // chunks issued so far
            bool ok = true;
            // a wait limit of 0 asks for the timeout path itself: the first wait
            // gives up (raising the flag) before any product is issued
            if (wait_ns == 0ull) ok = ptx::mbar_wait(never(), 0u, err, 0ull);
            Contraction c;
            for (int i = 0; ok && job(i, c); ++i) {
                const int KB = c.KB;
                for (int kb0 = 0; ok && kb0 < KB; kb0 += kBurst) {
                    const int nb = min(kBurst, KB - kb0);
                    const bool first = kb0 % kChunkKB == 0;
                    const bool end = !first || kb0 + nb >= KB;  // the chunk's last turn
                    for (int sub = 0; ok && sub < 2; ++sub) {
                        if (first) {
                            // the epilogue has read the sub-tile's previous chunk
                            if (!ptx::mbar_wait(tempty(sub), (ck & 1u) ^ 1u, err,
                                                wait_ns)) {
                                ok = false;
                                break;
                            }
                            ptx::tc_fence_after();
                        }
                        int stage = base;
                        uint32_t ph = base_ph;
                        for (int q = 0; q < nb; ++q) {
                            if (sub == 0) {
                                if (!ptx::mbar_wait(full(stage), ph, err, wait_ns)) {
                                    ok = false;
                                    break;
                                }
                                ptx::tc_fence_after();
                            }
                            const uint32_t s = this->base + (uint32_t)(stage * kStageBytes);
                            const uint64_t da = desc_k_plain(s);
                            const uint64_t db =
                                desc_k_plain(s + kAStage + sub * kBSub);
                            const uint32_t d = tmem + (uint32_t)sub * 256u;
                            const uint32_t acc = (first && q == 0) ? 0u : 1u;
                            // digit p of A against digits 0..min(6, 7 - p) of B; the
                            // long products last, so that the pipe has work while
                            // the next stage's barrier is polled
                            if (acc) {
#pragma unroll
                                for (int p = kDigits - 1; p >= 1; --p)
                                    ptx::mma_bf16(d + 32u * p, da + ((p * kASlice) >> 4), db,
                                                  ptx::idesc_f16_f32(128, 32 * (8 - p)), 1u);
                                ptx::mma_bf16(d, da, db, ptx::idesc_f16_f32(128, 224), 1u);
                            } else {  // d = 0..6 are new with digit 0, d = 7 with digit 1
                                ptx::mma_bf16(d, da, db, ptx::idesc_f16_f32(128, 224), 0u);
                                ptx::mma_bf16(d + 32u, da + (kASlice >> 4), db,
                                              ptx::idesc_f16_f32(128, 192), 1u);
                                ptx::mma_bf16(d + 224u, da + (kASlice >> 4),
                                              db + ((6 * kBSlice) >> 4),
                                              ptx::idesc_f16_f32(128, 32), 0u);
#pragma unroll
                                for (int p = kDigits - 1; p >= 2; --p)
                                    ptx::mma_bf16(d + 32u * p, da + ((p * kASlice) >> 4), db,
                                                  ptx::idesc_f16_f32(128, 32 * (8 - p)), 1u);
                            }
                            if (sub == 1) ptx::mma_commit(empty(stage));
                            if (++stage == kStages) {
                                stage = 0;
                                ph ^= 1u;
                            }
                        }
                        if (!ok) break;
                        if (end) ptx::mma_commit(tfull(sub));
                        if (sub == 1) {
                            base = stage;
                            base_ph = ph;
                        }
                    }
                    if (end) ++ck;
                }
            }
            ptx::mma_commit(drain());
            ptx::mbar_wait(drain(), 0u, err, 200000000ull, false);
    }

    // The four epilogue warps of sub-tile `sub`: chunk number ck of the CTA added
    // to the 64-bit sums hi = sum_{d < 4} D_d 2^{8 (3 - d)}, lo = sum_{d >= 4} D_d
    // 2^{8 (7 - d)} of this thread's row and the sub-tile's 32 columns; tb is the
    // sub-tile's TMEM address with the warp's lanes.
    __device__ __forceinline__ void add_chunk(uint32_t ck, int sub, uint32_t tb, int64_t (&hi)[32],
                                              int64_t (&lo)[32], volatile unsigned long long *err,
                                              uint64_t wait_ns) const {
        const int lane = threadIdx.x & 31;
        // on a timeout the epilogue keeps going without waiting
        ptx::mbar_wait(tfull(sub), ck & 1u, err, wait_ns);
        // the loads below are the whole warp's: lanes may come here apart, from the
        // wait or from what a caller does for some rows only
        __syncwarp();
        ptx::tc_fence_after();
        // 8 columns at a time: the sums hold 128 registers.  The other sub-tile's
        // turns (kBurst stages each, 2176 clocks) run meanwhile, but do not cover this
        // entirely: the conversions' 16 lanes per clock take 2048 for eight sums, so
        // D_0 and D_1, which are below 2^22, get theirs from an addition of 1.5 2^23,
        // and D_0 2^8 + D_1 and D_2 2^8 + D_3 (below 2^31) share a 64-bit addition.
#pragma unroll
        for (int c0 = 0; c0 < 32; c0 += 8) {
            float u[8], v[8];
            ptx::tmem_ld8(tb + (uint32_t)c0, u);
            ptx::tmem_ld8(tb + (uint32_t)(32 + c0), v);
            ptx::tmem_ld_wait();
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const uint32_t x = __float_as_uint(u[c] + 12582912.0f) * 256u +
                                   __float_as_uint(v[c] + 12582912.0f) - 0x4B400000u * 257u;
                hi[c0 + c] += (int64_t)(int)x * 65536;
            }
            ptx::tmem_ld8(tb + (uint32_t)(64 + c0), u);
            ptx::tmem_ld8(tb + (uint32_t)(96 + c0), v);
            ptx::tmem_ld_wait();
#pragma unroll
            for (int c = 0; c < 8; ++c) hi[c0 + c] += __float2int_rn(u[c]) * 256 + __float2int_rn(v[c]);
#pragma unroll
            for (int d = 4; d < 8; d += 2) {
                ptx::tmem_ld8(tb + (uint32_t)(32 * d + c0), u);
                ptx::tmem_ld8(tb + (uint32_t)(32 * d + 32 + c0), v);
                ptx::tmem_ld_wait();
                if (d == 6 && c0 == 24) {
                    ptx::tc_fence_before();
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(tempty(sub));
                }
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    lo[c0 + c] += (int64_t)__float2int_rn(u[c]) * (1 << (d == 4 ? 24 : 8)) +
                                  (int64_t)__float2int_rn(v[c]) * (1 << (d == 4 ? 16 : 0));
            }
        }
    }
};

}  // namespace f64tc
}  // namespace gbs
