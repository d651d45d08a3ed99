// K2 + K3, FP32 path (GBS_FP32): the propagation GEMM with T and the samples
// rounded to FP32 and their products accumulated in FP32, one fused
// multiply-add after the other along the N input modes, then the FP64
// occupation epilogue n'_i = alpha'_i beta'_i (see k_gemm_fp64.cu).
//
// Bound by the FP32 pipe (152 SMs x 128 lanes x 2.07 GHz = 80.5 TFLOP/s).  Tile: 64
// output modes (128 rows Re/Im) x 64 trajectories (64 alpha, 64 beta columns)
// per 256-thread block, 8 x 8 accumulators per thread as packed FP32x2
// multiply-adds (round to nearest per element, half the instructions of scalar
// ones), so that a step of k reads 64 bytes of shared memory for 64
// multiply-adds; two blocks per SM, one block's FP64 epilogue beside the
// other's products.  Both operands are stored in FP32 as the shared-memory
// images of a stage ([16 k][128 rows]), so a stage is two bulk copies and the
// conversion from FP64 is done once, not once per tile.  Measured at 700 x 615,
// 20001 trajectories: 3.75 ms for the FP64 kernel's tiling with FP32 registers
// (64 x 32 tile, 4 x 2 modes by trajectories per thread, operands converted as
// they were staged) -> 1.09 ms (66 TFLOP/s over the padded tiles, 0.82 of the pipe).
#include "gbs_internal.cuh"
#include "tc_ptx.cuh"

#include <algorithm>

namespace gbs {
namespace {

constexpr int kTM = kFp64TileModes;           // 64 modes
constexpr int kTS = kFp32TileSamples;         // 64 trajectories
constexpr int kKT = kFp32BlockK;              // k per stage
constexpr int kStageFloats = kKT * 128;       // one operand's
constexpr int kStageBytes = 2 * kStageFloats * 4;
constexpr int kStages = 4;
constexpr int kSmemBytes = kStages * kStageBytes + 128;
static_assert(16 * kTS * 16 <= kStages * kStageBytes, "reduction buffer in the ring");

__device__ __forceinline__ void fma2(float2 &acc, float2 a, float2 b) {
    asm("{\n"
        ".reg .b64 x, y, z;\n"
        "mov.b64 x, {%0, %1};\n"
        "mov.b64 y, {%2, %3};\n"
        "mov.b64 z, {%4, %5};\n"
        "fma.rn.f32x2 x, y, z, x;\n"
        "mov.b64 {%0, %1}, x;\n"
        "}\n"
        : "+f"(acc.x), "+f"(acc.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
}

__global__ void __launch_bounds__(256, 2)
    k_gemm_fp32(const float *__restrict__ A, const float *__restrict__ B, int KB, int mtiles,
                int64_t count, int64_t ld_part, double2 *__restrict__ nS_part, OccOut64 occ,
                uint64_t wait_ns, unsigned long long *err_ptr) {
    extern __shared__ __align__(128) uint8_t smem[];
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + kStages * kStageBytes);
    uint64_t *empty = full + kStages;
    uint64_t *never = empty + kStages;
    volatile unsigned long long *err = err_ptr;
    const int tid = threadIdx.x, lane = tid & 31;
    const int tx = tid & 15;  // 4 trajectories
    const int ty = tid >> 4;  // 4 modes
    const int mt = blockIdx.x % mtiles;
    const int64_t st = blockIdx.x / mtiles;
    const float *a_src = A + (size_t)mt * KB * kStageFloats;
    const float *b_src = B + (size_t)st * KB * kStageFloats;
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            ptx::mbar_init(ptx::smem_u32(&full[s]), 1);
            ptx::mbar_init(ptx::smem_u32(&empty[s]), 8);  // one arrival per warp
        }
        ptx::mbar_init(ptx::smem_u32(never), 1);  // nothing arrives on it
        ptx::fence_barrier_init();
    }
    __syncthreads();
    auto load = [&](int kb) {  // thread 0
        const int s = kb % kStages;
        const uint32_t bar = ptx::smem_u32(&full[s]);
        const uint32_t dst = ptx::smem_u32(smem + s * kStageBytes);
        ptx::mbar_arrive_expect_tx(bar, kStageBytes);
        ptx::bulk_load(dst, a_src + (size_t)kb * kStageFloats, kStageBytes / 2, bar);
        ptx::bulk_load(dst + kStageBytes / 2, b_src + (size_t)kb * kStageFloats, kStageBytes / 2, bar);
    };
    int issued = min(KB, kStages);  // stages that thread 0 has loaded
    if (tid == 0)
        for (int kb = 0; kb < issued; ++kb) load(kb);

    float2 acc[8][4];  // [row][alpha pair 0, 1, beta pair 0, 1]
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = make_float2(0.0f, 0.0f);

    // A warp whose wait gives up (wait_ns; the network's flag is raised) takes no
    // further stage; its missing arrivals stop the loads.  With wait_ns = 0 the
    // first wait is on a barrier that nothing arrives on.
    bool ok = true;
    if (wait_ns == 0ull) ok = __all_sync(0xffffffffu, ptx::mbar_wait(ptx::smem_u32(never), 0u, err, 0ull));
    for (int kb = 0; ok && kb < KB; ++kb) {
        const int s = kb % kStages;
        const uint32_t ph = (uint32_t)(kb / kStages) & 1u;
        ok = __all_sync(0xffffffffu, ptx::mbar_wait(ptx::smem_u32(&full[s]), ph, err, wait_ns));
        if (!ok) break;
        const float *As = reinterpret_cast<const float *>(smem + s * kStageBytes) + ty * 8;
        const float *Bs = reinterpret_cast<const float *>(smem + s * kStageBytes) + kStageFloats + tx * 4;
#pragma unroll
        for (int k = 0; k < kKT; ++k) {
            const float4 a0 = *reinterpret_cast<const float4 *>(As + k * 128);
            const float4 a1 = *reinterpret_cast<const float4 *>(As + k * 128 + 4);
            const float4 b0 = *reinterpret_cast<const float4 *>(Bs + k * 128);
            const float4 b1 = *reinterpret_cast<const float4 *>(Bs + k * 128 + 64);
            const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const float2 b[4] = {make_float2(b0.x, b0.y), make_float2(b0.z, b0.w),
                                 make_float2(b1.x, b1.y), make_float2(b1.z, b1.w)};
#pragma unroll
            for (int r = 0; r < 8; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) fma2(acc[r][c], make_float2(a[r], a[r]), b[c]);
        }
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&empty[s]));
        // (a stage after one that was not loaded is not either: `issued` counts them)
        if (tid == 0 && kb + kStages < KB && issued == kb + kStages &&
            ptx::mbar_wait(ptx::smem_u32(&empty[s]), ph, err, wait_ns)) {
            load(kb + kStages);
            ++issued;
        }
        __syncwarp();
    }
    // the ring becomes the reduction buffer, and another block's memory when this
    // one exits: every load issued here has landed first, given up or not
    if (tid == 0)
        for (int kb = max(0, issued - kStages); kb < issued; ++kb)
            ptx::mbar_wait(ptx::smem_u32(&full[kb % kStages]), (uint32_t)(kb / kStages) & 1u, err,
                           200000000ull, false);
    __syncthreads();  // and every warp has left it

    // occupations of this thread's 4 modes x 4 trajectories
    double2 *red = reinterpret_cast<double2 *>(smem);  // [16][kTS]
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        double re = 0.0, im = 0.0;
        const int64_t traj = st * kTS + tx * 4 + t;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const float2 *x = acc[2 * m], *y = acc[2 * m + 1];
            const double ar = (t & 1) ? x[t >> 1].y : x[t >> 1].x;
            const double ai = (t & 1) ? y[t >> 1].y : y[t >> 1].x;
            const double br = (t & 1) ? x[2 + (t >> 1)].y : x[2 + (t >> 1)].x;
            const double bi = (t & 1) ? y[2 + (t >> 1)].y : y[2 + (t >> 1)].x;
            if (occ.p && traj < count) {
                double *dst = occ.p + (size_t)(mt * kTM + ty * 4 + m) * occ.ld + traj;
                dst[0] = ar * br + ai * bi;
                dst[occ.plane] = ai * br - ar * bi;
            }
            re = fma(ai, bi, fma(ar, br, re));
            im = fma(-ar, bi, fma(ai, br, im));
        }
        red[ty * kTS + tx * 4 + t] = make_double2(re, im);
    }
    __syncthreads();
    if (tid < kTS) {
        double re = 0.0, im = 0.0;
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            re += red[q * kTS + tid].x;
            im += red[q * kTS + tid].y;
        }
        const int64_t traj = st * kTS + tid;
        if (traj < count) nS_part[(size_t)mt * ld_part + traj] = make_double2(re, im);
    }
}

// T64 [M][2][N] -> FP32 tiles [mode tile][K block][16 k][128 rows], zero padded.
__global__ void k_t32_tiles(const double *__restrict__ T64, int N, int M, int KB,
                            float *__restrict__ A) {
    const int mt = blockIdx.y, kb = blockIdx.x;
    float *dst = A + ((size_t)mt * KB + kb) * kStageFloats;
    for (int t = threadIdx.x; t < kStageFloats; t += blockDim.x) {
        const int row = t >> 4, k = t & 15;  // reads of 16 consecutive k
        const int i = mt * kTM + (row >> 1), j = kb * kKT + k;
        dst[k * 128 + row] = i < M && j < N ? (float)T64[((size_t)i * 2 + (row & 1)) * N + j] : 0.0f;
    }
}

}  // namespace

size_t fp32_A_floats(int N, int mtiles) {
    return (size_t)mtiles * ((N + kKT - 1) / kKT) * kStageFloats;
}

size_t fp32_B_bytes(int N, int64_t chunk) {
    return (size_t)((chunk + kTS - 1) / kTS) * ((N + kKT - 1) / kKT) * kStageFloats * sizeof(float);
}

int launch_t32_tiles(gbs_net *net) {
    GBS_CUDA_TRY(cudaFuncSetAttribute(k_gemm_fp32, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      kSmemBytes));
    const int KB = (net->N + kKT - 1) / kKT;
    k_t32_tiles<<<dim3((unsigned)KB, (unsigned)net->mtiles), 256, 0, net->stream>>>(
        net->d_T64, net->N, net->M, KB, net->d_T32);
    GBS_LAUNCH_CHECK();
    return GBS_OK;
}

int launch_gemm_fp32(gbs_net *net, int64_t count, OccOut64 occ) {
    const int64_t blocks = (count + kTS - 1) / kTS * net->mtiles;
    if (blocks > 0x7fffffff) return set_error(GBS_EINVAL, "chunk too large");
    k_gemm_fp32<<<(unsigned)blocks, 256, kSmemBytes, net->stream>>>(
        net->d_T32, static_cast<const float *>(net->d_B), (net->N + kKT - 1) / kKT, net->mtiles,
        count, net->chunk, net->d_nS_part, occ, net->wait_ns, net->d_flags + 1);
    GBS_LAUNCH_CHECK();
    return GBS_OK;
}

}  // namespace gbs
