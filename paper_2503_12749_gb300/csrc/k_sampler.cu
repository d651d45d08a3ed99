// K1: phase-space input sampler.
//
// Squeezed-vacuum inputs ("Applications to GBS"): per mode the +P density
// xi(alpha) xi(beta) e^{alpha beta} on the real plane is a bivariate Gaussian
// with covariance [[sinh r cosh r, sinh^2 r], [sinh^2 r, sinh r cosh r]],
// whose eigen-decomposition gives
//   alpha = sqrt(s+/2) w1 + sqrt(s-/2) w2,  beta = sqrt(s+/2) w1 - sqrt(s-/2) w2,
//   s+- = sinh(r) e^{+-r},  w1, w2 independent standard normals.
// The normals of trajectory e, input mode j come from one Philox-4x32-10 call
// (Salmon et al., SC'11) at counter (e_lo, e_hi, j, 0) with key (seed_lo,
// seed_hi): two 53-bit uniforms, then Box-Muller.  The same draws feed the
// matrix-P and +P estimators (both use the +P sampling procedure).
//
// Layouts written:
//   FP64 path: digit tiles (f64tc.cuh), or, for the networks the tensor cores do
//   not take, B[e][c][N] doubles, c = 0 (alpha), 1 (beta); FP32 path: FP32 tiles.
//   BF16 path: per 128-trajectory tile, 256 rows (128 alpha rows, then 128
//   beta rows); planes B0 = bf16(x), B1 = bf16(x - B0), B2 = bf16(x - B0 -
//   B1) stored plane-major, each plane K-blocked [ldK / 32][rows][32]
//   (mode j of row q at ((j / 32) * rows + q) * 32 + j % 32).
// Both also write n_e = sum_j alpha_j beta_j (FP64 result).  The BF16 path's
// device code (sampler_dev.cuh) also runs in the spare warps of the
// 3-product GEMM, which sample the next chunk.
#include "gbs_internal.cuh"
#include "f64tc.cuh"
#include "normal_f64.cuh"
#include "sampler_dev.cuh"

#include <algorithm>

namespace gbs {
namespace {

// Both amplitudes of (trajectory e, input mode j).
__device__ __forceinline__ void amplitudes(const NormTab &T, uint64_t seed, uint64_t e, uint32_t j,
                                           double2 q, double &a, double &b) {
    uint32_t c0 = (uint32_t)e, c1 = (uint32_t)(e >> 32), c2 = j, c3 = 0u;
    samp::philox4x32_10(c0, c1, c2, c3, (uint32_t)seed, (uint32_t)(seed >> 32));
    double w1, w2;
    nrm::normals(c0, c1, c2, c3, T, w1, w2);
    const double t = q.y * w2;
    a = fma(q.x, w1, t);
    b = fma(q.x, w1, -t);
}

// The tables in shared memory (lanes read them at unrelated indexes).
__device__ __forceinline__ void load_tab(NormTab &sh, const NormTab *__restrict__ tab) {
    static_assert(sizeof(NormTab) % 16 == 0, "table copied in 16-byte words");
    const uint4 *src = reinterpret_cast<const uint4 *>(tab);
    uint4 *dst = reinterpret_cast<uint4 *>(&sh);
    for (int t = threadIdx.x; t < (int)(sizeof(NormTab) / 16); t += blockDim.x) dst[t] = src[t];
    __syncthreads();
}

// ---------------------------------------------------------------------------
// FP64 path: one warp per trajectory, lanes stride over input modes.
// ---------------------------------------------------------------------------
__global__ void k_sample_fp64(const double2 *__restrict__ sq, const NormTab *__restrict__ tab, int N,
                              uint64_t seed, uint64_t e0, int64_t count, double *__restrict__ B,
                              double *__restrict__ n_out) {
    __shared__ __align__(16) NormTab sh;
    load_tab(sh, tab);
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = warp; i < count; i += nwarps) {
        const uint64_t e = e0 + (uint64_t)i;
        double *row_a = B + (size_t)i * 2 * N;
        double *row_b = row_a + N;
        double part = 0.0;
        for (int j = lane; j < N; j += 32) {
            double a, b;
            amplitudes(sh, seed, e, (uint32_t)j, sq[j], a, b);
            row_a[j] = a;
            row_b[j] = b;
            part += a * b;
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(0xffffffffu, part, off);
        if (lane == 0) n_out[i] = part;
    }
}

// ---------------------------------------------------------------------------
// FP32 path: the FP64 samples rounded to FP32 tiles [64 trajectories][K block]
// [16 k][64 alpha, 64 beta] (k_gemm_fp32.cu).  A block holds 32 trajectories, a
// lane each, and its 8 warps take every eighth mode (128-byte stores).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
    k_sample_fp32(const double2 *__restrict__ sq, const NormTab *__restrict__ tab, int N, int KB,
                  uint64_t seed, uint64_t e0, int64_t count, float *__restrict__ B,
                  double *__restrict__ n_out) {
    __shared__ __align__(16) NormTab sh;
    __shared__ double s_n[8][32];
    load_tab(sh, tab);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int kRow = 2 * kFp32TileSamples;
    for (int64_t i0 = (int64_t)blockIdx.x * 32; i0 < count; i0 += (int64_t)gridDim.x * 32) {
        const int64_t i = i0 + lane;
        float *tile =
            B + (size_t)(i / kFp32TileSamples) * KB * kFp32BlockK * kRow + i % kFp32TileSamples;
        double p[4] = {0.0, 0.0, 0.0, 0.0};  // 32 chains of N / 32 terms, joined pairwise
        if (i < count)
            for (int j = warp; j < KB * kFp32BlockK; j += 8) {
                double a = 0.0, b = 0.0;
                if (j < N) {
                    amplitudes(sh, seed, e0 + (uint64_t)i, (uint32_t)j, sq[j], a, b);
                    const double s = fma(a, b, p[0]);
                    p[0] = p[1];
                    p[1] = p[2];
                    p[2] = p[3];
                    p[3] = s;
                }
                tile[(size_t)j * kRow] = (float)a;
                tile[(size_t)j * kRow + kFp32TileSamples] = (float)b;
            }
        s_n[warp][lane] = (p[0] + p[1]) + (p[2] + p[3]);
        __syncthreads();
        if (warp == 0 && i < count) {
            double v[4];
#pragma unroll
            for (int w = 0; w < 4; ++w) v[w] = s_n[2 * w][lane] + s_n[2 * w + 1][lane];
            n_out[i] = (v[0] + v[1]) + (v[2] + v[3]);
        }
        __syncthreads();
    }
}

// a + b rounded, its rounding error added to err (TwoSum; Knuth, "The Art of
// Computer Programming" 2, 4.2.2).
__device__ __forceinline__ double two_sum(double a, double b, double &err) {
    const double s = a + b, bb = s - a;
    err += (a - (s - bb)) + (b - bb);
    return s;
}

// ---------------------------------------------------------------------------
// FP64 path on the tensor cores: the digit tiles of f64tc.cuh.  `wpg` of a
// block's 8 warps (1, 2, 4 or 8, by the number of modes) hold 8 trajectories (one
// core matrix); a warp takes 4 groups of 8 consecutive modes per pass, a lane one
// group of one trajectory: it stores 16 bytes per digit, the 8 lanes of a group
// one 128-byte core matrix.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256, 2)
    k_sample_f64tc(const double2 *__restrict__ sq, const NormTab *__restrict__ tab,
                   const int *__restrict__ col_exp, int N, int KB, int wpg, uint64_t seed,
                   uint64_t e0, int64_t count, uint8_t *__restrict__ B, double *__restrict__ n_out) {
    using namespace f64tc;
    __shared__ __align__(16) NormTab sh;
    __shared__ double s_n[8][8], s_err[8][8];
    load_tab(sh, tab);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int per = 8 / wpg * 8;  // trajectories per block and turn
    for (int64_t i0 = (int64_t)blockIdx.x * per; i0 < count; i0 += (int64_t)gridDim.x * per) {
        const int64_t i = i0 + warp / wpg * 8 + (lane & 7);
        const uint64_t e = e0 + (uint64_t)i;
        const int row = (int)(i & 15);
        uint8_t *tile = B + (size_t)(i / kTrajTile) * KB * kBStage + ((i >> 4) & 1) * kBSub;
        double sum[4] = {0.0, 0.0, 0.0, 0.0};  // chains of two modes of eight each
        if (i < count)
            for (int oct = (warp & (wpg - 1)) * 4 + (lane >> 3); oct < 2 * KB; oct += 4 * wpg) {
                uint32_t da[kDigits][4], db[kDigits][4];
#pragma unroll
                for (int t = 0; t < 8; t += 2) {
                    int64_t xa[2] = {0, 0}, xb[2] = {0, 0};
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int j = oct * 8 + t + h;
                        if (j < N) {
                            double a, b;
                            amplitudes(sh, seed, e, (uint32_t)j, sq[j], a, b);
                            sum[t >> 1] = fma(a, b, sum[t >> 1]);
                            const int s = 55 + kTrajBits - col_exp[j];
                            xa[h] = to_fixed(a, s);
                            xb[h] = to_fixed(b, s);
                        }
                    }
                    uint32_t w[kDigits];
                    digit_pairs<true>(xa[0], xa[1], w);
#pragma unroll
                    for (int q = 0; q < kDigits; ++q) da[q][t >> 1] = w[q];
                    digit_pairs<true>(xb[0], xb[1], w);
#pragma unroll
                    for (int q = 0; q < kDigits; ++q) db[q][t >> 1] = w[q];
                }
                uint8_t *p = tile + (size_t)(oct >> 1) * kBStage;
                const int k = (oct & 1) * 8;
#pragma unroll
                for (int q = 0; q < kDigits; ++q) {
                    *reinterpret_cast<uint4 *>(p + q * kBSlice + core_offset(row, k)) =
                        make_uint4(da[q][0], da[q][1], da[q][2], da[q][3]);
                    *reinterpret_cast<uint4 *>(p + q * kBSlice + core_offset(16 + row, k)) =
                        make_uint4(db[q][0], db[q][1], db[q][2], db[q][3]);
                }
            }
        // the last additions with their rounding errors, rounded once: they err the most
        // of a pairwise sum, and an unequal last part adds one (N = 130: 8.5e-17 of sum
        // |alpha beta| without, 7.4e-17 for 32 interleaved chains, 6.3e-17 so).  Where
        // warps follow, theirs are enough, and the lanes' cost 0.5 % of a call at N = 1000.
        double part = (sum[0] + sum[1]) + (sum[2] + sum[3]), err = 0.0;
        if (wpg <= 2) {
            part = two_sum(part, __shfl_xor_sync(0xffffffffu, part, 8), err);
            err += __shfl_xor_sync(0xffffffffu, err, 16);
            part = two_sum(part, __shfl_xor_sync(0xffffffffu, part, 16), err);
        } else {
            part += __shfl_xor_sync(0xffffffffu, part, 8);
            part += __shfl_xor_sync(0xffffffffu, part, 16);
        }
        if (lane < 8) {
            s_n[warp][lane] = part;
            s_err[warp][lane] = err;
        }
        __syncthreads();
        if ((warp & (wpg - 1)) == 0 && lane < 8 && i < count) {
            for (int w = 1; w < wpg; ++w) {
                err += s_err[warp + w][lane];
                part = two_sum(part, s_n[warp + w][lane], err);
            }
            n_out[i] = part + err;
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// BF16 split path: FP32 arithmetic; each lane handles 4 consecutive modes.
// ---------------------------------------------------------------------------
template <bool kSfu>
__global__ void k_sample_bf16(const SampleJob job) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    samp::sample_warps_bf16<kSfu, false>(job, warp, nwarps, lane);
}

int grid_for_warps(gbs_net *net, int64_t warps_needed, int threads) {
    const int64_t per_block = threads / 32;
    int64_t blocks = (warps_needed + per_block - 1) / per_block;
    const int64_t cap = (int64_t)net->sm_count * 16;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    return (int)blocks;
}

}  // namespace

int launch_sample_fp64(gbs_net *net, uint64_t seed, uint64_t e0, int64_t count) {
    net->pre_valid = false;  // the operands are overwritten
    if (count <= 0) return GBS_OK;
    if (net->d_Aq) {
        // modes in groups of 8, 4 groups per warp and pass
        const int KB = f64tc_kblocks(net->N);
        int wpg = 1;
        while (wpg < 8 && wpg * 4 < 2 * KB) wpg *= 2;
        const int64_t blocks = (count + 64 / wpg - 1) / (64 / wpg);
        k_sample_f64tc<<<(unsigned)std::min<int64_t>(blocks, 2 * (int64_t)net->sm_count), 256, 0,
                         net->stream>>>(net->d_sq64, net->d_ntab, net->d_colexp, net->N, KB, wpg,
                                        seed, e0, count, static_cast<uint8_t *>(net->d_B), net->d_n);
    } else if (net->d_T32) {
        k_sample_fp32<<<(unsigned)std::min<int64_t>((count + 31) / 32, 8 * (int64_t)net->sm_count), 256,
                        0, net->stream>>>(net->d_sq64, net->d_ntab, net->N,
                                          (net->N + kFp32BlockK - 1) / kFp32BlockK, seed, e0, count,
                                          static_cast<float *>(net->d_B), net->d_n);
    } else {
        k_sample_fp64<<<grid_for_warps(net, count, 256), 256, 0, net->stream>>>(
            net->d_sq64, net->d_ntab, net->N, seed, e0, count, static_cast<double *>(net->d_B),
            net->d_n);
    }
    GBS_LAUNCH_CHECK();
    return GBS_OK;
}

const NormTab *norm_tab() {
    static const NormTab T = [] {
        NormTab t;
        fill_norm_tab(t);
        return t;
    }();
    return &T;
}

size_t norm_tab_bytes() { return sizeof(NormTab); }

SampleJob sample_job_bf16(gbs_net *net, void *B, double *n, uint64_t seed, uint64_t e0,
                          int64_t count) {
    SampleJob j;
    const int64_t tiles = (net->chunk + kTcTileSamples - 1) / kTcTileSamples;
    j.sq = net->d_sq32;
    j.B = static_cast<__nv_bfloat16 *>(B);
    j.n_out = n;
    j.rows = (size_t)tiles * 256;
    j.plane_stride = j.rows * net->ldK;
    j.seed = seed;
    j.e0 = e0;
    j.count = count;
    j.N = net->N;
    j.ldK = net->ldK;
    j.planesB = net->planesB;
    return j;
}

int launch_sample_bf16(gbs_net *net, uint64_t seed, uint64_t e0, int64_t count) {
    net->pre_valid = false;  // the operands are overwritten
    if (count <= 0) return GBS_OK;
    const int threads = 256;
    const SampleJob job = sample_job_bf16(net, net->d_B, net->d_n, seed, e0, count);
    auto kern = net->planesB == 2 ? k_sample_bf16<true> : k_sample_bf16<false>;
    kern<<<grid_for_warps(net, count, threads), threads, 0, net->stream>>>(job);
    GBS_LAUNCH_CHECK();
    return GBS_OK;
}

}  // namespace gbs
