// K2 + K3, FP64 path on the tensor cores: propagation alpha' = T alpha,
// beta' = T* beta ("Applications to GBS") as an exact integer contraction,
// fused with the FP64 occupation epilogue n'_i = alpha'_i beta'_i.
//
// Both operands are written as fixed-point numbers of seven balanced 8-bit
// digits and the digit products are contracted without rounding on the FP16
// tensor cores (the error-free splitting of Ozaki, Ogita, Oishi, Rump,
// "Error-free transformations of matrix multiplication by using fast routines
// of matrix multiplication and its applications", Numer. Algorithms 59, 2012,
// in its fixed-point form):
//   T_ij 2^{e_j - f_i} = 2^-55 sum_{p=0..6} a_p 2^{8 (6 - p)},   |a_p| <= 128,
//   alpha_j 2^{-e_j}   = 2^-58 sum_{q=0..6} b_q 2^{8 (6 - q)},   |b_q| <= 128, |b_0| <= 1024,
//   D_d = sum_j sum_{p + q = d} a_p b_q   (d = 0..7),
//   alpha'_i = 2^{f_i - 73} sum_d D_d 2^{8 (7 - d)}.
// e_j bounds |alpha_j|, |beta_j| for every possible draw (the Box-Muller
// radius of a 53-bit uniform is below 8.67), f_i bounds row i of T 2^{e_j}.
// A digit is an integer of at most 11 bits, so it is an FP16 number, and every FP32
// accumulator value is an exact integer below 2^24 over 128 input modes (one
// chunk): the products without b_0, d (of D_7: 6) of at most 2^21 per D_d, by their
// bound; the one with it, a_d b_0 summed, because b_0 is Gaussian of standard
// deviation below 118.2 (2^10 / 8.67), so that the sum over 128 modes has at most
// 2^17.4 whatever T is and exceeds the 2^21 that D_1 leaves (the drain wants D_0 and
// D_1 below 2^22) by 12.3 standard deviations, the 2^22 of the others by 24:
// less than once in 1e33 sums.
// The accumulators are added to 64-bit integers every 128 modes, so the only
// errors are the quantisation of the operands (amplitudes above 1/32 of their
// scale and entries of T above 1/8 of their row's largest are exact, smaller ones
// err by 2^-59 and 2^-56 of it), the digit pairs p + q >= 8 (below 2^-64) and
// the sum's rounding to 53 bits, against a rounding at every term of a chain of
// FP64 FMAs.  So it is the more accurate one however few entries a row of T has;
// kTrajBits = 0 was not (the figures in parentheses below).
//
// Why: GB300 has 2 FP64 FMA lanes per SM and clock (1.25 TFLOP/s) but 4096
// 16-bit ones, so 34 exact 16-bit products cost a fiftieth of one FP64 product.
// Measured (one GB300): N = M = 1000, 32768 trajectories 5.50 ms against 216.4
// for the FP64 FMA kernel (34 products at 0.84 of the measured BF16 rate; 6.27 with
// a conversion for every sum and 32 columns read at once, f64tc_pipe.cuh);
// N = M = 16, 16384 trajectories 0.043 against 0.149.  Root mean square error of
// n_S against 113-bit arithmetic, relative to sum |alpha'_i| |beta'_i|, real and
// imaginary part (the input samples' own rounding included): N = 16 9.8e-17 and
// 2.2e-17 against 1.18e-16 and 4.0e-17, N = 64 7.6e-17 and 1.3e-17 against 1.09e-16
// and 3.8e-17, N = 200 8.6e-17 and 5.4e-18 against 1.17e-16 and 4.0e-17, N = 400
// 9.1e-17 and 4.4e-18 against 1.12e-16 and 3.7e-17.  Median relative error of an
// occupation n'_i, N = 32, likewise: diagonal T 2.09e-16 against 2.11e-16 (3.2e-16
// with kTrajBits = 0), blocks of 2 modes 1.90e-16 against 1.98e-16 (2.9e-16), of 4
// 1.93e-16 against 2.10e-16 (2.8e-16), dense 2.03e-16 against 3.08e-16 (2.8e-16).
//
// Tile: 64 output modes (128 rows Re/Im) x 32 trajectories, as two sub-tiles
// of 16 trajectories (16 alpha and 16 beta columns).  A sub-tile's eight D_d
// are 8 x 32 TMEM columns side by side, so that digit p of A times the stacked
// digits 0..min(6, 7 - p) of B is ONE instruction whose columns land on
// d = p..: 7 MMAs per 16 modes instead of 34.  Both sub-tiles fill the 512
// TMEM columns; the issuer works on them in turn, 4 stages each, so that one
// is drained while the other is multiplied.
//
// Operands are stored in global memory as the exact shared-memory images
// (no swizzle, 8 x 16-byte core matrices), so a stage is two plain bulk copies.
#include "gbs_internal.cuh"
#include "f64tc_pipe.cuh"

#include <algorithm>
#include <cmath>
#include <vector>

namespace gbs {
namespace {

using namespace f64tc;

constexpr int kRedBytes = 4 * 2 * 32 * 8;  // [quarter][sub-tile][16 re, 16 im]
constexpr int kSmemBytes = kPipeBytes + kRedBytes;
static_assert(kSmemBytes <= 227 * 1024, "shared memory of the FP64 tensor-core GEMM");
// mode tiles per band of the tile order: 8 mode tiles x 19 trajectory tiles
// make one wave of 152 CTAs, the most square split of its operand traffic
constexpr int kBand = 8;

struct Tile {
    int mt, st;
};
__device__ __forceinline__ Tile tile_of(int t, int mtiles, int stiles) {
    const int per = kBand * stiles;
    const int b = t / per, rem = t - b * per;
    const int bw = min(kBand, mtiles - b * kBand);
    Tile r;
    r.mt = b * kBand + rem % bw;
    r.st = rem / bw;
    return r;
}

// Sum over the 16 lanes of the same parity of 16 values per lane: lanes 2 q and
// 2 q + 1 return their parity's sum of value q, in a fixed order.
__device__ __forceinline__ double transpose_sum(double (&v)[16], int lane) {
#pragma unroll
    for (int w = 8; w >= 1; w >>= 1) {
        const bool up = (lane & (2 * w)) != 0;
#pragma unroll
        for (int i = 0; i < w; ++i) {
            const double send = up ? v[i] : v[i + w];
            const double keep = up ? v[i + w] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 2 * w);
        }
    }
    return v[0];
}

__global__ void __launch_bounds__(kThreads, 1)
    k_gemm_f64tc(const uint8_t *__restrict__ A, const uint8_t *__restrict__ B,
                 const int *__restrict__ row_exp, int KB, int mtiles, int stiles,
                 int64_t count, int64_t ld_part, double2 *__restrict__ nS_part, OccOut64 occ,
                 uint64_t wait_ns, unsigned long long *err_ptr) {
    extern __shared__ uint8_t smem_raw[];
    Pipe pipe(smem_raw);
    double *red = reinterpret_cast<double *>(pipe.rest(smem_raw));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile unsigned long long *err = err_ptr;
    const uint32_t tmem = pipe.open();
    const int ntiles = mtiles * stiles;
    const int nchunk = (KB + kChunkKB - 1) / kChunkKB;

    auto job = [&](int i, Contraction &c) {
        const int64_t t = blockIdx.x + (int64_t)i * gridDim.x;
        if (t >= ntiles) return false;
        const Tile tl = tile_of((int)t, mtiles, stiles);
        c = {A + (size_t)tl.mt * KB * kAStage, B + (size_t)tl.st * KB * kBStage, kAStage, kBStage, KB};
        return true;
    };

    if (warp == 0) {
        if (lane == 0) pipe.load(job, err, wait_ns);
    } else if (warp == 1) {
        if (lane == 0) pipe.multiply(job, tmem, err, wait_ns);
    } else {
        const int quarter = warp & 3;
        const int sub = (warp - 2) >> 2;
        const int row = quarter * 32 + lane;
        const uint32_t tb = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)sub * 256u;
        uint32_t ck = 0;
        for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
            const Tile tl = tile_of(t, mtiles, stiles);
            int64_t hi[32], lo[32];
#pragma unroll
            for (int c = 0; c < 32; ++c) hi[c] = lo[c] = 0;
            for (int k = 0; k < nchunk; ++k, ++ck) pipe.add_chunk(ck, sub, tb, hi, lo, err, wait_ns);
            // alpha' (columns 0..15) and beta' (16..31) of this row; the
            // partner lane holds the other of (Re, Im) of the same mode
            const int f = row_exp[tl.mt * 128 + row] - 70 - kTrajBits;
            const bool odd = (lane & 1) != 0;
            // even lanes (Re rows) form the real parts ar br + ai bi, odd lanes
            // the imaginary parts ai br - ar bi
            const int64_t e0 = (int64_t)tl.st * 32 + sub * 16;
            double v[16];
#pragma unroll
            for (int c = 0; c < 16; ++c) {
                const double a = fixed_to_double(hi[c], lo[c], f);
                const double b = fixed_to_double(hi[16 + c], lo[16 + c], f);
                const double pa = __shfl_xor_sync(0xffffffffu, a, 1);
                const double pb = __shfl_xor_sync(0xffffffffu, b, 1);
                v[c] = fma(a, odd ? pb : b, odd ? -(pa * b) : pa * pb);
            }
            if (occ.p) {
                const int mode = tl.mt * 64 + (row >> 1);
                double *dst = occ.p + (size_t)mode * occ.ld + (odd ? occ.plane : 0);
#pragma unroll
                for (int c = 0; c < 16; ++c)
                    if (e0 + c < count) dst[e0 + c] = v[c];
            }
            const double s = transpose_sum(v, lane);
            red[(quarter * 2 + sub) * 32 + (odd ? 16 : 0) + (lane >> 1)] = s;
            // the four lane quarters of this sub-tile
            asm volatile("bar.sync %0, 128;" ::"r"(1 + sub) : "memory");
            if (quarter == 0 && lane < 16) {
                double re = 0.0, im = 0.0;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    re += red[(q * 2 + sub) * 32 + lane];
                    im += red[(q * 2 + sub) * 32 + 16 + lane];
                }
                if (e0 + lane < count) nS_part[(size_t)tl.mt * ld_part + e0 + lane] = make_double2(re, im);
            }
            asm volatile("bar.sync %0, 128;" ::"r"(1 + sub) : "memory");
        }
    }
    pipe.close(tmem);
}

// One block per 8 rows (a row of core matrices) and 256 k of the padded operand: the
// rows' scales, a warp each, then the digits of 8 consecutive k of a row per thread,
// so that a digit's 8 rows are one 128-byte store.  bad counts the rows whose scale
// lies outside the range the digits are used for.  Bound by latency, so every load of
// a thread is in flight at once and the scales are formed again in each of a row's
// blocks: N = M = 1000 24 us; a row per block with 16-bit stores 43, loads one by one
// and FP64 comparisons 36.
constexpr int kSplitRows = 8;
// (integer instructions: an FP64 comparison takes 16 clocks of a warp)
__device__ __forceinline__ bool nonzero(double v) { return (__double_as_longlong(v) << 1) != 0; }
__device__ __forceinline__ int exponent_of(double v) {  // ilogb for v != 0
    const int e = (__double2hiint(v) >> 20) & 0x7ff;
    return e ? e - 1023 : ilogb(v);
}
__global__ void __launch_bounds__(32 * kSplitRows)
    k_f64tc_split_T(const double *__restrict__ T64, const int *__restrict__ col_exp, int N, int M,
                    int KB, uint8_t *__restrict__ A, int *__restrict__ row_exp,
                    unsigned long long *__restrict__ bad) {
    __shared__ int s_ex[kSplitRows];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int row0 = blockIdx.x * kSplitRows;
    {
        const int row = row0 + warp, i = row >> 1;
        const double *src = T64 + ((size_t)i * 2 + (row & 1)) * N;
        int ex = kExpNone;
        for (int j0 = lane; i < M && j0 < N; j0 += 256) {
            double v[8];
            int e[8];
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const int j = j0 + 32 * t;
                v[t] = j < N ? src[j] : 0.0;
                e[t] = j < N ? col_exp[j] : kExpVacuum;
            }
#pragma unroll
            for (int t = 0; t < 8; ++t)
                if (nonzero(v[t]) && e[t] != kExpVacuum) ex = max(ex, exponent_of(v[t]) + 1 + e[t]);
        }
        ex = __reduce_max_sync(0xffffffffu, ex);
        if (ex == kExpNone) ex = 0;
        if (lane == 0) s_ex[warp] = ex;
        if (lane == 0 && blockIdx.y == 0) {
            row_exp[row] = ex;
            if (ex < -kExpRange || ex > kExpRange) atomicAdd(bad, 1ull);
        }
    }
    __syncthreads();
    const int row = row0 + (threadIdx.x & (kSplitRows - 1)), i = row >> 1;
    const int ex = s_ex[threadIdx.x & (kSplitRows - 1)];
    const double *src = T64 + ((size_t)i * 2 + (row & 1)) * N;
    uint8_t *tile = A + (size_t)(row >> 7) * KB * kAStage;
    const int g = blockIdx.y * 32 + threadIdx.x / kSplitRows;  // group of 8 k
    if (g < 2 * KB) {
        double v[8];
        int e[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) {  // every load in flight at once
            const int j = 8 * g + t;
            const bool in = i < M && j < N;
            v[t] = in ? src[j] : 0.0;
            e[t] = in ? col_exp[j] : kExpVacuum;
        }
        uint32_t dg[kDigits][4];
#pragma unroll
        for (int t = 0; t < 8; t += 2) {
            int64_t x[2];
#pragma unroll
            for (int h = 0; h < 2; ++h)
                x[h] = nonzero(v[t + h]) && e[t + h] != kExpVacuum ? to_fixed(v[t + h], 55 + e[t + h] - ex) : 0;
            uint32_t d[kDigits];
            digit_pairs(x[0], x[1], d);
#pragma unroll
            for (int q = 0; q < kDigits; ++q) dg[q][t >> 1] = d[q];
        }
        uint8_t *p = tile + (size_t)(g >> 1) * kAStage + core_offset(row & 127, 8 * (g & 1));
#pragma unroll
        for (int q = 0; q < kDigits; ++q)
            *reinterpret_cast<uint4 *>(p + q * kASlice) = make_uint4(dg[q][0], dg[q][1], dg[q][2], dg[q][3]);
    }
}

}  // namespace

// Column exponents: 2^{e_j} above 8.67 hypot(q+, q-) >= |alpha_j|, |beta_j|.
bool f64tc_column_exponents(const std::vector<double2> &sq, std::vector<int> &e) {
    e.resize(sq.size());
    for (size_t j = 0; j < sq.size(); ++j) {
        const double h = 8.67 * std::hypot(sq[j].x, sq[j].y);
        if (!std::isfinite(h)) return false;
        // an input in the vacuum state contributes nothing, whatever T couples to it
        e[j] = h > 0.0 ? std::ilogb(h) + 1 : kExpVacuum;
        if (h > 0.0 && (e[j] < -kExpRange || e[j] > kExpRange)) return false;
    }
    return true;
}

size_t f64tc_A_bytes(int N, int mtiles) { return (size_t)mtiles * f64tc_kblocks(N) * kAStage; }

size_t f64tc_B_bytes(int N, int64_t chunk) {
    return (size_t)((chunk + kTrajTile - 1) / kTrajTile) * f64tc_kblocks(N) * kBStage;
}

int launch_f64tc_split_T(gbs_net *net, unsigned long long *d_bad) {
    GBS_CUDA_TRY(cudaFuncSetAttribute(k_gemm_f64tc, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      kSmemBytes));
    const dim3 grid((unsigned)(net->mtiles * 128 / kSplitRows), (unsigned)((2 * f64tc_kblocks(net->N) + 31) / 32));
    k_f64tc_split_T<<<grid, 32 * kSplitRows, 0, net->stream>>>(
        net->d_T64, net->d_colexp, net->N, net->M, f64tc_kblocks(net->N), net->d_Aq, net->d_rowexp,
        d_bad);
    GBS_LAUNCH_CHECK();
    return GBS_OK;
}

int launch_gemm_f64tc(gbs_net *net, int64_t count, OccOut64 occ) {
    if (count <= 0) return GBS_OK;
    const int64_t stiles = (count + kTrajTile - 1) / kTrajTile;
    const int64_t ntiles = stiles * net->mtiles;
    if (ntiles > 0x3fffffff) return set_error(GBS_EINVAL, "chunk too large");
    const int grid = (int)std::min<int64_t>(ntiles, net->sm_count);
    k_gemm_f64tc<<<grid, kThreads, kSmemBytes, net->stream>>>(
        net->d_Aq, static_cast<const uint8_t *>(net->d_B), net->d_rowexp, f64tc_kblocks(net->N),
        net->mtiles, (int)stiles, count, net->chunk, net->d_nS_part, occ, net->wait_ns,
        net->d_flags + 1);
    GBS_LAUNCH_CHECK();
    return GBS_OK;
}

}  // namespace gbs
