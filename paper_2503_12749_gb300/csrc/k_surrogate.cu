// The surrogate's representation of a network and of its count distribution
// (features, their statistics and standardisation, encoding a distribution
// into the network's output grid and decoding an output back into P(m)).
// Not part of the paper; the distribution it represents is the binned total
// count of Eq. total_counts.  Definitions:
//   mu  = t^2 sum_j sinh^2 r_j,  s^2 = sum_j [t^2 sinh^2 r_j + t^4 sinh^2 r_j cosh 2 r_j]
//   (mean and variance of the total count for T = t U, from the cumulants of
//   the uniform-loss determinant generating function);
//   grid x_i = -8 + 16 (i + 1/2) / 256, output o[p*256 + i] = 100 (f_p(x_i) - phi(x_i)/2),
//   f_p(x) = (s/2) P(mu + s x) on the counts of parity p;
//   interpolation: Catmull-Rom cubic (Catmull & Rom 1974) in Hermite form.
// Every reduction runs in a fixed order, so results do not depend on timing.
#include "gbs_internal.cuh"
#include "gbs_surrogate.h"

#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <vector>

namespace cg = cooperative_groups;

namespace gbs {
namespace {

constexpr int kGrid = GBS_SUR_GRID;
constexpr int kRec = GBS_SUR_RECORD;
constexpr int kFeat = GBS_SUR_FEATURES;
constexpr double kXLo = -8.0;
constexpr double kDx = 16.0 / kGrid;
constexpr double kOutScale = 100.0;
constexpr double kInvSqrt2Pi = 0.3989422804014327;  // 1 / sqrt(2 pi)

struct NetIn {
    double t;
    int64_t m_off;
    int64_t r0;
    int N, M, K1, pad;
};

__device__ __forceinline__ double cr(double ym1, double y0, double y1, double y2, double u) {
    const double u2 = u * u, u3 = u2 * u;
    const double h00 = 2.0 * u3 - 3.0 * u2 + 1.0;
    const double h10 = u3 - 2.0 * u2 + u;
    const double h01 = -2.0 * u3 + 3.0 * u2;
    const double h11 = u3 - u2;
    return h00 * y0 + h10 * 0.5 * (y1 - ym1) + h01 * y1 + h11 * 0.5 * (y2 - y0);
}

__device__ __forceinline__ double half_phi(double x) { return 0.5 * kInvSqrt2Pi * exp(-0.5 * x * x); }

template <int kThreadsT>
__device__ __forceinline__ double block_sum(double v, double *red) {
    red[threadIdx.x] = v;
    __syncthreads();
    for (int w = kThreadsT / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    const double s = red[0];
    __syncthreads();
    return s;
}

// Sums over the squeezing parameters, in two kernels: bound by the FP64 pipe (2
// lanes per SM and clock), so the transcendental part is spread over blocks of
// 512 parameters (one block per network left an 8000-mode network on one SM),
// with sinh from one expm1 (sinh r = (u + u / (u + 1)) / 2, u = e^r - 1) and cosh
// 2r = 1 + 2 sinh^2 r.  One pass over r, which may lie in host memory: sums of
// r - c, c the network's first parameter, and squared deviations about each
// block's own mean, which k_sur_features joins (Chan, Golub, LeVeque, "Algorithms
// for computing the sample variance", Amer. Statist. 37, 1983): nothing cancels,
// whatever c is.
// part[net][chunk] = sum r - c, sum (r - c - its chunk mean)^2, sum eta sinh^2, sum
// (eta sinh^2)^2 (finite wherever the variance is), min, max.
constexpr int kFeatChunk = 512;
constexpr int kFeatPart = 6;

__global__ void __launch_bounds__(256) k_sur_feature_parts(const NetIn *__restrict__ nets,
                                                           const double *__restrict__ r,
                                                           int chunks, double *__restrict__ part) {
    __shared__ double red[8][kFeatPart];
    const NetIn n = nets[blockIdx.y];
    const int j0 = blockIdx.x * kFeatChunk;
    if (j0 >= n.N) return;
    const double *rj = r + n.r0;
    const double c = rj[0], eta = n.t * n.t;
    double v[kFeatPart] = {0.0, 0.0, 0.0, 0.0, INFINITY, -INFINITY};
    auto join = [](double (&a)[kFeatPart], const double (&b)[kFeatPart]) {
#pragma unroll
        for (int q = 0; q < 4; ++q) a[q] += b[q];
        a[4] = fmin(a[4], b[4]);
        a[5] = fmax(a[5], b[5]);
    };
    double dev[kFeatChunk / 256] = {};
#pragma unroll
    for (int t = 0; t < kFeatChunk / 256; ++t) {
        const int j = j0 + t * 256 + threadIdx.x;
        if (j >= n.N) break;
        const double x = rj[j];
        const double u = expm1(x);
        const double sh = 0.5 * (u + (u < 0x1p60 ? u / (u + 1.0) : 1.0));
        const double m = eta * (sh * sh);
        dev[t] = x - c;
        join(v, {dev[t], 0.0, m, m * m, x, x});
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        double w[kFeatPart];
#pragma unroll
        for (int q = 0; q < kFeatPart; ++q) w[q] = __shfl_xor_sync(0xffffffffu, v[q], o);
        join(v, w);
    }
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int q = 0; q < kFeatPart; ++q) red[threadIdx.x >> 5][q] = v[q];
    __syncthreads();
    double mean = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) mean += red[w][0];
    mean /= (double)min(kFeatChunk, n.N - j0);
    double m2 = 0.0;
#pragma unroll
    for (int t = 0; t < kFeatChunk / 256; ++t)
        if (j0 + t * 256 + (int)threadIdx.x < n.N) m2 += (dev[t] - mean) * (dev[t] - mean);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m2 += __shfl_xor_sync(0xffffffffu, m2, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][1] = m2;
    __syncthreads();
    if (threadIdx.x == 0) {
        v[1] = m2;
        for (int w = 1; w < 8; ++w) join(v, red[w]);
        double *o = part + ((size_t)blockIdx.y * chunks + blockIdx.x) * kFeatPart;
#pragma unroll
        for (int q = 0; q < kFeatPart; ++q) o[q] = v[q];
    }
}

// One warp per network: its chunks in order, and the record.
__global__ void k_sur_features(const NetIn *__restrict__ nets, const double *__restrict__ r,
                               const double *__restrict__ part, int chunks, int count,
                               double *__restrict__ rec) {
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (i >= count) return;
    const NetIn n = nets[i];
    double v = 0.0;
    if (lane < kFeatPart) {
        const double *p = part + (size_t)i * chunks * kFeatPart + lane;
        v = p[0];
        for (int c = 1; c * kFeatChunk < n.N; ++c) {
            const double w = p[c * kFeatPart];
            v = lane < 4 ? v + w : lane == 4 ? fmin(v, w) : fmax(v, w);
        }
    }
    double t[kFeatPart];
#pragma unroll
    for (int q = 0; q < kFeatPart; ++q) t[q] = __shfl_sync(0xffffffffu, v, q);
    const double eta = n.t * n.t;
    const double mu = t[2];
    // sum of eta sinh^2 + eta^2 sinh^2 (1 + 2 sinh^2)
    const double s = sqrt(mu + eta * mu + 2.0 * t[3]);
    const double d = t[0] / (double)n.N;
    // the chunk means' own deviations, a chunk per lane
    double between = 0.0;
    for (int c = lane; c * kFeatChunk < n.N; c += 32) {
        const double cnt = (double)min(kFeatChunk, n.N - c * kFeatChunk);
        const double e = part[((size_t)i * chunks + c) * kFeatPart] / cnt - d;
        between += cnt * e * e;
    }
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) between += __shfl_xor_sync(0xffffffffu, between, w);
    double *o = rec + (size_t)i * kRec;
    // the logarithms side by side in the lanes
    double x = 1.0;
    if (lane == 0) x = (double)n.N;
    if (lane == 1) x = (double)n.M;
    if (lane == 8) x = mu;
    if (lane == 9) x = s;
    const double lg = log(x);
    if (lane == 0 || lane == 1 || lane == 8 || lane == 9) o[lane] = lg;
    if (lane == 2) o[2] = r[n.r0] + d;
    if (lane == 3) o[3] = sqrt((t[1] + between) / (double)n.N);
    if (lane == 4) o[4] = t[4];
    if (lane == 5) o[5] = t[5];
    if (lane == 6) o[6] = n.t;
    if (lane == 7) o[7] = (double)(31 - __clz(n.K1));  // a power of two
    if (lane == 10) o[10] = mu;
    if (lane == 11) o[11] = s;
    if (lane == 12) o[12] = (double)n.m_off;
    if (lane == 13) o[13] = (double)n.K1;
}

// One block of 32 x kFeat threads: warp f handles feature f.
__global__ void k_sur_stats(const double *__restrict__ rec, int count, double *__restrict__ stats) {
    const int f = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    double s = 0.0, lo = INFINITY, hi = -INFINITY;
    for (int i = lane; i < count; i += 32) {
        const double x = rec[(size_t)i * kRec + f];
        s += x;
        lo = fmin(lo, x);
        hi = fmax(hi, x);
    }
    for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    const double mean = s / (double)count;
    double d2 = 0.0;
    for (int i = lane; i < count; i += 32) {
        const double d = rec[(size_t)i * kRec + f] - mean;
        d2 += d * d;
    }
    for (int o = 16; o > 0; o >>= 1) d2 += __shfl_xor_sync(0xffffffffu, d2, o);
    if (lane == 0) {
        stats[f] = mean;
        stats[kFeat + f] = sqrt(d2 / (double)count);
        stats[2 * kFeat + f] = lo;
        stats[3 * kFeat + f] = hi;
    }
}

__global__ void k_sur_standardize(const double *__restrict__ rec, int count,
                                  const double *__restrict__ stats, float *__restrict__ X,
                                  int *__restrict__ in_domain) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    int ok = 1;
    for (int f = 0; f < kFeat; ++f) {
        const double u = rec[(size_t)i * kRec + f];
        const double sd = stats[kFeat + f];
        X[(size_t)i * kFeat + f] = sd > 1e-12 ? (float)((u - stats[f]) / sd) : 0.0f;
        const double lo = stats[2 * kFeat + f], hi = stats[3 * kFeat + f];
        const double pad = 0.02 * (hi - lo);
        if (!(u >= lo - pad && u <= hi + pad)) ok = 0;
    }
    if (in_domain) in_domain[i] = ok;
}

// One block of 2 * kGrid threads per network: output o = p * kGrid + i.
__global__ void k_sur_encode(const double *__restrict__ rec, const double *__restrict__ P,
                             int64_t ldP, float *__restrict__ Y) {
    const double *q = rec + (size_t)blockIdx.x * kRec;
    const double mu = q[10], s = q[11];
    const int64_t m_off = (int64_t)q[12];
    const int64_t K1 = min((int64_t)q[13], ldP);
    const double *Pn = P + (size_t)blockIdx.x * ldP;
    const int p = threadIdx.x / kGrid;
    const int i = threadIdx.x % kGrid;
    const double x = kXLo + kDx * (i + 0.5);
    const double pos = (mu + s * x - p) / 2.0;  // on the lattice m = p + 2 pos
    const double q0 = floor(pos);
    const double u = pos - q0;
    double y[4];
#pragma unroll
    for (int d = 0; d < 4; ++d) {
        const int64_t m = p + 2 * ((int64_t)q0 + d - 1);
        const int64_t j = m - m_off;
        y[d] = (j >= 0 && j < K1) ? Pn[j] : 0.0;
    }
    const double f = 0.5 * s * cr(y[0], y[1], y[2], y[3], u);
    Y[(size_t)blockIdx.x * 2 * kGrid + threadIdx.x] = (float)(kOutScale * (f - half_phi(x)));
}

// phi(x_i) / 2 on the output grid (host table, passed by value).
struct HalfPhi {
    double v[kGrid];
};

HalfPhi half_phi_table() {
    HalfPhi t;
    for (int i = 0; i < kGrid; ++i) {
        const double x = kXLo + kDx * (i + 0.5);
        t.v[i] = 0.5 * kInvSqrt2Pi * std::exp(-0.5 * x * x);
    }
    return t;
}

// P(m) on the window, then renormalised (which also cancels the factor 2 / s of
// a density): a cluster of kDecodeBlocks blocks (256 threads) per network, the
// total through distributed shared memory.  Bound by the FP64 pipe: with one
// block per network and the exponentials, divisions and Hermite basis written
// out, 4096 counts took 129 us of one SM (under ncu).
constexpr int kDecodeBlocks = 4;

__global__ void __cluster_dims__(kDecodeBlocks, 1, 1) __launch_bounds__(256)
    k_sur_decode(const double *__restrict__ rec, const float *__restrict__ Y, const HalfPhi hp,
                 double *__restrict__ P, int64_t ldP) {
    __shared__ double f[2][kGrid + 4];  // two zeros before and after the grid
    __shared__ double red[256];
    __shared__ double part;
    cg::cluster_group cluster = cg::this_cluster();
    const int net = blockIdx.x / kDecodeBlocks, rank = blockIdx.x % kDecodeBlocks;
    const double *q = rec + (size_t)net * kRec;
    const double mu = q[10], inv = 1.0 / (q[11] * kDx);
    const int64_t m_off = (int64_t)q[12];
    const int64_t K1 = min((int64_t)q[13], ldP);
    const float *o = Y + (size_t)net * 2 * kGrid;
    for (int k = threadIdx.x; k < 2 * (kGrid + 4); k += 256) {
        const int p = k / (kGrid + 4), i = k % (kGrid + 4) - 2;
        f[p][i + 2] = i >= 0 && i < kGrid ? (double)o[p * kGrid + i] / kOutScale + hp.v[i] : 0.0;
    }
    __syncthreads();
    double *Pn = P + (size_t)net * ldP;
    double sum = 0.0;
    for (int64_t j = rank * 256 + threadIdx.x; j < K1; j += 256 * kDecodeBlocks) {
        const int64_t m = m_off + j;
        const double g = (m - mu) * inv - (kXLo + 0.5 * kDx) / kDx;
        double v = 0.0;
        if (g >= 0.0 && g <= kGrid - 1) {
            const double g0 = floor(g);
            const double u = g - g0;
            // Catmull-Rom (cr) in powers of u
            const double *y = &f[m & 1][(int)g0 + 1];
            const double c1 = 0.5 * (y[2] - y[0]);
            const double d = y[1] - y[2];
            const double c3 = 0.5 * (y[3] - y[0]) + 1.5 * d;
            const double c2 = -(c1 + c3) - d;
            v = fmax(fma(fma(fma(c3, u, c2), u, c1), u, y[1]), 0.0);
        }
        Pn[j] = v;
        sum += v;
    }
    sum = block_sum<256>(sum, red);
    if (threadIdx.x == 0) part = sum;
    cluster.sync();
    double total = 0.0;
#pragma unroll
    for (int b = 0; b < kDecodeBlocks; ++b) total += *cluster.map_shared_rank(&part, b);
    cluster.sync();  // every block has read the parts
    if (total > 0.0) {
        const double scale = 1.0 / total;
        for (int64_t j = rank * 256 + threadIdx.x; j < K1; j += 256 * kDecodeBlocks) Pn[j] *= scale;
    }
}

// Whether every r[j] is finite and positive (written to vectorise).
__attribute__((optimize("O3"))) bool all_positive(const double *r, int64_t n) {
    int64_t bad = 0;
    for (int64_t j = 0; j < n; ++j) bad += !(r[j] > 0.0 && r[j] <= 1.7976931348623157e308);
    return bad == 0;
}

int check_records(int count, const void *feat) {
    if (count < 1) return set_error(GBS_EINVAL, "count must be >= 1");
    if (count > 2147483647 / 512) return set_error(GBS_EINVAL, "count too large");
    if (!feat) return set_error(GBS_EINVAL, "feature records are NULL");
    return GBS_OK;
}

}  // namespace
}  // namespace gbs

using namespace gbs;

extern "C" {

int gbs_surrogate_features(int count, const int *N, const int *M, const double *t, const int *K1,
                           const int64_t *m_off, const double *r, const int64_t *r_off, void *stream,
                           double *feat_dev) {
    int rc;
    if ((rc = check_records(count, feat_dev))) return rc;
    if (!N || !M || !t || !K1 || !m_off || !r || !r_off)
        return set_error(GBS_EINVAL, "NULL host array");
    if (r_off[0] != 0) return set_error(GBS_EINVAL, "r_off[0] must be 0");
    std::vector<NetIn> h((size_t)count);
    for (int i = 0; i < count; ++i) {
        if (N[i] < 1 || M[i] < 1 || r_off[i + 1] - r_off[i] != N[i])
            return set_error(GBS_EINVAL, "network %d: N, M >= 1 and r_off[i+1] - r_off[i] = N", i);
        if (K1[i] < 2 || K1[i] > (1 << 24) || (K1[i] & (K1[i] - 1)))
            return set_error(GBS_EINVAL, "network %d: K1 must be a power of two in [2, 2^24]", i);
        if (!(t[i] > 0.0 && t[i] <= 1.0)) return set_error(GBS_EINVAL, "network %d: t outside (0, 1]", i);
        if (m_off[i] < 0) return set_error(GBS_EINVAL, "network %d: m_off < 0", i);
        h[(size_t)i] = NetIn{t[i], m_off[i], r_off[i], N[i], M[i], K1[i], 0};
    }
    const int64_t nr = r_off[count];
    if (!all_positive(r, nr))
        for (int64_t j = 0; j < nr; ++j)
            if (!(std::isfinite(r[j]) && r[j] > 0.0))
                return set_error(GBS_EINVAL, "r[%lld] must be finite and > 0", (long long)j);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int Nmax = 0;
    for (int i = 0; i < count; ++i) Nmax = N[i] > Nmax ? N[i] : Nmax;
    const int chunks = (Nmax + kFeatChunk - 1) / kFeatChunk;
    // Where the device reads the host's own page tables (Grace), r is read in place,
    // once, over the host link; else it is uploaded: also where pageable memory is
    // addressable but its pages would migrate, and an r that is not 8-byte aligned.
    // The call synchronises before it returns, so r is not read afterwards.
    int dev = 0, direct = 0;
    if (reinterpret_cast<uintptr_t>(r) % sizeof(double) == 0 &&
        (cudaGetDevice(&dev) != cudaSuccess ||
         cudaDeviceGetAttribute(&direct, cudaDevAttrPageableMemoryAccessUsesHostPageTables, dev) !=
             cudaSuccess)) {
        cudaGetLastError();
        direct = 0;
    }
    // stream-ordered work space: no allocation by the driver on each call
    void *d_nets = nullptr, *d_r = nullptr, *d_part = nullptr;
    if ((rc = pool_alloc(&d_nets, sizeof(NetIn) * (size_t)count, s, "network parameters")) ||
        (!direct && (rc = pool_alloc(&d_r, sizeof(double) * (size_t)nr, s, "squeezing parameters"))) ||
        (rc = pool_alloc(&d_part, sizeof(double) * (size_t)count * chunks * kFeatPart, s,
                         "feature sums"))) {
        pool_free_raw(d_nets, s);
        pool_free_raw(d_r, s);
        return rc;
    }
    if (cudaMemcpyAsync(d_nets, h.data(), sizeof(NetIn) * (size_t)count, cudaMemcpyHostToDevice, s) !=
            cudaSuccess ||
        (!direct && cudaMemcpyAsync(d_r, r, sizeof(double) * (size_t)nr, cudaMemcpyHostToDevice, s) !=
                        cudaSuccess))
        rc = set_error(GBS_ECUDA, "upload of the network parameters failed");
    if (!rc) {
        const double *rp = direct ? r : static_cast<const double *>(d_r);
        const NetIn *np = static_cast<const NetIn *>(d_nets);
        double *pp = static_cast<double *>(d_part);
        // grid.y holds at most 65535 networks
        for (int i0 = 0; i0 < count; i0 += 65535)
            k_sur_feature_parts<<<dim3((unsigned)chunks, (unsigned)std::min(65535, count - i0)), 256, 0,
                                  s>>>(np + i0, rp, chunks, pp + (size_t)i0 * chunks * kFeatPart);
        k_sur_features<<<(count + 7) / 8, 256, 0, s>>>(np, rp, pp, chunks, count, feat_dev);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) rc = set_error(GBS_ECUDA, "feature kernel: %s", cudaGetErrorString(e));
    }
    if (cudaStreamSynchronize(s) != cudaSuccess && !rc)
        rc = set_error(GBS_ECUDA, "feature kernel failed");
    pool_free_raw(d_nets, s);
    pool_free_raw(d_r, s);
    pool_free_raw(d_part, s);
    return rc;
}

int gbs_surrogate_feature_stats(int count, const double *feat_dev, void *stream, double *stats_dev) {
    int rc;
    if ((rc = check_records(count, feat_dev))) return rc;
    if (!stats_dev) return set_error(GBS_EINVAL, "stats_dev is NULL");
    k_sur_stats<<<1, 32 * kFeat, 0, static_cast<cudaStream_t>(stream)>>>(feat_dev, count, stats_dev);
    GBS_LAUNCH_CHECK();
    return GBS_OK;
}

int gbs_surrogate_standardize(int count, const double *feat_dev, const double *stats_dev,
                              void *stream, float *X_dev, int *in_domain_dev) {
    int rc;
    if ((rc = check_records(count, feat_dev))) return rc;
    if (!stats_dev || !X_dev) return set_error(GBS_EINVAL, "NULL device array");
    k_sur_standardize<<<(count + 127) / 128, 128, 0, static_cast<cudaStream_t>(stream)>>>(
        feat_dev, count, stats_dev, X_dev, in_domain_dev);
    GBS_LAUNCH_CHECK();
    return GBS_OK;
}

int gbs_surrogate_encode(int count, const double *feat_dev, const double *P_dev, int64_t ldP,
                         void *stream, float *Y_dev) {
    int rc;
    if ((rc = check_records(count, feat_dev))) return rc;
    if (!P_dev || !Y_dev || ldP < 1) return set_error(GBS_EINVAL, "NULL device array or ldP < 1");
    k_sur_encode<<<count, 2 * kGrid, 0, static_cast<cudaStream_t>(stream)>>>(feat_dev, P_dev, ldP,
                                                                             Y_dev);
    GBS_LAUNCH_CHECK();
    return GBS_OK;
}

int gbs_surrogate_decode(int count, const double *feat_dev, const float *Y_dev, void *stream,
                         double *P_dev, int64_t ldP) {
    int rc;
    if ((rc = check_records(count, feat_dev))) return rc;
    if (!P_dev || !Y_dev || ldP < 1) return set_error(GBS_EINVAL, "NULL device array or ldP < 1");
    static const HalfPhi hp = half_phi_table();
    k_sur_decode<<<count * kDecodeBlocks, 256, 0, static_cast<cudaStream_t>(stream)>>>(
        feat_dev, Y_dev, hp, P_dev, ldP);
    GBS_LAUNCH_CHECK();
    return GBS_OK;
}

}  // extern "C"
