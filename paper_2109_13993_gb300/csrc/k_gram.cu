// k_gram.cu -- CalculateCovMat (Algorithm 3): Sigma = Xn Xn^T / (n-1)
// of the normalised rows, the covariance the closed forms of Sec. III-E start
// from.  The FP64 path's version, and the mixed path's for the small problems of a batch.  The
// diagonal is exactly 1 (normalised rows).
#include <algorithm>

#include "common.cuh"
#include "launch.h"

namespace lingam {

// ------------------------------------------------------------------ FP64
// 32 x 32 tiles of the upper triangle times splits of the sample axis, so that the whole GPU works
// also on few variables; a thread has 2 x 2 elements, and chunks of 32 samples of the tile's rows and
// columns are staged in shared memory, the next chunk loaded into registers meanwhile.  Bound by the
// FP64 rate (1.7 FMAs a clock and SM), so small tiles cost nothing: their operand reads hide behind
// it, and less of the triangle is padding.  A covariance call at p = 300, n = 5000 took 5.87 ms
// with 64 x 64 tiles and no split (15 CTAs), 0.89 ms now (0.47 ms of it the FMAs at that rate).  The splits' partial tiles are added in split order by a second kernel.
constexpr int kGT = 32;        // output tile
constexpr int kGK = 32;        // samples per chunk
constexpr int kGSplitCtas = 608;   // CTAs wanted: four per SM, so that the last round is short

__device__ __forceinline__ void gram_tile(int tile, int nt, int& bi, int& bj) {
    bi = 0;
    while (tile >= nt - bi) {
        tile -= nt - bi;
        ++bi;
    }
    bj = bi + tile;
}
__device__ __forceinline__ void gram_store(const Fit& f, int i, int j, double s) {
    const int p = f.p;
    if (i >= p || j >= p || i > j) return;
    const double v = i == j ? 1.0 : s * (1.0 / double(f.n - 1));
    f.sig[size_t(i) * p + j] = v;
    f.sig[size_t(j) * p + i] = v;
    f.sig0[size_t(i) * p + j] = v;
    f.sig0[size_t(j) * p + i] = v;
}

__global__ void __launch_bounds__(256) k_gram(Fit f, double* __restrict__ partial, int nt, int nsplit) {
    __shared__ double As[kGT][kGK + 1], Bs[kGT][kGK + 1];
    const int p = f.p, ld = f.ld, tid = threadIdx.x;
    const int tile = blockIdx.x / nsplit, split = blockIdx.x - tile * nsplit;
    int bi, bj;
    gram_tile(tile, nt, bi, bj);
    const int nch = ld / kGK, c0 = int((long long)split * nch / nsplit), c1 = int((long long)(split + 1) * nch / nsplit);
    const double* xt = static_cast<const double*>(f.xt);
    const int lane = tid & 31, w = tid >> 5;   // warp w stages rows w, w + 8, ...
    const int ty = tid >> 4, tx = tid & 15;
    double ra[4], rb[4];
    auto load = [&](int c) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = bi * kGT + w + 8 * q, j = bj * kGT + w + 8 * q;
            ra[q] = i < p ? xt[size_t(i) * ld + c * kGK + lane] : 0.0;
            rb[q] = j < p ? xt[size_t(j) * ld + c * kGK + lane] : 0.0;
        }
    };
    double acc[2][2] = {};
    if (c0 < c1) load(c0);
    for (int c = c0; c < c1; ++c) {
        __syncthreads();   // the previous chunk is consumed
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            As[w + 8 * q][lane] = ra[q];
            Bs[w + 8 * q][lane] = rb[q];
        }
        __syncthreads();
        if (c + 1 < c1) load(c + 1);
#pragma unroll 8
        for (int k = 0; k < kGK; ++k) {
            const double a0 = As[ty][k], a1 = As[ty + 16][k], b0 = Bs[tx][k], b1 = Bs[tx + 16][k];
            acc[0][0] = fma(a0, b0, acc[0][0]);
            acc[0][1] = fma(a0, b1, acc[0][1]);
            acc[1][0] = fma(a1, b0, acc[1][0]);
            acc[1][1] = fma(a1, b1, acc[1][1]);
        }
    }
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const int i = ty + 16 * a, j = tx + 16 * b;
            if (nsplit > 1) partial[(size_t(blockIdx.x) * kGT + i) * kGT + j] = acc[a][b];
            else gram_store(f, bi * kGT + i, bj * kGT + j, acc[a][b]);
        }
}

__global__ void __launch_bounds__(256) k_gram_reduce(Fit f, const double* __restrict__ partial, int nt, int nsplit) {
    int bi, bj;
    gram_tile(blockIdx.x, nt, bi, bj);
    const int e = blockIdx.y * 256 + threadIdx.x, i = e / kGT, j = e % kGT;
    const double* src = partial + size_t(blockIdx.x) * nsplit * kGT * kGT + e;
    double s = 0.0;
    int k = 0;
    for (; k + 8 <= nsplit; k += 8) {   // split order, eight loads in flight
        double v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = src[size_t(k + q) * kGT * kGT];
#pragma unroll
        for (int q = 0; q < 8; ++q) s += v[q];
    }
    for (; k < nsplit; ++k) s += src[size_t(k) * kGT * kGT];
    gram_store(f, bi * kGT + i, bj * kGT + j, s);
}

// (the partial tiles take at most 608 x 8 KB, or nothing: they fit the FP64 path's partial-moment
// region, at least 64 KB per tile of 32 variables and 32 samples, up to 320 of them)
cudaError_t launch_gram(const Fit& f, size_t partial_bytes, cudaStream_t st, long long* launches) {
    const int nt = (f.p + kGT - 1) / kGT, ntri = nt * (nt + 1) / 2;
    const int room = int(std::min<size_t>(partial_bytes / (size_t(ntri) * kGT * kGT * sizeof(double)), 1 << 20));
    const int nsplit = std::max(1, std::min(std::min(kGSplitCtas / ntri, f.ld / kGK), room));
    double* partial = static_cast<double*>(f.partials);
    k_gram<<<ntri * nsplit, 256, 0, st>>>(f, partial, nt, nsplit);
    cudaError_t e = cudaGetLastError();
    if (launches) *launches += nsplit > 1 ? 2 : 1;
    if (e != cudaSuccess || nsplit == 1) return e;
    k_gram_reduce<<<dim3(ntri, kGT * kGT / 256), 256, 0, st>>>(f, partial, nt, nsplit);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ small problems of a batch
// CalculateCovMat of every problem of a batch table with p <= kSmallGramP and rows of at most
// kSmallGramLd samples (mixed path) in one launch, where the per-problem tensor-core Gram
// would pay three launches and their fixed costs per problem.  A CTA takes 256 elements of
// one problem's upper triangle, one per thread, in the order t = j (j + 1) / 2 + i (i <= j),
// so that a warp's threads read consecutive rows of the staged chunk; every chunk of kSGK
// samples of all the problem's rows is staged in shared memory.  Each product of two FP32
// row values is split exactly into hi + lo (TwoProd by fma) and added into a float-float
// sum, so the result is the exact Gram of the FP32 rows up to the float-float rounding, like
// the tensor-core version's.
constexpr int kSGOut = 256;
constexpr int kSGK = 32;

__host__ __device__ inline int small_gram_units(long long p, long long ld) {
    if (p < 1 || p > kSmallGramP || ld > kSmallGramLd) return 0;
    const long long tri = p * (p + 1) / 2;
    return int((tri + kSGOut - 1) / kSGOut);
}

__device__ __forceinline__ void ff_mac(float a, float b, float& hi, float& lo) {
    const float pr = a * b, pe = fmaf(a, b, -pr);   // a b = pr + pe exactly
    const float s = hi + pr, bb = s - hi;
    lo += ((hi - (s - bb)) + (pr - bb)) + pe;        // TwoSum error of hi + pr
    hi = s;
}

__global__ void __launch_bounds__(kSGOut) k_gram_small_batch(const Fit* __restrict__ fits, int count) {
    constexpr int NW = kSGOut / 32;
    __shared__ int s_off[kBatchLaunchMax + 1];
    __shared__ int s_wsum[NW];
    __shared__ float xs[kSGK][kSmallGramP + 1];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    // the problems' first units (an exclusive prefix over the table, count <= kBatchLaunchMax)
    int run = 0;
    for (int base = 0; base < count; base += kSGOut) {
        const int d = base + tid;
        const int u = d < count ? small_gram_units(fits[d].p, fits[d].ld) : 0;
        int x = u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_wsum[wid] = x;
        __syncthreads();
        int wo = 0, tot = 0;
        for (int w = 0; w < NW; ++w) {
            wo += w < wid ? s_wsum[w] : 0;
            tot += s_wsum[w];
        }
        if (d < count) s_off[d] = run + wo + x - u;
        run += tot;
        __syncthreads();
    }
    if (tid == 0) s_off[count] = run;
    __syncthreads();
    const int b = int(blockIdx.x);
    if (b >= s_off[count]) return;   // the whole CTA
    int d = 0, hi_d = count - 1;     // the last problem whose first unit is at most b
    while (d < hi_d) {
        const int mid = (d + hi_d + 1) >> 1;
        if (s_off[mid] <= b) d = mid;
        else hi_d = mid - 1;
    }
    const Fit& f = fits[d];
    const int p = f.p, ld = f.ld;
    const int t = (b - s_off[d]) * kSGOut + tid;
    const bool mine = t < p * (p + 1) / 2;
    int j = 0, i = 0;
    if (mine) {
        j = int((sqrtf(8.f * float(t) + 1.f) - 1.f) * 0.5f);
        while (j * (j + 1) / 2 > t) --j;
        while ((j + 1) * (j + 2) / 2 <= t) ++j;
        i = t - j * (j + 1) / 2;
    }
    float shi = 0.f, slo = 0.f;
    const float* xt = static_cast<const float*>(f.xt);
    const int nst = p * kSGK;
    for (int k0 = 0; k0 < ld; k0 += kSGK) {
        __syncthreads();   // the previous chunk is consumed
        for (int e = tid; e < nst; e += kSGOut) {
            const int r = e >> 5, kk = e & (kSGK - 1);
            xs[kk][r] = xt[size_t(r) * ld + k0 + kk];
        }
        __syncthreads();
#pragma unroll 8
        for (int kk = 0; kk < kSGK; ++kk) ff_mac(xs[kk][i], xs[kk][j], shi, slo);
    }
    if (!mine) return;
    const double v = i == j ? 1.0 : (double(shi) + double(slo)) / double(f.n - 1);
    f.sig[size_t(i) * p + j] = v;
    f.sig[size_t(j) * p + i] = v;
    f.sig0[size_t(i) * p + j] = v;
    f.sig0[size_t(j) * p + i] = v;
    const float2 vf = sig_pair_f(v);
    f.sigf[size_t(i) * p + j] = vf;
    f.sigf[size_t(j) * p + i] = vf;
}

int gram_small_batch_units(const long long* p, const int* ld, int count) {
    int u = 0;
    for (int k = 0; k < count; ++k) u += small_gram_units(p[k], ld[k]);
    return u;
}

cudaError_t launch_gram_small_batch(const Fit* fits_dev, int count, int units, cudaStream_t st) {
    if (count < 1 || count > kBatchLaunchMax || units < 1) return cudaErrorInvalidValue;
    k_gram_small_batch<<<units, kSGOut, 0, st>>>(fits_dev, count);
    return cudaGetLastError();
}

}  // namespace lingam
