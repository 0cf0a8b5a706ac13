// k_bfit.cu -- causal strengths B from the causal order (Algorithm 1, last
// line; "conventional covariance-based regression", Sec. II-C), FP64.
//
// B row K[k] holds the least-squares coefficients of x_{K[k]} on its
// predecessors x_{K[0..k-1]}.  With C the covariance of the original variables
// permuted into the order K and C = R R^T its Cholesky factorisation (R lower
// triangular), the innovations e = diag(R) R^{-1} x are uncorrelated and
// x = (I - diag(R) R^{-1}) x + e, so B_K = I - diag(R) R^{-1}, strictly lower
// triangular; B is B_K with rows and columns mapped back to variable indices.
#include <algorithm>

#include "common.cuh"
#include "launch.h"

namespace lingam {

// C[a][b] = sd_{K[a]} sd_{K[b]} Sigma0[K[a]][K[b]]  (original units)
__global__ void k_perm_cov(Fit f) {
    const int p = f.p;
    const int a = blockIdx.y * 16 + (threadIdx.x >> 4), b = blockIdx.x * 16 + (threadIdx.x & 15);
    if (a >= p || b >= p) return;
    const int ia = f.order[a], ib = f.order[b];
    f.cmat[size_t(a) * p + b] = f.sd[ia] * f.sd[ib] * f.sig0[size_t(ia) * p + ib];
}

// Right-looking Cholesky C = R R^T (R lower) in one cooperative launch, as a data flow
// over rows.  The working matrix is the upper triangle U of C (row k of U holds column k
// of C, so every access below is along a row).  At step k, row k of rmat receives
// R[i][k] = U[k][i] / sqrt(U[k][k]) (i >= k) and the rows i > k lose the rank-one term
// U[i][j] -= U[k][i] U[k][j] / U[k][k] (j >= i).  Row i belongs to CTA i mod G for the
// whole factorisation, so its successive updates follow one another inside one CTA;
// step k needs only row k final, which its owner publishes (ready[k] = 1) as soon as
// it has applied step k - 1 to it, before its other rows, so the next steps start while
// the bulk of the current one is still running.  A non-positive pivot records
// LINGAM_EDEGENERATE (every CTA reads the same final pivot, so all leave at the same
// step); every wait is bounded by the fit's timeout.
constexpr int kCholThreads = 256;
constexpr int kCholRows = 128;   // rows of one CTA staged at a time
constexpr int kCholBatch = 8;    // elements per thread with their loads in flight together

// U[i][j] -= a U[k][j] for the rows i0, i0 + G, ... (< p, at most kCholRows of them) and
// j >= i, their elements numbered one after another over the CTA's threads.
__device__ void chol_rows(double* U, const double* uk, double inv, int p, int i0, int G, int* s_i, int* s_off,
                          double* s_a) {
    const int tid = threadIdx.x;
    const int nr = min(kCholRows, (p - 1 - i0) / G + 1);
    __syncthreads();   // the previous row table is no longer read
    for (int r = tid; r < nr; r += kCholThreads) {
        const int i = i0 + r * G;
        s_i[r] = i;
        s_a[r] = __ldcg(uk + i) * inv;
    }
    if (tid == 0) {
        int o = 0;
        for (int r = 0; r < nr; ++r) {
            s_off[r] = o;
            o += p - (i0 + r * G);
        }
        s_off[nr] = o;
    }
    __syncthreads();
    const int tot = s_off[nr];
    for (int base = tid; base < tot; base += kCholBatch * kCholThreads) {
        size_t at[kCholBatch];
        int jj[kCholBatch];
        double av[kCholBatch], x[kCholBatch], y[kCholBatch];
#pragma unroll
        for (int q = 0; q < kCholBatch; ++q) {
            const int idx = base + q * kCholThreads;
            jj[q] = -1;
            if (idx < tot) {
                int lo = 0, hi = nr - 1;   // the row: last r with s_off[r] <= idx
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (s_off[mid] <= idx) lo = mid;
                    else hi = mid - 1;
                }
                const int i = s_i[lo];
                jj[q] = i + (idx - s_off[lo]);
                at[q] = size_t(i) * p + jj[q];
                av[q] = s_a[lo];
            }
        }
#pragma unroll
        for (int q = 0; q < kCholBatch; ++q)
            if (jj[q] >= 0) {
                x[q] = __ldcg(uk + jj[q]);
                y[q] = __ldcg(U + at[q]);
            }
#pragma unroll
        for (int q = 0; q < kCholBatch; ++q)
            if (jj[q] >= 0) U[at[q]] = fma(-av[q], x[q], y[q]);
    }
}

__global__ void __launch_bounds__(kCholThreads) k_chol_coop(Fit f) {
    __shared__ int s_i[kCholRows], s_off[kCholRows + 1];
    __shared__ double s_a[kCholRows];
    __shared__ int s_ok;
    const int p = f.p, tid = threadIdx.x, b = blockIdx.x, G = gridDim.x;
    double* U = f.cmat;
    int* ready = f.scratch;   // ready[k] = 1: row k final (zeroed by the host)
    for (int k = 0; k < p; ++k) {
        if (tid == 0) {
            int ok = 1;
            if (k > 0) {
                ok = wait_flag_set(ready + k, f.ctl) ? 1 : 0;
                __threadfence();
            }
            s_ok = ok;
        }
        __syncthreads();   // also orders this CTA's writes of step k - 1 before its reads
        if (!s_ok) return;
        const double* uk = U + size_t(k) * p;
        const double ukk = __ldcg(uk + k);
        if (!(ukk > 0.0)) {
            if (tid == 0 && b == k % G) set_status(f.ctl, LINGAM_EDEGENERATE);
            return;
        }
        const double inv = 1.0 / ukk;
        // row k + 1 first, published as soon as it is final
        const int i1 = k + 1;
        if (i1 < p && i1 % G == b) {
            chol_rows(U, uk, inv, p, i1, p, s_i, s_off, s_a);   // stride p: this row alone
            __syncthreads();
            if (tid == 0) {
                __threadfence();
                atomicExch(ready + i1, 1);
            }
        }
        if (b == k % G) {
            const double rk = sqrt(ukk);
            for (int i = k + tid; i < p; i += kCholThreads) f.rmat[size_t(k) * p + i] = __ldcg(uk + i) / rk;
        }
        // this CTA's other rows i > k + 1 (i = b mod G), in blocks of kCholRows
        const int ifirst = k + 2 + ((b - (k + 2)) % G + G) % G;
        for (int i0 = ifirst; i0 < p; i0 += kCholRows * G) chol_rows(U, uk, inv, p, i0, G, s_i, s_off, s_a);
    }
}

// Column j of R^{-1} by forward substitution (one CTA per column):
//   y_k = ([k == j] - sum_{m<k} R[k][m] y_m) / R[k][k],  k = j..p-1.
// For p <= NT kTriPer, thread t owns the entries i = t, t + NT, ... of the running sums, in
// registers; column k + 1 of R is loaded while step k runs, so a step's critical path is one
// barrier, a shared-memory read and a few FMAs; and the diagonal's reciprocals are formed
// first, all at once (FP64 divisions are slow on this part).  Larger p: the plain loop.
constexpr int kTriThreads = 256;
constexpr int kTriPer = 4;
__global__ void __launch_bounds__(kTriThreads) k_tri_inv(Fit f) {
    extern __shared__ double sm_tri[];
    double* acc = sm_tri;        // [p] running sums (entries of other threads read at step k)
    const int p = f.p, j = blockIdx.x, tid = threadIdx.x;
    for (int i = tid; i < p; i += kTriThreads) acc[i] = 0.0;
    if (p <= kTriThreads * kTriPer) {
        double* invd = sm_tri + p;   // [p] 1 / R[k][k]
        for (int i = tid; i < p; i += kTriThreads) invd[i] = i >= j ? 1.0 / f.rmat[size_t(i) * p + i] : 0.0;
        __syncthreads();
        double a[kTriPer], cur[kTriPer];
#pragma unroll
        for (int q = 0; q < kTriPer; ++q) {
            a[q] = 0.0;
            const int i = tid + q * kTriThreads;
            cur[q] = i < p ? f.rmat[size_t(j) * p + i] : 0.0;
        }
        for (int k = j; k < p; ++k) {
            double nxt[kTriPer];
            if (k + 1 < p) {
#pragma unroll
                for (int q = 0; q < kTriPer; ++q) {
                    const int i = tid + q * kTriThreads;
                    nxt[q] = i < p ? __ldg(f.rmat + size_t(k + 1) * p + i) : 0.0;
                }
            }
            const double y = ((k == j ? 1.0 : 0.0) - acc[k]) * invd[k];
            if (tid == 0) f.rinv[size_t(k) * p + j] = y;
#pragma unroll
            for (int q = 0; q < kTriPer; ++q) {
                const int i = tid + q * kTriThreads;
                if (i > k && i < p) {
                    a[q] = fma(cur[q], y, a[q]);
                    if (i == k + 1) acc[i] = a[q];   // the only sum step k + 1 reads
                }
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < kTriPer; ++q) cur[q] = nxt[q];
        }
    } else {
        __syncthreads();
        for (int k = j; k < p; ++k) {
            const double* rk = f.rmat + size_t(k) * p;   // column k of R: rk[i] = R[i][k]
            const double y = ((k == j ? 1.0 : 0.0) - acc[k]) / rk[k];
            if (tid == 0) f.rinv[size_t(k) * p + j] = y;
            for (int i = k + 1 + tid; i < p; i += kTriThreads) acc[i] = fma(rk[i], y, acc[i]);
            __syncthreads();
        }
    }
}

// B[K[a]][K[b]] = -R[a][a] Rinv[a][b] for a > b, 0 elsewhere.
__global__ void k_B_out(Fit f) {
    const int p = f.p;
    const int a = blockIdx.y * 16 + (threadIdx.x >> 4), b = blockIdx.x * 16 + (threadIdx.x & 15);
    if (a >= p || b >= p) return;
    const double v = a > b ? -f.rmat[size_t(a) * p + a] * f.rinv[size_t(a) * p + b] : 0.0;
    f.bout[size_t(f.order[a]) * p + f.order[b]] = v;
}

// The same fit for a problem of p <= kBSmall in one CTA (batches: one CTA per
// problem): C in shared memory, Cholesky C = L L^T in place (L lower, L = R), then
// thread b solves column b of L^{-1} by forward substitution into the problem's rinv
// (column-major, scratch) and writes B[K[a]][K[b]] = -L[a][a] Linv[a][b] for a > b.
// Problems with p > kBSmall, or whose status is bad, are left to other launches.
constexpr int kBSmall = 128;
constexpr int kBThreads = 256;

__global__ void __launch_bounds__(kBThreads) k_bfit_small(const Fit* __restrict__ fits, int count) {
    extern __shared__ double C[];
    const Fit f = fits[blockIdx.x];
    const int p = f.p, tid = threadIdx.x;
    if (p > kBSmall || ((volatile Ctl*)f.ctl)->status != 0) return;
    for (int idx = tid; idx < p * p; idx += kBThreads) {
        const int a = idx / p, b = idx - a * p;
        const int ia = f.order[a], ib = f.order[b];
        C[idx] = f.sd[ia] * f.sd[ib] * f.sig0[size_t(ia) * p + ib];
    }
    __syncthreads();
    for (int k = 0; k < p; ++k) {
        const double ckk = C[k * p + k];
        if (!(ckk > 0.0)) {   // every thread reads the same value: a uniform exit
            if (tid == 0) set_status(f.ctl, LINGAM_EDEGENERATE);
            return;
        }
        const double rk = sqrt(ckk);
        __syncthreads();
        for (int i = k + 1 + tid; i < p; i += kBThreads) C[i * p + k] /= rk;
        if (tid == 0) C[k * p + k] = rk;
        __syncthreads();
        const int m = p - k - 1;
        for (int idx = tid; idx < m * m; idx += kBThreads) {
            const int i = k + 1 + idx / m, j = k + 1 + idx % m;
            if (j <= i) C[i * p + j] -= C[i * p + k] * C[j * p + k];
        }
        __syncthreads();
    }
    double* y = f.rinv;   // column b of L^{-1} at y[b * p + a], a >= b
    for (int b = tid; b < p; b += kBThreads) {
        const int kb = f.order[b];
        for (int a = 0; a < b; ++a) f.bout[size_t(f.order[a]) * p + kb] = 0.0;
        for (int a = b; a < p; ++a) {
            double acc = a == b ? 1.0 : 0.0;
            for (int m2 = b; m2 < a; ++m2) acc = fma(-C[a * p + m2], y[size_t(b) * p + m2], acc);
            const double ya = acc / C[a * p + a];
            y[size_t(b) * p + a] = ya;
            f.bout[size_t(f.order[a]) * p + kb] = a > b ? -C[a * p + a] * ya : 0.0;
        }
    }
}

// ------------------------------------------------------------------ from the ordering's factorisation
// The ordering kernel's covariance updates are the elimination steps of Sigma0 = L diag(d) L^T in causal
// order, so it leaves them behind: rmat[k p + v] = L[position of v][k] d_k for the variables v from
// position k on (d_k at v = K[k]; the last d is not needed).  In the normalised variables x = L e with e
// the innovations, so B = I - L^{-1} there, and B[K[a]][K[b]] = -(L^{-1})[a][b] sd_{K[a]} / sd_{K[b]}
// (a > b) in the original units: no Cholesky, whose p row steps of 3.5 us took most of the fit: a call of
// p = 300 takes 0.9 ms less (of 11.0), p = 1000 4.3 ms (of 72.9), p = 20 0.07 ms (of 0.70).  Its errors against long double are a little
// below the Cholesky's (24 random graphs each, n = 500, FP64, geometric means of the norms: p = 20 3.1e-14
// and 3.6e-14, p = 50 1.04e-13 and 1.17e-13, p = 80 1.77e-13 and 1.82e-13).
//
// A CTA solves two columns of L^{-1} by forward substitution in blocks of 32 rows: a warp per column
// solves the block's triangle with shuffles, then all threads add the block's columns of L to the
// running sums of the rows below.  A step per 32 rows instead of one barrier per row; two columns share
// the reads of L, and more would leave the last SMs idle (the FP64 rate bounds it: p^3 / 6 FMAs).
constexpr int kFacThreads = 256;
constexpr int kFacCols = 2;
// Up to this many variables L is read in place (L1 and L2 take the scattered reads, and a batch's
// problems share one launch); above it a permuted copy, read in rows, is worth its launch of 3 us.
constexpr int kFacGather = 128;

// The ordering ran to its end (a single fit's may have been handed over to the tile kernels; of a batch that ran out of time some may not have: their orders are not
// read).
__device__ __forceinline__ bool ordered(const Fit& f) {
    const volatile Ctl* c = f.ctl;
    return c->status == 0 && c->it == 0 && (f.p == 1 || c->waves > 0);
}

// The factor in causal order: cmat[k p + i] = L[i][k] d_k, i >= k.
__global__ void __launch_bounds__(kFacThreads) k_factor_order(Fit f) {
    const int p = f.p, k = blockIdx.y, i = blockIdx.x * kFacThreads + threadIdx.x;
    if (i < p && i >= k && ordered(f)) f.cmat[size_t(k) * p + i] = f.rmat[size_t(k) * p + f.order[i]];
}

template <bool GATHER>
__device__ __forceinline__ void factor_columns(const Fit& f, int j0, double* y /* [kFacCols][p] */) {
    __shared__ double s_z[kFacCols][32];   // the block's y_k / d_k
    const int p = f.p, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const double* L = GATHER ? f.rmat : f.cmat;
    const int nc = min(kFacCols, p - j0);
    for (int i = tid; i < kFacCols * p; i += kFacThreads) y[i] = 0.0;
    if (tid < kFacCols * 32) s_z[tid >> 5][tid & 31] = 0.0;
    __syncthreads();
    for (int k0 = j0 / 32 * 32; k0 < p; k0 += 32) {
        const int kn = min(32, p - k0);
        if (wid < nc) {
            // rows k0 + lane: y_i = [i = j] - sum_{k < i} L[i][k] d_k (y_k / d_k)
            const int i = k0 + lane, at = GATHER && lane < kn ? f.order[i] : i;
            double l[32];
#pragma unroll
            for (int k = 0; k < 32; ++k) l[k] = k < lane && lane < kn ? L[size_t(k0 + k) * p + at] : 0.0;
            const double inv = i < p - 1 ? 1.0 / L[size_t(i) * p + at] : 0.0;
#pragma unroll
            for (int k = 0; k < 32; ++k) l[k] *= __shfl_sync(0xffffffffu, inv, k);
            double r = lane < kn ? (i == j0 + wid ? 1.0 : 0.0) - y[wid * p + i] : 0.0;
#pragma unroll
            for (int k = 0; k < 32; ++k) r = fma(-l[k], __shfl_sync(0xffffffffu, r, k), r);
            if (lane < kn) y[wid * p + i] = r;
            s_z[wid][lane] = r * inv;
        }
        __syncthreads();
        for (int i = k0 + 32 + tid; i < p; i += kFacThreads) {
            const int at = GATHER ? f.order[i] : i;
            double s[kFacCols] = {};
#pragma unroll
            for (int kk = 0; kk < 32; kk += 16) {
                double l[16];
#pragma unroll
                for (int k = 0; k < 16; ++k) l[k] = L[size_t(k0 + kk + k) * p + at];
#pragma unroll
                for (int k = 0; k < 16; ++k)
#pragma unroll
                    for (int c = 0; c < kFacCols; ++c) s[c] = fma(l[k], s_z[c][kk + k], s[c]);
            }
#pragma unroll
            for (int c = 0; c < kFacCols; ++c) y[c * p + i] += s[c];
        }
        __syncthreads();
    }
    for (int c = 0; c < nc; ++c) {
        const int j = j0 + c, vj = f.order[j];
        const double inv = 1.0 / f.sd[vj];
        for (int i = tid; i < p; i += kFacThreads) {
            const int vi = f.order[i];
            f.bout[size_t(vi) * p + vj] = i > j ? -y[c * p + i] * (f.sd[vi] * inv) : 0.0;
        }
    }
}
template <bool GATHER>
__global__ void __launch_bounds__(kFacThreads) k_factor_B(Fit f) {
    extern __shared__ double sm_fac[];
    if (!ordered(f)) return;
    factor_columns<GATHER>(f, blockIdx.x * kFacCols, sm_fac);
}
// Problems of a batch with p <= kFacGather (the others, and those of bad status, are left out).
__global__ void __launch_bounds__(kFacThreads) k_factor_B_batch(const Fit* __restrict__ fits) {
    extern __shared__ double sm_fac[];
    const Fit& f = fits[blockIdx.x];
    if (f.p > kFacGather || int(blockIdx.y) * kFacCols >= f.p || !ordered(f)) return;
    factor_columns<true>(f, blockIdx.y * kFacCols, sm_fac);
}

cudaError_t launch_factor_B(const Fit& f, cudaStream_t st, long long* launches) {
    const int p = f.p, grid = (p + kFacCols - 1) / kFacCols;
    const size_t smem = size_t(kFacCols) * p * sizeof(double);
    if (launches) *launches += p <= kFacGather ? 1 : 2;
    if (p <= kFacGather) {
        k_factor_B<true><<<grid, kFacThreads, smem, st>>>(f);
        return cudaGetLastError();
    }
    k_factor_order<<<dim3((p + kFacThreads - 1) / kFacThreads, p), kFacThreads, 0, st>>>(f);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    e = ensure_smem_attr(reinterpret_cast<const void*>(k_factor_B<false>), smem);
    if (e != cudaSuccess) return e;
    k_factor_B<false><<<grid, kFacThreads, smem, st>>>(f);
    return cudaGetLastError();
}

cudaError_t launch_factor_B_batch(const Fit* fits_dev, const int* p_host, int count, const Fit* fits_host, cudaStream_t st) {
    int pmax = 0;
    for (int k = 0; k < count; ++k)
        if (p_host[k] <= kFacGather) pmax = std::max(pmax, p_host[k]);
    if (pmax > 0) {
        k_factor_B_batch<<<dim3(count, (pmax + kFacCols - 1) / kFacCols), kFacThreads, size_t(kFacCols) * pmax * sizeof(double), st>>>(
            fits_dev);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    for (int k = 0; k < count; ++k)
        if (p_host[k] > kFacGather) {
            const cudaError_t e = launch_factor_B(fits_host[k], st, nullptr);
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

cudaError_t launch_fit_B_batch(const Fit* fits_dev, const int* p_host, int count, const Fit* fits_host,
                               cudaStream_t st) {
    int pmax_small = 0;
    for (int k = 0; k < count; ++k)
        if (p_host[k] <= kBSmall && p_host[k] > pmax_small) pmax_small = p_host[k];
    if (pmax_small > 0) {
        const size_t smem = size_t(pmax_small) * pmax_small * sizeof(double);
        cudaError_t e = ensure_smem_attr(reinterpret_cast<const void*>(k_bfit_small), smem);
        if (e != cudaSuccess) return e;
        k_bfit_small<<<count, kBThreads, smem, st>>>(fits_dev, count);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    for (int k = 0; k < count; ++k)
        if (p_host[k] > kBSmall) {
            const cudaError_t e = launch_fit_B(fits_host[k], st);
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

cudaError_t launch_fit_B(const Fit& f, cudaStream_t st) {
    const int p = f.p;
    dim3 g2((p + 15) / 16, (p + 15) / 16);
    k_perm_cov<<<g2, 256, 0, st>>>(f);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    int dev = 0, nsm = 0, per_sm = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_chol_coop, kCholThreads, 0)) != cudaSuccess)
        return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    if ((e = cudaMemsetAsync(f.scratch, 0, size_t(p) * sizeof(int), st)) != cudaSuccess) return e;   // row flags
    {
        // one CTA per SM at most (co-resident: cooperative launch), no more than rows
        const int grid = std::max(1, std::min(nsm, p));
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(grid);
        cfg.blockDim = dim3(kCholThreads);
        cfg.dynamicSmemBytes = 0;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if ((e = cudaLaunchKernelEx(&cfg, k_chol_coop, f)) != cudaSuccess) return e;
    }
    const size_t smem = (p <= kTriThreads * kTriPer ? 2 : 1) * size_t(p) * sizeof(double);
    e = ensure_smem_attr(reinterpret_cast<const void*>(k_tri_inv), smem);
    if (e != cudaSuccess) return e;
    k_tri_inv<<<p, kTriThreads, smem, st>>>(f);
    k_B_out<<<g2, 256, 0, st>>>(f);
    return cudaGetLastError();
}

}  // namespace lingam
