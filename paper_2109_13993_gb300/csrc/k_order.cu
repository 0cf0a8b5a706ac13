// k_order.cu -- the ordering loop (Algorithm 3: ParaFindRoot, UpdateData, UpdateCovMat) of one
// problem, or of many at once, in one persistent cooperative launch.
//
// A problem is worked on by a group of CTAs: one lane of control, the group's rank 0 (the
// "controller"), and the workers (the other CTAs; in groups below kDedicated CTAs rank 0 works
// too).  A single fit's group is the whole grid; a batch's problems get groups sized by their
// work, and small ones queue for groups of one.  Groups never wait for each other.
//
// Which pairs are compared.  As in the tile kernels, a wave completes up to kMaxCols candidates
// (the columns) against every variable that was not a column yet (the rows), and the lowest
// complete score bounds the root's score exactly (threshold, Sec. III-B).  Two things keep the
// waves few and narrow:
//   - every variable remembers the partner that contributed most to its score (its killer).  The
//     first wave of an iteration also compares each row with its killer, which alone nearly
//     always puts the row's partial score above the bound: one pair instead of a column;
//   - candidates are taken in the order of their last known score without the contribution of
//     the variable just removed, so that the children of the removed root come first.
// Neither changes the root: a partial score is a lower bound of the score whatever pairs it holds.
// Where they leave most pairs to compare, a single fit goes on in the tile kernels (kHandCols).
// Pairs evaluated, of all pairs: p = 300, n = 5000 graphs with one causal order 82 % -> 6 %, p = 1000,
// n = 10^4 79 % -> 1.7 %, random graphs of in-degree 3 at p = 300 31 % -> 19 %, with 1.0-1.7 waves per
// iteration instead of 1.4-8.9.  Whole fits against the tile kernels with a barrier per phase:
// p = 1000, n = 10^4 1145 -> 66 ms (a random graph 589 -> 567), p = 300, n = 5000 56 -> 9.2 ms,
// p = 100, n = 10^4 11.1 -> 2.8, p = 20, n = 2000 1.23 -> 0.51 ms; FP64 p = 65, n = 2001 72 -> 4.3 ms.
//
// One hand-over per wave.  The first wave of an iteration removes the previous root on the way:
// a worker reads the old rows, forms (x_w - Sigma[w,root] x_root) / sqrt(1 - Sigma[w,root]^2) of
// the rows, columns and killers it needs in registers and shared memory, and writes the rows it
// owns to the other of two copies; the pair coefficients come from the old covariance the same
// way, and the covariance downdate itself (Eq. CovUpdate, FP64, upper triangle) goes to its other
// copy.  So no barrier separates removal and comparison: the workers arrive once per wave, the
// controller merges, decides and publishes the next wave in one word.  The removed root's column of
// the covariance stays behind in Fit::rmat, the factorisation that the B fit solves with.
//
// Work split of a wave: nseg segments of the sample axis times W / nseg row groups; a worker
// stages its segment of the columns (and of the root) in shared memory and streams its rows from
// L2.  A warp takes a unit of samples of one row against four columns (one on the FP64 path; lanes
// across the samples, coalesced), closes it with one lg2 per residual and lane and adds the lanes in a
// fixed tree; the units and segments are added in order in float-float (the last worker of a row
// group to arrive adds the segments), so that a sum does not depend on how the units were spread over
// warps and CTAs (beyond 2^-48).
//
// What bounds it.  Small fits: the chain of a wave, about 60,000 clocks of which the two flags take
// 2,000-2,800 each (a word written by one SM and read by another costs 1,100-1,500), the row table 4,500,
// coefficients 6,000, staging 3,000, the units 6,000-12,000, the controller 15,000.  Large ones: the
// units, at 60 % of the exponentials' rate with four warps a quarter (1024 samples of a row against
// four columns 13,700 clocks; 8,200 at 32 ex2 a clock and SM), and a row's own unit at 40 %.
#include <algorithm>
#include <queue>
#include <type_traits>
#include <utility>
#include <vector>

#include "common.cuh"
#include "launch.h"
#include "pair_math.cuh"

namespace lingam {

constexpr int kMaxCols = 16;     // columns of a wave at most (four quads)
// A unit of a warp's work is 1024 samples or less (Fit::unit) on the FP32 path (up to 32 per lane, one
// lg2 per residual), 256 or less on the FP64 path, of one row against quad() columns: four on the FP32
// path (the row's reads serve four pairs), one on the FP64 path, where a warp alone has only its SM
// quarter's FP64 unit.  max_unit: what the shared memory is sized for.
template <class T>
__host__ __device__ constexpr int max_unit() { return sizeof(T) == 4 ? 1024 : 256; }
template <class T>
__host__ __device__ constexpr int quad() { return sizeof(T) == 4 ? 4 : 1; }
constexpr int kRowBatch = 32;    // rows of a worker between two CTA barriers
// A single fit on the mixed path is left to the tile kernels once kHandIters iterations in a row (after the
// first) took kHandCols columns or more: killer pairs do not help there, and 32-column waves are cheaper.
// The time of the rest of a fit, tile kernels over this one, by the columns an iteration takes: pure noise
// 300 x 500 0.94 at 165 columns, 300 x 5000 0.98 at 176, 500 x 1000 0.78 at 310 and 1.00 at 133, 1000 x 4000
// 0.67 at 681 and 0.96 at 193; random graphs 1000 x 1300 0.97 at 178 and 1.01 at 157, 1000 x 10000 0.98 at
// 207 and 1.01 at 181, 2000 x 2300 0.70 at 375.
constexpr int kHandCols = 176;
constexpr int kHandIters = 4;
constexpr int kDedicated = 8;    // groups of this many CTAs or more have a controller that does not work

extern __shared__ __align__(128) unsigned char smem_order[];

template <class T>
struct OrderTraits;
template <>
struct OrderTraits<float> {
    using V = float4;                      // consecutive samples of a lane
    using Sum = float2;                    // float-float sum
    static constexpr int VN = 4;
};
template <>
struct OrderTraits<double> {
    using V = double2;
    using Sum = double;
    static constexpr int VN = 2;
};

// A row of the current wave (rows 0 .. ncol - 1 are its columns).
struct __align__(16) RowEnt {
    int var;       // variable
    float off;     // its 32-sample log-cosh offset (FP32 path)
    int kvar;      // its killer (-1: none)
    float koff;    // the killer's offset
};
static_assert(sizeof(RowEnt) == 16, "one 16-byte load");

__device__ __forceinline__ RowEnt load_row(const RowEnt* t) {
    const int4 v = __ldcg(reinterpret_cast<const int4*>(t));
    return RowEnt{v.x, __int_as_float(v.y), v.z, __int_as_float(v.w)};
}

// The wave word: sequence number (bits 51-63), done (50), removal (49), killers (48), columns
// (43-47), rows (30-42), the root to remove (16-29), segments (0-15).
struct OrderWave {
    int done, removal, kill, ncol, nrow, nseg, root;
};
__device__ __forceinline__ unsigned long long pack_order_wave(unsigned seq, const OrderWave& w) {
    return (static_cast<unsigned long long>(seq & 0x1fffu) << 51) | (static_cast<unsigned long long>(w.done) << 50) |
           (static_cast<unsigned long long>(w.removal) << 49) | (static_cast<unsigned long long>(w.kill) << 48) |
           (static_cast<unsigned long long>(w.ncol) << 43) | (static_cast<unsigned long long>(w.nrow) << 30) |
           (static_cast<unsigned long long>(w.root & 0x3fff) << 16) | static_cast<unsigned long long>(w.nseg);
}
__device__ __forceinline__ OrderWave unpack_order_wave(unsigned long long w) {
    return {int((w >> 50) & 1), int((w >> 49) & 1), int((w >> 48) & 1), int((w >> 43) & 31), int((w >> 30) & 0x1fff),
            int(w & 0xffff), int((w >> 16) & 0x3fff)};
}

// ------------------------------------------------------------------ sums
__device__ __forceinline__ float2 sum_of(float v) { return make_float2(v, 0.f); }
__device__ __forceinline__ double sum_of(double v) { return v; }
__device__ __forceinline__ float2 sum_add(float2 a, float2 b) { return ff_add(a, b); }
__device__ __forceinline__ double sum_add(double a, double b) { return a + b; }
__device__ __forceinline__ float sum_val(float2 a) { return a.x + a.y; }
__device__ __forceinline__ double sum_val(double a) { return a; }
__device__ __forceinline__ float2 shfl_xor_sum(float2 v, int o) {
    return make_float2(__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o));
}
__device__ __forceinline__ double shfl_xor_sum(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }

// The 32 lanes' sums of N values (a power of two up to 16), in a fixed tree; lane l ends with the
// total of value lane_value<N>(l).
template <int N, class T>
__device__ __forceinline__ T lane_totals(T (&v)[N]) {
    const int lane = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int h = N / 2; h >= 1; h >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const T keep = up ? v[i + h] : v[i], send = up ? v[i] : v[i + h];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
        o >>= 1;
    }
    T s = v[0];
    for (; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}
template <int N>
__device__ __forceinline__ int lane_value() {
    const int lane = threadIdx.x & 31;
    int idx = 0, o = 16;
#pragma unroll
    for (int h = N / 2; h >= 1; h >>= 1) {
        idx += (lane & o) ? h : 0;
        o >>= 1;
    }
    return idx;
}

// ------------------------------------------------------------------ sample blocks
__device__ __forceinline__ float4 reduce_root(float4 a, float4 r, float c, float inv) {
    return make_float4(fmaf(-c, r.x, a.x) * inv, fmaf(-c, r.y, a.y) * inv, fmaf(-c, r.z, a.z) * inv,
                       fmaf(-c, r.w, a.w) * inv);
}
__device__ __forceinline__ double2 reduce_root(double2 a, double2 r, double c, double inv) {
    return make_double2(fma(-c, r.x, a.x) * inv, fma(-c, r.y, a.y) * inv);
}
__device__ __forceinline__ float4 zero_of(float4) { return make_float4(0.f, 0.f, 0.f, 0.f); }
__device__ __forceinline__ double2 zero_of(double2) { return make_double2(0.0, 0.0); }

// Moments of one residual over a lane's samples of a block.
struct AccD {
    double A, P, G;
};
template <class T>
struct AccOf;
template <>
struct AccOf<float> {
    using Acc = Acc2;
};
template <>
struct AccOf<double> {
    using Acc = AccD;
};
__device__ __forceinline__ void acc_start(Acc2& a) { acc_init(a); }
__device__ __forceinline__ void acc_start(AccD& a) {
    a.A = 0.0;
    a.P = 1.0;
    a.G = 0.0;
}
// FP64 exponentials.  DFMA runs at 1.7 lanes a clock and SM on this part, so the operations of an
// exponential are counted: e^{-c w}, w >= 0, by the table-driven method (Tang, "Table-driven
// implementation of the exponential function in IEEE floating-point arithmetic", ACM TOMS 1989):
// c w = -k ln2 / 256 + c r with k the nearest integer (<= 0), e^{-c w} = 2^{k/256} e^{-c r}, the
// table 2^{j/256} in shared memory and a polynomial of degree 4 in r (|c r| <= ln2 / 512: its error is
// below 2^-54).  Eight FP64 operations, against about sixty of the library's exp().  The argument is
// reduced with one constant: an absolute error below 2^-53 c w e^{-c w}, and the terms are summed.
constexpr int kExpTab = 256;
__device__ __forceinline__ double exp_neg(double w, const double c, const double* tab) {
    const double kln2 = 0.69314718055994530942;
    const double magic = 6755399441055744.0;   // 1.5 2^52: rounds to an integer in the low word
    const double t = fma(w, -c * (kExpTab / kln2), magic);
    const int k = __double2loint(t);
    const double r = fma(t - magic, kln2 / kExpTab / c, w);
    double h = fma(r, c * c * c * c / 24.0, -c * c * c / 6.0);
    h = fma(r, h, c * c / 2.0);
    h = fma(r, h, -c);
    h = r * h;
    const double e = tab[k & (kExpTab - 1)];
    // times 2^(k >> 8) in the exponent field; zero below about e^-700 (c w >= 700)
    const int big = __double2hiint(w) >= (c > 1.0 ? 0x4075e000 : 0x4095e000);   // 350, 1400
    const double s = __hiloint2double(big ? 0 : __double2hiint(e) + (k >> 8) * (1 << 20), big ? 0 : __double2loint(e));
    return fma(s, h, s);
}
__device__ __forceinline__ void acc_one(AccD& s, double u, const double* tab) {
    const double a = fabs(u);
    s.P = fma(s.P, exp_neg(a, 2.0, tab), s.P);
    s.A += a;
    s.G = fma(u, exp_neg(u * u, 0.5, tab), s.G);
}
// Both residuals of a pair: s x_i - sr x_j and s x_j - sr x_i.
__device__ __forceinline__ void acc_pair(Acc2& aa, Acc2& ab, float4 xi, float4 xj, float s, float sr, const double*) {
    acc_pair4(aa, ab, xi, xj, make_float2(s, s), make_float2(-sr, -sr));
}
__device__ __forceinline__ void acc_pair(AccD& aa, AccD& ab, double2 xi, double2 xj, double s, double sr,
                                         const double* tab) {
    acc_one(aa, fma(s, xi.x, -sr * xj.x), tab);
    acc_one(ab, fma(s, xj.x, -sr * xi.x), tab);
    acc_one(aa, fma(s, xi.y, -sr * xj.y), tab);
    acc_one(ab, fma(s, xj.y, -sr * xi.y), tab);
}
// The variable itself (its own moments).
__device__ __forceinline__ void acc_self(Acc2& a, float4 x, const double*) {
    const float2 k = make_float2(kScale, kScale);
    acc2_add(a, __fmul2_rn(k, make_float2(x.x, x.y)));
    acc2_add(a, __fmul2_rn(k, make_float2(x.z, x.w)));
}
__device__ __forceinline__ void acc_self(AccD& a, double2 x, const double* tab) {
    acc_one(a, x.x, tab);
    acc_one(a, x.y, tab);
}
// Closes a warp's unit: per residual i the lanes' centred log-cosh sum and their sum of u e^{-u^2/2}
// (FP32: of u' = kScale u), totals 2 i and 2 i + 1 in lane order (lane_value<2 N>).  off is the offset
// of 32 samples and part the lane's share of them; its low mantissa bits are zero (var_offset), so
// that the product is exact.  FP32: one lg2 per residual and lane.  FP64: the lanes' products are
// multiplied first (at most 2^256 for 8 samples a lane) and each log is taken once per warp.
template <int N>
__device__ __forceinline__ float close_unit(const Acc2 (&a)[N], const float (&off)[N], float part) {
    float v[2 * N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        v[2 * i] = fmaf(float(kLn2), lg2_approx(a[i].P.x * a[i].P.y), fmaf(a[i].A.x + a[i].A.y, kInvScale / -kC3, off[i] * part));
        v[2 * i + 1] = a[i].G.x + a[i].G.y;
    }
    return lane_totals<2 * N>(v);
}
template <int N>
__device__ __forceinline__ double close_unit(const AccD (&a)[N], const double (&off)[N], double part) {
    double v[2 * N], pr[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        v[2 * i] = fma(off[i], part, a[i].A);
        v[2 * i + 1] = a[i].G;
        pr[i] = a[i].P;
    }
    const int lane = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int h = N / 2; h >= 1; h >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const double keep = up ? pr[i + h] : pr[i], send = up ? pr[i] : pr[i + h];
            pr[i] = keep * __shfl_xor_sync(0xffffffffu, send, o);
        }
        o >>= 1;
    }
    const int odd = o;   // this bit of the lane tells a total's kind: 0 the log-cosh sum, else the other
    double q = pr[0];
    for (; o > 0; o >>= 1) q *= __shfl_xor_sync(0xffffffffu, q, o);
    const double lg = log(q);
    return lane_totals<2 * N>(v) + ((lane & odd) ? 0.0 : lg);
}
__device__ __forceinline__ float pair_scale(double om, float) { return kScale / sqrtf(float(om)); }
__device__ __forceinline__ double pair_scale(double om, double) { return 1.0 / sqrt(om); }
// The 32-sample offset of the log-cosh sums: the variable's (FP32), beta's (FP64).
__device__ __forceinline__ float pair_offset(float off, float) { return off; }
__device__ __forceinline__ double pair_offset(float, double) { return -double(kSub) * (kLn2 + kBeta); }

// One unit of one row against Q columns: the 4 Q sums (per pair the row's residual's two, then the
// column's two) in lane order.  m steps of 32 V's; xg the old row at this lane, rs the staged root,
// cs the staged columns (cstr elements apart), all at this lane's first sample.  The row is loaded two
// steps ahead.  (One copy of the step's code: the kernel's size counts, every wave runs through most
// of it once.)
template <class T, class V, int Q>
__device__ __forceinline__ T quad_unit(const V* __restrict__ xg, const V* rs, const T* cs, int cstr, int m, T c, T inv,
                                       const T* sc, T off_r, const T* offc, T part, const double* tab) {
    typename AccOf<T>::Acc acc[2 * Q];
    T s[Q], sr[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        s[q] = sc[2 * q];
        sr[q] = sc[2 * q + 1];
        acc_start(acc[2 * q]);
        acc_start(acc[2 * q + 1]);
    }
    V n0 = __ldcg(xg), n1 = n0;
    if (m > 1) n1 = __ldcg(xg + 32);
#pragma unroll 1
    for (int k = 0; k < m; ++k) {
        const V u = reduce_root(n0, rs[32 * k], c, inv);
        n0 = n1;
        if (k + 2 < m) n1 = __ldcg(xg + 32 * (k + 2));
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const V w = *(reinterpret_cast<const V*>(cs + q * cstr) + 32 * k);
            acc_pair(acc[2 * q], acc[2 * q + 1], u, w, s[q], sr[q], tab);
        }
    }
    T off[2 * Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        off[2 * q] = off_r;
        off[2 * q + 1] = offc[q];
    }
    return close_unit<2 * Q>(acc, off, part);
}

// One unit of one row on its own: the row without the root is written to its new copy with its
// moments, and compared with its killer.  Eight sums: the killer pair's four, the row's two, 0, 0.
template <class T, class V>
__device__ __forceinline__ T own_unit(const V* __restrict__ xg, const V* __restrict__ kg, const V* rs, V* __restrict__ out,
                                      int m, T c, T inv, T kc, T kinv, T s, T sr, T off_r, T off_k, T part,
                                      const double* tab) {
    typename AccOf<T>::Acc acc[4];   // the row's and the killer's residual, the row, nothing
#pragma unroll
    for (int q = 0; q < 4; ++q) acc_start(acc[q]);
    V n0 = __ldcg(xg), n1 = n0, k0 = n0, k1 = n0;
    if (m > 1) n1 = __ldcg(xg + 32);
    if (kg) {
        k0 = __ldcg(kg);
        if (m > 1) k1 = __ldcg(kg + 32);
    }
#pragma unroll 1
    for (int k = 0; k < m; ++k) {
        const V r = rs[32 * k], u = reduce_root(n0, r, c, inv), y = k0;
        n0 = n1;
        k0 = k1;
        if (k + 2 < m) {
            n1 = __ldcg(xg + 32 * (k + 2));
            if (kg) k1 = __ldcg(kg + 32 * (k + 2));
        }
        out[32 * k] = u;
        acc_self(acc[2], u, tab);
        if (kg) acc_pair(acc[0], acc[1], u, reduce_root(y, r, kc, kinv), s, sr, tab);
    }
    const T off[4] = {off_r, off_k, off_r, T(0)};
    return close_unit<4>(acc, off, part);
}

// 16 bytes from global to shared memory through L2, asynchronously.
__device__ __forceinline__ void copy16_async(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(unsigned(__cvta_generic_to_shared(dst))), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// ------------------------------------------------------------------ the group and its memory
struct Group {
    int rank, size;      // this CTA's rank in the group, CTAs of the group
    int W, wk;           // workers, this CTA's worker index (-1: the controller of a large group)
    unsigned work;       // offset of the work area in shared memory
    unsigned cap;        // bytes of the work area
    unsigned tab;        // offset of the table 2^{j/256} (FP64)
};

// Controller state per variable slot (shared memory).
constexpr size_t kSlotBytes = 16 + 8 + 4 * 10;
// A worker's tables before the staged rows: the batch's rows and the columns, the pairs'
// coefficients, the warps' sums, and the rows' and columns' coefficients and offsets.
template <class T>
__host__ __device__ constexpr int unit_slots() { return sizeof(T) == 4 ? 192 : 384; }   // units of a batch of rows
template <class T>
__host__ __device__ constexpr int slot_sums() { return 4 * quad<T>() > 8 ? 4 * quad<T>() : 8; }
template <class T>
__host__ __device__ constexpr size_t order_fixed_bytes() {
    return size_t(kRowBatch + kMaxCols) * sizeof(RowEnt) + size_t(kRowBatch) * (kMaxCols + 1) * 2 * sizeof(T) +
           size_t(unit_slots<T>()) * slot_sums<T>() * sizeof(T) +
           size_t(2 * kRowBatch + kMaxCols) * 2 * sizeof(double) +                       // S[root][v], new D
           (size_t(kRowBatch) * 6 + size_t(kMaxCols) * 4) * sizeof(T);
}
// Columns a wave may have with a work area of `cap` bytes and nrow rows: one unit of the root and
// of the columns must fit beside the fixed tables, and the controller's I table (one T per row and
// column or killer) into ctl_cap bytes.
template <class T>
__host__ __device__ inline int order_max_cols(unsigned cap, int nrow, unsigned ctl_cap) {
    for (int c = kMaxCols; c >= 4; c -= 4)
        if (unsigned(order_fixed_bytes<T>()) + unsigned((c + 1) * max_unit<T>()) * sizeof(T) <= cap &&
            unsigned((c + 1) | 1) * nrow * sizeof(T) <= ctl_cap)
            return c;
    return 0;
}
__host__ __device__ inline size_t order_state_bytes(int p) { return (size_t(p) * kSlotBytes + 127) / 128 * 128; }

// Units of a staged pass of a worker with `us` units of the sample axis: as few passes as the work area
// of `cap` bytes allows, of equal length.
template <class T>
__host__ __device__ inline int most_units(int ncol, int unit, unsigned cap) {
    const int q = quad<T>(), nq = (ncol + q - 1) / q;
    const int room = int((cap - unsigned(order_fixed_bytes<T>())) / (unsigned((nq * q + 1) * unit) * unsigned(sizeof(T))));
    const int slots = unit_slots<T>() / (nq + 1);   // one row's units at least
    return room < slots ? room : slots;
}
template <class T>
__host__ __device__ inline int pass_units(int us, int ncol, int unit, unsigned cap) {
    const int most = most_units<T>(ncol, unit, cap);
    if (us <= most) return us;
    const int passes = (us + most - 1) / most;
    return (us + passes - 1) / passes;
}
// a / b for 0 <= a < 2^16, 0 < b (the quotient in FP32 is off by less than half of 1 / b).
__device__ __forceinline__ int small_div(int a, int b) { return int(__fdividef(float(a) + 0.5f, float(b))); }

// Estimated SM clocks of a wave with nseg segments of the sample axis.  A worker evaluates its rows'
// pairs at about 5 pair-samples a clock (FP64: one in 14 clocks), stages its columns at about 40
// bytes a clock in passes of about 12,000 clocks of their own, and several segments cost an exchange
// between a row group's workers.
template <class T>
__device__ __forceinline__ float seg_cost(int nseg, int nrow, int ncol, int W, int nw, int nunit, int unit, int pass_most,
                                          int extra) {
    constexpr bool f32 = sizeof(T) == 4;
    const float groups = floorf(__fdividef(float(W) + 0.5f, float(nseg)));
    const float rows = ceilf(__fdividef(float(nrow) - 0.5f, groups)), us = ceilf(__fdividef(float(nunit) - 0.5f, float(nseg)));
    const int cols = (ncol + quad<T>() - 1) / quad<T>() * quad<T>();
    const float one = (f32 ? 1.f / 5.f : 14.f) * unit;             // a unit of one pair, at the SM's rate
    const int q = quad<T>();
    // the warps' rounds of units, each a warp's unit at a sixteenth of that rate (a quarter at most)
    const float nu = rows * us * (cols / q + extra), rounds = ceilf(__fdividef(nu, float(nw)));
    const float conc = fminf(nu, float(nw));
    const float work = fmaxf(rows * us * (float(cols) + extra * 2.f) * one, rounds * q * one * fmaxf(conc, 4.f));
    const float stage = us * (ncol + 1) * (unit * sizeof(T) / 40.f);
    const float passes = ceilf(__fdividef(us - 0.5f, float(pass_most))) * 12000.f;
    // the segments' sums: added by the last worker of each row group
    const float merge = nseg > 1 ? 4500.f + rows * (ncol + extra) * nseg * 0.3f : 0.f;
    return work + stage + passes + merge;
}

// ------------------------------------------------------------------ a worker's part of a wave

// 1 / sqrt(x) in FP64 from the FP32 value y0 (relative error e0 below 2^-21) by one step of fourth
// order: with h = 1 - x y0^2, 1/sqrt(1 - h) = 1 + h/2 + 3 h^2/8 + O(h^3), h^3 below 2^-60.
__device__ __forceinline__ double rsqrt_fast(double x) {
    const double y = double(rsqrtf(float(x)));
    const double h = fma(-x, y * y, 1.0);
    return fma(y * h, fma(h, 0.375, 0.5), y);
}

// The removal's coefficients of variable v: S the covariance of the un-normalised remaining rows and
// D their scales, 1 / sqrt(S[v][v]) (row = residual times D, so Sigma[v][w] = S[v][w] D[v] D[w]); with
// rho = S[v][root] D[v] D[root], the normalised row loses rho times the root's and is scaled by
// 1 / sqrt(1 - rho^2) = D_new / D.
struct Removal {
    double rho, inv;
};

// Four totals of a record.
__device__ __forceinline__ void load4(float (&v)[4], const float* p) {
    const float4 a = __ldcg(reinterpret_cast<const float4*>(p));
    v[0] = a.x;
    v[1] = a.y;
    v[2] = a.z;
    v[3] = a.w;
}
__device__ __forceinline__ void load4(double (&v)[4], const double* p) {
    const double2 a = __ldcg(reinterpret_cast<const double2*>(p)), b = __ldcg(reinterpret_cast<const double2*>(p) + 1);
    v[0] = a.x;
    v[1] = a.y;
    v[2] = b.x;
    v[3] = b.y;
}

// A pair's measure from its four sums and the two variables' statistics.
__device__ __forceinline__ float measure_of(const Fit& f, const float (&v)[4], float4 si, float4 sj) {
    return pair_measure_f(v[0], v[1], v[2], v[3], si, sj, __frcp_rn(float(f.n)));
}
__device__ __forceinline__ double measure_of(const Fit& f, const double (&v)[4], double hi, double hj) {
    const double pad = double(f.ld - f.n) * kBeta;
    return (hj - hi) + (hterm_inv(v[0] + pad, v[1], f.inv_n) - hterm_inv(v[2] + pad, v[3], f.inv_n));
}
// The statistics of the rows of a wave without a removal, in the order of its table.
__device__ __forceinline__ float4* row_stats(const Fit& f, float) { return f.vstat; }
__device__ __forceinline__ double* row_stats(const Fit& f, double) { return f.hx; }
// The pitch of such a wave's measures.
__device__ __forceinline__ int measure_pitch(int ncol) { return (ncol + 3) & ~3; }

// Total t of row e: sum v of its record; four consecutive lanes have a pair's.  A removal's are left as
// they are (its new statistics are not known to every worker).  Otherwise they are pair (e, column
// v / 4)'s, and its measure is left: a quarter of what the controller would read, and no work of its own
// per pair (16 columns: 8,400 -> 3,600 clocks with 300 rows, 36,000 -> 12,000 with 565).
template <class T>
__device__ __forceinline__ void close_total(const Fit& f, const OrderWave& wv, T* tot, T t, int e, int v) {
    if (wv.removal) {
        constexpr int Q = quad<T>();
        tot[e * (4 * Q * ((wv.ncol + Q - 1) / Q) + 8) + v] = t;
    } else {
        const int lane = threadIdx.x & 31, c = v >> 2;
        T m[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) m[i] = __shfl_sync(0xfu << (lane & 28), t, (lane & 28) + i);
        if ((v & 3) == 0 && c < wv.ncol) {
            T x = T(0);
            if (f.reuse ? e >= wv.ncol || c < e : e != c) {
                const auto* st = row_stats(f, T());
                x = measure_of(f, m, __ldcg(st + e), __ldcg(st + c));
                if (!isfinite(x)) set_status(f.ctl, LINGAM_EDEGENERATE);
            }
            tot[e * measure_pitch(wv.ncol) + c] = x;
        }
    }
}

template <class T, int NT>
__device__ __noinline__ void worker_wave(const Fit& f, const OrderWave wv, const Group g, const T* __restrict__ xold,
                                         T* __restrict__ xnew, const double* __restrict__ sold, double* __restrict__ snew,
                                         const double* __restrict__ dold, double* __restrict__ dnew) {
    using V = typename OrderTraits<T>::V;
    using Sum = typename OrderTraits<T>::Sum;
    constexpr int VN = OrderTraits<T>::VN, NW = NT / 32, STEP = 32 * VN, Q = quad<T>();
    constexpr int SLOT = slot_sums<T>();
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int p = f.p, ld = f.ld, unit = f.unit, spu = unit / STEP, nst = ld / STEP, nun = (nst + spu - 1) / spu;
    const int ncol = wv.ncol, nrow = wv.nrow, nseg = wv.nseg, nq = (ncol + Q - 1) / Q;
    const bool rm = wv.removal != 0;
    const int has_k = wv.removal;             // the rows' own units (new copy, moments, killer)
    const int ntypes = nq + has_k, RECN = 4 * Q * nq + 8 * has_k, np = ncol + has_k;
    const RowEnt* tab = static_cast<const RowEnt*>(f.rowtab);
    // the wave's sums: per segment (several segments or passes), then the totals of every row
    Sum* rec = static_cast<Sum*>(f.rec);
    T* tot_out = reinterpret_cast<T*>(rec + size_t(nseg) * nrow * RECN);
    // shared memory
    unsigned char* work = smem_order + g.work;
    RowEnt* s_row = reinterpret_cast<RowEnt*>(work);
    RowEnt* s_col = s_row + kRowBatch;
    T* s_sc = reinterpret_cast<T*>(s_col + kMaxCols);                       // [row][kMaxCols + 1][2]
    T* s_f = s_sc + kRowBatch * (kMaxCols + 1) * 2;                           // [unit][SLOT]
    // per item (row j: j; its killer: kRowBatch + j; column c: 2 kRowBatch + c): S[root][v], new D
    double* s_sr = reinterpret_cast<double*>(s_f + unit_slots<T>() * SLOT);
    double* s_dn = s_sr + 2 * kRowBatch + kMaxCols;
    T* s_rc = reinterpret_cast<T*>(s_dn + 2 * kRowBatch + kMaxCols);         // [row][4]: rho, inv, killer's
    T* s_cc = s_rc + kRowBatch * 4;                                         // [column][2]: rho, inv
    T* s_offr = s_cc + kMaxCols * 2;                                        // [row][2]: offset, killer's
    T* s_offc = s_offr + kRowBatch * 2;                                     // [column]
    T* s_root = reinterpret_cast<T*>(work + order_fixed_bytes<T>());
    const double* etab = reinterpret_cast<const double*>(smem_order + g.tab);
    const int ngr = small_div(g.W, nseg), grp = small_div(g.wk, nseg), seg = g.wk - grp * nseg;
    const int b0 = nseg == 1 ? 0 : seg * nun / nseg, b1 = nseg == 1 ? nun : (seg + 1) * nun / nseg;
    const int nr = grp < ngr && grp < nrow ? small_div(nrow - 1 - grp, ngr) + 1 : 0;
    const int bp = pass_units<T>(b1 - b0, ncol, unit, g.cap);
    const int cstr = bp * unit;
    T* s_cols = s_root + cstr;

    __shared__ double s_rcp;
    __shared__ int s_next;   // units taken from the batch, beyond a warp's first

    const int root = wv.root;
    const double droot = rm ? __ldcg(dold + root) : 0.0;

    if (nr == 0) return;

#pragma unroll 1
    for (int bs = b0; bs < b1; bs += bp) {
        const int nb = min(bp, b1 - bs);
        const int rbatch = min(kRowBatch, small_div(unit_slots<T>(), ntypes * nb));   // rows whose units have slots
#pragma unroll 1
        for (int r0 = 0; r0 < nr; r0 += rbatch) {
            const int nrb = min(rbatch, nr - r0);
            const bool stage = r0 == 0;
            if (tid < nrb) {
                const RowEnt e = load_row(tab + grp + (r0 + tid) * ngr);
                s_row[tid] = e;
                s_offr[2 * tid] = pair_offset(e.off, T());
                s_offr[2 * tid + 1] = pair_offset(e.koff, T());
            } else if (tid >= 64 && tid < 64 + kMaxCols && stage && bs == b0) {
                const int c = tid - 64;
                RowEnt e = {-1, 0.f, -1, 0.f};
                if (c < ncol) e = load_row(tab + c);
                s_col[c] = e;
                s_offc[c] = pair_offset(e.off, T());
            }
            __syncthreads();   // the tables are there; the previous batch's sums were read
            // everything that depends on the tables alone is in flight before the coefficients are
            // formed: the segment of the root and of the columns, and the covariance's elements
            const int base = bs * spu * 32, nv = min(nb * spu, nst - bs * spu) * 32;
            if (stage) {
#pragma unroll 1
                for (int t = tid; t < nv; t += NT) {
                    V* dst = reinterpret_cast<V*>(s_root) + t;
                    if (rm) copy16_async(dst, reinterpret_cast<const V*>(xold + size_t(root) * ld) + base + t);
                    else *dst = zero_of(V());
#pragma unroll 1
                    for (int c = 0; c < ncol; ++c)
                        copy16_async(reinterpret_cast<V*>(s_cols + c * cstr) + t,
                                     reinterpret_cast<const V*>(xold + size_t(s_col[c].var) * ld) + base + t);
                }
            }
            // the pairs: row j against column c (c == ncol: its killer)
            constexpr int PU = (kRowBatch * (kMaxCols + 1) + NT - 1) / NT;
            double pc[PU];
            int pu[PU];   // the pair's row and item, or -1
#pragma unroll
            for (int q = 0; q < PU; ++q) {
                const int u = tid + q * NT;
                pu[q] = -1;
                if (u < nrb * np) {
                    const int j = small_div(u, np), c = u - j * np, e = grp + (r0 + j) * ngr;
                    const bool kill = c == ncol;
                    const int vi = s_row[j].var, vj = kill ? s_row[j].kvar : s_col[c].var;
                    if (vj >= 0 && (kill || (f.reuse ? e >= ncol || c < e : e != c)) &&
                        LINGAM_INBOUNDS(f.ctl, vi >= 0 && vi < p && vj < p)) {
                        pu[q] = j | (kill ? kMaxCols : c) << 8;
                        pc[q] = __ldcg(sold + min(vi, vj) * p + max(vi, vj));
                    }
                }
            }
            // UpdateCovMat (Eq. CovUpdate) on S, FP64, upper triangle by variable index, into the other
            // copy: S[w][j] - S[w][root] S[j][root] / S[root][root] for the batch's rows w and every j >= w
            // (of a removed j the element is never read again), in chunks of 32 elements a warp; the
            // segments' workers share a row's chunks.  Four of a warp's chunks are in flight, the first here.
            const int nch = (p + 31) >> 5, mych = small_div(nch + nseg - 1 - seg, nseg);   // chunks seg, seg + nseg, ...
            int ci = small_div(wid, mych > 0 ? mych : 1), cc = wid - ci * mych;
            const bool cov = rm && bs == b0 && mych > 0;
            int cat[4], crow[4];
            double ca[4], cb[4];
            auto load_chunks = [&]() {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    cat[q] = -1;
                    if (cov && ci < nrb) {
                        const int w = s_row[ci].var, j = (seg + cc * nseg) * 32 + lane;
                        crow[q] = ci;
                        if (j >= w && j < p) {
                            cat[q] = w * p + j;   // (p <= 4096)
                            ca[q] = __ldcg(sold + cat[q]);
                            cb[q] = __ldcg(sold + min(j, root) * p + max(j, root));
                        }
                        cc += NW;
                        while (cc >= mych) {
                            cc -= mych;
                            ++ci;
                        }
                    } else {
                        crow[q] = -1;
                    }
                }
            };
            load_chunks();
            if (rm && tid == NT - 1) {   // (droot^2 for 1 / S[root][root] had B 2 to 10 % further off)
                const double srr = __ldcg(sold + root * p + root);
                s_rcp = 1.0 / srr;
                if (g.wk == 0 && r0 == 0 && bs == b0) f.rmat[size_t(p - 1 - nrow) * p + root] = srr;
            }
            // the rows', killers' and columns' removal coefficients (FP64)
            if (tid < 2 * nrb + ncol) {
                const int k = tid < nrb ? tid : tid < 2 * nrb ? kRowBatch + tid - nrb : 2 * kRowBatch + tid - 2 * nrb;
                const int v = k < kRowBatch ? s_row[k].var : k < 2 * kRowBatch ? s_row[k - kRowBatch].kvar : s_col[k - 2 * kRowBatch].var;
                double sr = 0.0, d = 0.0, rho = 0.0, inv = 1.0;
                if (v >= 0) {
                    d = __ldcg(dold + v);
                    if (rm) {
                        sr = __ldcg(sold + min(v, root) * p + max(v, root));
                        const double svv = __ldcg(sold + v * p + v);
                        rho = sr * (d * droot);
                        double om = fma(-rho, rho, 1.0);
                        if (!(om > degenerate_om(sizeof(T) == 4))) {
                            set_status(f.ctl, LINGAM_EDEGENERATE);
                            om = 1.0;
                        }
                        // the new scale from the element itself, so that no rounding is carried on from
                        // iteration to iteration (an element that cancelled to nothing: from the old scale)
                        const double left = fma(-sr * (droot * droot), sr, svv);
                        const bool own = left > 1e-30;
                        const double y = rsqrt_fast(own ? left : om);
                        inv = own ? y * (svv * d) : y;
                        d = own ? y : d * y;
                        if (k < kRowBatch && bs == 0) {   // (one worker per row: the first segment's)
                            dnew[v] = d;
                            f.rmat[size_t(p - 1 - nrow) * p + v] = sr;   // (for the B fit)
                        }
                    }
                }
                s_sr[k] = sr;
                s_dn[k] = d;
                T* rc = k < kRowBatch ? s_rc + 4 * k : k < 2 * kRowBatch ? s_rc + 4 * (k - kRowBatch) + 2 : s_cc + 2 * (k - 2 * kRowBatch);
                rc[0] = T(rho);
                rc[1] = T(inv);
            }
            __syncthreads();
            const double rcp = s_rcp;   // 1 / S[root][root]
#pragma unroll
            for (int q = 0; q < PU; ++q)
                if (pu[q] >= 0) {
                    const int j = pu[q] & 0xff, c = pu[q] >> 8, it = c == kMaxCols ? kRowBatch + j : 2 * kRowBatch + c;
                    double cv = pc[q];
                    if (rm) cv = fma(-s_sr[j] * rcp, s_sr[it], cv);
                    double rho = cv * (s_dn[j] * s_dn[it]);
                    double om = fma(-rho, rho, 1.0);
                    constexpr bool f32 = sizeof(T) == 4;
                    if (!((f32 ? double(float(om)) : om) > (f32 ? double(float(degenerate_om(true))) : degenerate_om(false)))) {
                        set_status(f.ctl, LINGAM_EDEGENERATE);
                        rho = 0.0;
                        om = 1.0;
                    }
                    const T s = pair_scale(om, T());
                    T* sc = s_sc + (j * (kMaxCols + 1) + c) * 2;
                    sc[0] = s;
                    sc[1] = s * T(rho);
                }
            while (crow[0] >= 0) {
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (cat[q] >= 0) snew[cat[q]] = fma(-s_sr[crow[q]] * rcp, cb[q], ca[q]);
                load_chunks();
            }
            if (tid == 0) s_next = 0;
            if (stage) {
                // the columns without the root (each thread the vectors it copied)
                copy_wait();
                if (rm) {
#pragma unroll 1
                    for (int t = tid; t < nv; t += NT) {
                        const V r = reinterpret_cast<const V*>(s_root)[t];
#pragma unroll 1
                        for (int c = 0; c < ncol; ++c) {
                            V* x = reinterpret_cast<V*>(s_cols + c * cstr) + t;
                            *x = reduce_root(*x, r, s_cc[2 * c], s_cc[2 * c + 1]);
                        }
                    }
                }
            }
            __syncthreads();
            // the units of all rows, first those against columns (row, quad, unit of the segment), then
            // the rows' own (the short ones last); each leaves its sums in a slot.  Dealt out to the warps in
            // turn, in a batch's CTAs, whose warps have many each, taken by the next warp that is free (64
            // uneven datasets 10.24 -> 9.92 ms; single fits gain and lose less than 1%, and the FP64 quarters
            // are loaded evenly only in turn).
            const int nQ = nrb * nq * nb, nU = nQ + nrb * has_k * nb;
            const auto next_unit = [&](int i) {
                if constexpr (sizeof(T) == 8 || NT == 512) return i + NW;
                else return NW + __shfl_sync(0xffffffffu, lane == 0 ? atomicAdd(&s_next, 1) : 0, 0);
            };
            for (int i = wid; i < nU; i = next_unit(i)) {
                const bool own = i >= nQ;
                const int g2 = small_div(own ? i - nQ : i, nb), b = (own ? i - nQ : i) - g2 * nb;   // (row, quad) or row
                const int j = own ? g2 : small_div(g2, nq), t = own ? 0 : g2 - j * nq;
                const int st0 = (bs + b) * spu, m = min(spu, nst - st0);
                const T part = T(m) * (T(VN) / T(kSub));   // a lane's samples, of 32
                const T c = s_rc[4 * j], inv = s_rc[4 * j + 1], off_r = s_offr[2 * j];
                const V* xg = reinterpret_cast<const V*>(xold + size_t(s_row[j].var) * ld) + st0 * 32 + lane;
                const V* rs = reinterpret_cast<const V*>(s_root) + b * spu * 32 + lane;
                if (!own) {
                    const T* cs = s_cols + (Q * t) * cstr + (b * spu * 32 + lane) * VN;
                    const T tot = quad_unit<T, V, Q>(xg, rs, cs, cstr, m, c, inv, s_sc + (j * (kMaxCols + 1) + Q * t) * 2,
                                                     off_r, s_offc + Q * t, part, etab);
                    if ((lane & (32 / (4 * Q) - 1)) == 0) s_f[i * SLOT + lane_value<4 * Q>()] = tot;
                } else {
                    const int kv = s_row[j].kvar;
                    const V* kg = kv >= 0 ? reinterpret_cast<const V*>(xold + size_t(kv) * ld) + st0 * 32 + lane : nullptr;
                    V* out = reinterpret_cast<V*>(xnew + size_t(s_row[j].var) * ld) + st0 * 32 + lane;
                    const T* sk = s_sc + (j * (kMaxCols + 1) + kMaxCols) * 2;
                    const T tot = own_unit<T, V>(xg, kg, rs, out, m, c, inv, s_rc[4 * j + 2], s_rc[4 * j + 3], sk[0], sk[1],
                                                 off_r, s_offr[2 * j + 1], part, etab);
                    if ((lane & 3) == 0) s_f[i * SLOT + lane_value<8>()] = tot;
                }
            }
            __syncthreads();
            // the units' sums of each (row, quad or own) in order, to the wave's records
            for (int x = tid; x < nrb * RECN; x += NT) {
                const int j = small_div(x, RECN), v = x - j * RECN;
                const int t = min(v / (4 * Q), nq), val = v - 4 * Q * t;
                const T* src = s_f + ((t < nq ? (j * nq + t) * nb : nQ + j * nb)) * SLOT + val;
                Sum s = sum_of(src[0]);
                for (int b = 1; b < nb; ++b) s = sum_add(s, sum_of(src[b * SLOT]));
                const int e = grp + (r0 + j) * ngr;
                const size_t at = (size_t(seg) * nrow + e) * RECN + v;
                if (LINGAM_INBOUNDS(f.ctl, (at + 1) * sizeof(Sum) <= f.rec_bytes)) {
                    if (bs != b0) s = sum_add(rec[at], s);
                    if (nseg > 1 || bs + bp < b1) rec[at] = s;
                    else close_total(f, wv, tot_out, sum_val(s), e, v);
                }
            }
        }
    }
    // several segments: the last of a row group's workers to get here adds them
    if (nseg > 1) {
        __shared__ int s_last;
        int* count = f.gcount + grp;
        __syncthreads();
        if (tid == 0) {
            s_last = atom_add_acq_rel(count, 1) == nseg - 1;
            if (s_last) *count = 0;   // for the next wave
        }
        __syncthreads();
        if (!s_last) return;
        for (int x = tid; x < nr * RECN; x += NT) {
            const int j = x < 0x10000 ? small_div(x, RECN) : x / RECN, v = x - j * RECN, e = grp + j * ngr;
            const Sum* src = rec + size_t(e) * RECN + v;
            const size_t stride = size_t(nrow) * RECN;
            Sum s = Sum();
            int k = 0;
            for (; k + 8 <= nseg; k += 8) {
                Sum y[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) y[q] = __ldcg(src + (k + q) * stride);
#pragma unroll
                for (int q = 0; q < 8; ++q) s = sum_add(s, y[q]);
            }
#pragma unroll 2
            for (; k < nseg; ++k) s = sum_add(s, __ldcg(src + k * stride));
            close_total(f, wv, tot_out, sum_val(s), e, v);
        }
    }
}

// ------------------------------------------------------------------ the controller
// Scores: float-float sums of FP32 contributions, or FP64.
__device__ __forceinline__ double score_out(float2 a) { return double(a.x) + double(a.y); }
__device__ __forceinline__ double score_out(double a) { return a; }
__device__ __forceinline__ float score_float(float2 a) { return a.x; }
__device__ __forceinline__ float score_float(double a) { return float(a); }
// Scores are >= 0 (or +inf): 64-bit integers in their order.
__device__ __forceinline__ long long score_key(float2 a) {
    const unsigned lo = __float_as_uint(a.y);
    const unsigned l = (lo & 0x80000000u) ? ~lo : (lo | 0x80000000u);
    return static_cast<long long>((static_cast<unsigned long long>(__float_as_uint(a.x)) << 32) | l);
}
__device__ __forceinline__ long long score_key(double a) { return __double_as_longlong(a); }
constexpr long long kMaxScore = 0x7fffffffffffffffll;
__device__ __forceinline__ float2 score_of_key(long long k, float2) {
    const unsigned l = unsigned(static_cast<unsigned long long>(k) & 0xffffffffu);
    return make_float2(__uint_as_float(unsigned(static_cast<unsigned long long>(k) >> 32)),
                       __uint_as_float((l & 0x80000000u) ? (l & 0x7fffffffu) : ~l));
}
__device__ __forceinline__ double score_of_key(long long k, double) { return __longlong_as_double(k); }
// Adds the square of a contribution.
__device__ __forceinline__ void add_square(float2& s, float m) {
    FF t;
    t.hi = s.x;
    t.lo = s.y;
    t.add_sq(m);
    s = make_float2(t.hi, t.lo);
}
__device__ __forceinline__ void add_square(double& s, double m) { s = fma(m, m, s); }

// As a float, rounded towards zero.
__device__ __forceinline__ float toward_zero(float x) { return x; }
__device__ __forceinline__ float toward_zero(double x) { return __double2float_rz(x); }

// Order-preserving bits of a float.
__device__ __forceinline__ unsigned key_bits(float x) {
    const unsigned b = __float_as_uint(x);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
constexpr unsigned kNoKey = 0xffffffffu;

// What the controller keeps between waves, the same for all its threads.
struct CtlState {
    int r, a, it, bestv;
    long long best;   // key of the iteration's lowest complete score
    double gamma;
    OrderWave wave;   // the next wave
};
struct OrderShared {
    CtlState st;
    unsigned long long word;
    int ok, nseg, npick, nswap, qnext;
    long long col[kMaxCols];      // the wave's complete scores (keys)
    unsigned ckey[16 * kMaxCols];   // select_lowest: the warps' keys and slots, the exchanges
    int cslot[16 * kMaxCols];
    int xhole[kMaxCols], xback[kMaxCols];
    long long lred[16];
    int ired[16], nkill[16];
    // to be reported once the next wave is published
    int rep_ncol, rep_nrow, rep_nw, rep_it, rep_root, rep_bestv;
    int wide;     // iterations in a row that took kHandCols columns or more
    int raised;   // the threshold schedule has raised its threshold in this fit
    long long rep_best, rep_rootpt;
};

// Barrier of the controller's first `nt` threads (a multiple of 32), and with an "or" over them.
__device__ __forceinline__ void part_bar(int nt) { asm volatile("bar.sync 1, %0;" ::"r"(nt) : "memory"); }
__device__ __forceinline__ int part_or(int nt, int v) {
    int out;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.s32 p, %1, 0;\n\tbar.red.or.pred q, 1, %2, p;\n\tselp.s32 %0, 1, 0, q;\n\t}"
        : "=r"(out)
        : "r"(v), "r"(nt)
        : "memory");
    return out;
}

// The 32-sample offset of a variable from its 2 (m - beta).
__device__ __forceinline__ float stat_offset(float y) {
    return var_offset(-float(kSub) * (float(kLn2 + kBeta) + 0.5f * y));
}

// Slots 0 .. r - 1 hold the remaining variables: first those that were columns in this iteration's
// earlier waves (a of them), then the current wave's columns, then the others; so the current
// wave's rows are the slots a .. r - 1.  Only the first nt threads take part once the pairs' measures
// are formed (two slots a thread, four warps at least): the steps are chains of short dependent
// operations, which idle warps would only slow down.
template <class T, int NT>
struct Controller {
    using Sum = typename OrderTraits<T>::Sum;
    static constexpr bool f32 = std::is_same<T, float>::value;
    static constexpr int NW = NT / 32, Q = quad<T>();
    const Fit& f;
    const Group& g;
    OrderShared& sh;
    // per slot
    float4* st;       // {corr, 2 (m - beta), g, offset} (FP32), or {H(x) - H(nu)} as a double (FP64)
    Sum* part;        // score so far; complete for columns
    float* kc;        // the killer pair's contribution of this iteration, rounded down
    float* kv0;       // the two largest known contributions, and their partners
    float* kv1;
    int* keval;       // the killer that was compared (-1: none)
    int* kp0;
    int* kp1;
    int* var;
    int* slot;        // slot of each variable
    int* fl;          // kNoRoot
    int* row;         // candidate keys of a selection
    T* I;             // the wave's pair measures
    const double* cov;     // S and the rows' scales after the last removal
    const double* scale;
    unsigned icap;
    int iters;
    bool gmode, prunes;
    int r, a, it, nt;
    // thread 0: counters
    int waves = 0;
    long long pairs = 0, total = 0, gsteps = 0;

    __device__ __forceinline__ Controller(const Fit& f_, const Group& g_, OrderShared& sh_, unsigned smem_bytes, int iters_)
        : f(f_), g(g_), sh(sh_) {
        const int p = f.p;
        st = reinterpret_cast<float4*>(smem_order);
        part = reinterpret_cast<Sum*>(st + p);
        kc = reinterpret_cast<float*>(part + p);
        kv0 = kc + p;
        kv1 = kv0 + p;
        keval = reinterpret_cast<int*>(kv1 + p);
        kp0 = keval + p;
        kp1 = kp0 + p;
        var = kp1 + p;
        slot = var + p;
        fl = slot + p;
        row = fl + p;
        const unsigned state = unsigned(order_state_bytes(p));
        I = reinterpret_cast<T*>(smem_order + state);
        icap = smem_bytes - state;
        iters = iters_;
        prunes = f.prune && f.reuse;
        gmode = f.gamma0 > 0.0 && prunes;
        r = p;
        a = it = 0;
        nt = NT;
    }
    __device__ __forceinline__ int max_cols(int nrow) const { return order_max_cols<T>(g.cap, nrow, icap); }
    __device__ __forceinline__ void bar() const { part_bar(nt); }

    // The slot of a wave's row (without pair reuse the rows are all variables, the columns first).
    __device__ __forceinline__ int row_slot(int e) const { return a + e < r ? a + e : a + e - r; }
    // Exchanges two slots, array `what` of the ten (the 4-byte arrays kc .. var, and fl, lie one after
    // another); the variables' slots are not updated.
    __device__ __forceinline__ void swap_part(int what, int x, int y) {
        if (what == 0) {
            const float4 t = st[x];
            st[x] = st[y];
            st[y] = t;
        } else if (what == 1) {
            const Sum t = part[x];
            part[x] = part[y];
            part[y] = t;
        } else {
            int* q = reinterpret_cast<int*>(kc) + (what < 9 ? what - 2 : 8) * f.p;
            const int t = q[x];
            q[x] = q[y];
            q[y] = t;
        }
    }
    // Exchanges two slots (one warp).
    __device__ __forceinline__ void swap_slots(int x, int y) {
        if (x == y) return;
        const int lane = threadIdx.x & 31;
        if (lane < 10) swap_part(lane, x, y);
        __syncwarp();
        if (lane < 2) slot[var[lane ? y : x]] = lane ? y : x;
        __syncwarp();
    }

    // The `n` slots of [lo, hi) of lowest key (row[k]: the key's bits, kNoKey not a candidate) to the
    // positions lo, lo + 1, ...; sh.npick of them.  The keys are in registers, a warp takes its lowest
    // one after another by warp minima, and with several selecting warps the first takes the lowest of
    // their lists.  drop >= 0: that slot leaves first (to position hi; not a candidate).  Ends with a
    // barrier.
    __device__ __forceinline__ void select_lowest(int lo, int hi, int n, int drop) {
        constexpr int KPT = 8;   // keys a lane; p <= 32 KPT NT / 32
        const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
        const int end = drop >= 0 ? hi + 1 : hi;
        const int sw = end - lo <= 32 * KPT ? 1 : nt >> 5;   // selecting warps
        int got = 0, pick = 0;   // lane i of the first warp: the i-th pick's slot
        if (wid == 1 && drop >= 0) swap_slots(drop, hi);   // (no key changes place)
        if (wid < sw) {
            unsigned key[KPT], b = kNoKey;   // the lane's keys, the lowest and its slot
            int at = -1;
#pragma unroll
            for (int q = 0; q < KPT; ++q) {
                const int k = lo + tid + q * 32 * sw;
                key[q] = k < end ? unsigned(row[k]) : kNoKey;
                if (key[q] < b) {
                    b = key[q];
                    at = k;
                }
            }
#pragma unroll 1
            for (; got < n; ++got) {
                const unsigned m = __reduce_min_sync(0xffffffffu, b);
                if (m == kNoKey) break;
                const int src = __ffs(__ballot_sync(0xffffffffu, b == m)) - 1;
                const int k = __shfl_sync(0xffffffffu, at, src);
                if (lane == got) {
                    pick = k;
                    sh.ckey[wid * kMaxCols + lane] = m;
                }
                if (lane == src) {
                    b = kNoKey;
#pragma unroll
                    for (int q = 0; q < KPT; ++q) {
                        const int kq = lo + tid + q * 32 * sw;
                        if (kq == k) key[q] = kNoKey;
                        if (key[q] < b) {
                            b = key[q];
                            at = kq;
                        }
                    }
                }
            }
            if (sw > 1) {
                if (lane < got) sh.cslot[wid * kMaxCols + lane] = pick;
                else if (lane < n) sh.ckey[wid * kMaxCols + lane] = kNoKey;
            }
        }
        if (sw > 1) {
            bar();
            if (wid == 0) {
                int pos = 0;   // lane w walks the ascending list of warp w
                unsigned b = lane < sw ? sh.ckey[lane * kMaxCols] : kNoKey;
#pragma unroll 1
                for (got = 0; got < n; ++got) {
                    const unsigned m = __reduce_min_sync(0xffffffffu, b);
                    if (m == kNoKey) break;
                    const int src = __ffs(__ballot_sync(0xffffffffu, b == m)) - 1;
                    const int from = __shfl_sync(0xffffffffu, pos, src);
                    if (lane == got) pick = src * kMaxCols + from;
                    if (lane == src) {
                        ++pos;
                        b = pos < n ? sh.ckey[lane * kMaxCols + pos] : kNoKey;
                    }
                }
                if (lane < got) pick = sh.cslot[pick];
            }
        }
        if (wid == 0) {
            // the picks behind the first `got` slots change places with the slots among those that
            // were not picked (as many)
            if (pick == hi && drop >= 0) pick = drop;
            const bool mine = lane < got, front = mine && pick < lo + got;
            const unsigned infront = __reduce_or_sync(0xffffffffu, front ? 1u << (pick - lo) : 0u);
            const unsigned back = __ballot_sync(0xffffffffu, mine && !front), lt = (1u << lane) - 1u;
            const unsigned holes = (got < 32 ? (1u << got) - 1u : 0xffffffffu) & ~infront;
            if (holes >> lane & 1u) sh.xhole[__popc(holes & lt)] = lo + lane;
            if (mine && !front) sh.xback[__popc(back & lt)] = pick;
            if (lane == 0) {
                sh.npick = got;
                sh.nswap = __popc(back);
            }
        }
        bar();
        const int ns = sh.nswap;
#pragma unroll 1
        for (int u = tid; u < 10 * ns; u += nt) {
            const int i = small_div(u, 10), what = u - 10 * i, x = sh.xhole[i], y = sh.xback[i];
            swap_part(what, x, y);
            if (what == 8) {   // var
                slot[var[x]] = x;
                slot[var[y]] = y;
            }
        }
        bar();
    }

    // The wave's rows, and (last of the warps) its segments.  Nothing of it is read before the CTA's
    // next barrier.
    __device__ __forceinline__ void write_wave(bool removal, bool kill, int ncol, int root) {
        const int tid = threadIdx.x, nrow = f.reuse ? r - a : r, has_k = removal ? 1 : 0;
        RowEnt* tab = static_cast<RowEnt*>(f.rowtab);
        if (tid < nt - 32) {
#pragma unroll 1
            for (int i = tid; i < nrow; i += nt - 32) {
                const int k = row_slot(i);
                RowEnt e = {var[k], st[k].w, -1, 0.f};
                if (kill) {
                    int kv = -1;
                    if (k >= ncol && !(fl[k] & kNoRoot) && kv0[k] > 0.f) {
                        kv = kp0[k];
                        if (kv >= 0 && slot[kv] < ncol) kv = -1;   // a column: compared anyway
                    }
                    keval[k] = kv;
                    if (kv >= 0) {
                        e.kvar = kv;
                        e.koff = st[slot[kv]].w;
                    }
                } else if (a == 0) {
                    keval[k] = -1;
                }
                if (a == 0) kc[k] = 0.f;
                if (LINGAM_INBOUNDS(f.ctl, i < f.p && e.var < f.p)) {
                    tab[i] = e;
                    if (!removal) {
                        if constexpr (f32) f.vstat[i] = st[k];
                        else f.hx[i] = *reinterpret_cast<const double*>(&st[k]);
                    }
                }
            }
        } else {
            const int lane = tid & 31;
            const int unit = f.unit, nun = (f.ld + unit - 1) / unit, cols = (ncol + Q - 1) / Q * Q;
            const int pm = most_units<T>(ncol, unit, g.cap);
            const unsigned recb = unsigned(4 * cols + 8 * has_k) * 8u * unsigned(nrow);
            const unsigned room = unsigned(min(f.rec_bytes, 0xffffffffull)) / recb - 1u;   // (the totals behind them)
            int most = min(min(nun, g.W), int(min(room, 0x7fffffffu)));
            if (f.split_n > 0) most = min(most, f.split_n);
            float b = INFINITY;
            int at = 1;
#pragma unroll 1
            for (int n = 1 + lane; n <= most; n += 32) {
                const float c = seg_cost<T>(n, nrow, ncol, g.W, NW, nun, unit, pm, has_k);
                if (c < b) {
                    b = c;
                    at = n;
                }
            }
            const unsigned m = __reduce_min_sync(0xffffffffu, __float_as_uint(b));
            at = __reduce_min_sync(0xffffffffu, __float_as_uint(b) == m ? at : 0x7fffffff);
            if (lane == 0) sh.st.wave = OrderWave{0, has_k, kill ? 1 : 0, ncol, nrow, at, root};
        }
    }

    // Iteration 0: every variable, most non-Gaussian first, nothing known of the pairs (all threads).
    __device__ __forceinline__ void start() {
#pragma unroll 1
        for (int v = threadIdx.x; v < f.p; v += NT) {
            var[v] = v;
            slot[v] = v;
            part[v] = Sum();
            kc[v] = kv0[v] = kv1[v] = 0.f;
            keval[v] = kp0[v] = kp1[v] = -1;
            fl[v] = f.prior && __ldcg(f.anc_cnt + v) > 0 ? kNoRoot : 0;
            const double h = __ldcg(f.hx + v);
            if constexpr (f32) {
                st[v] = __ldcg(f.vstat + v);
            } else {
                st[v] = make_float4(0.f, 0.f, 0.f, 0.f);
                *reinterpret_cast<double*>(&st[v]) = h;
            }
            row[v] = int(fl[v] ? kNoKey : key_bits(float(h)));
            f.dscale[0][v] = 1.0;
        }
        for (int k = threadIdx.x; k < kOrderSlots; k += NT) f.gcount[k] = 0;
        if (threadIdx.x == 0) sh.rep_nw = 0;
        const int cm = max_cols(r);
        new_iteration();
        __syncthreads();
        next_wave(0, -1, false, 0);
        if (r > 1) {
            next_wave(first_cols(cm, kMaxCols), -1, false, 0);
        } else {
            last_variable();
            done();
        }
    }
    __device__ __forceinline__ void new_iteration() {
        if (threadIdx.x == 0) {
            sh.st.r = r;
            sh.st.a = 0;
            sh.st.it = it;
            sh.st.best = kMaxScore;
            sh.st.bestv = -1;
            sh.st.gamma = f.gamma0;
        }
    }
    __device__ __forceinline__ void done() {
        if (threadIdx.x == 0) sh.st.wave = OrderWave{1, 0, 0, 0, 0, 0, 0};
    }

    // Algorithm 2: a single remaining variable is the root.
    __device__ __forceinline__ void last_variable() {
        if (threadIdx.x == 0) {
            f.order[it] = var[0];
            f.rep_root_score[it] = 0.0;
            f.rep_margin[it] = INFINITY;
            f.rep_pairs[it] = 0;
            if (f.timing) f.prev[it] = 0.0;   // no wave, so no time of its own
        }
        if (f.want_scores)
#pragma unroll 1
            for (int v = threadIdx.x; v < f.p; v += nt) f.rep_scores[size_t(it) * f.p + v] = v == var[0] ? 0.0 : NAN;
    }

    // What the next wave is, for make_wave.  drop: the slot of the root that leaves, or -1.
    int nx_n, nx_drop, nx_removal, nx_root;
    __device__ __forceinline__ void next_wave(int n, int drop, bool removal, int root) {
        nx_n = n;
        nx_drop = drop;
        nx_removal = removal;
        nx_root = root;
    }
    // The next wave: columns of lowest key (row[] holds the keys); in the first wave of an iteration
    // killers of the others.
    __device__ __forceinline__ void make_wave() {
        if (nx_n == 0 || int(threadIdx.x) >= nt) return;
        if (f.want_scores && a == 0)
#pragma unroll 1
            for (int v = threadIdx.x; v < f.p; v += nt) f.rep_scores[size_t(it) * f.p + v] = NAN;
        select_lowest(a, r, nx_n, nx_drop);
        write_wave(nx_removal, nx_removal && prunes, sh.npick, nx_root);
    }
    // Columns of an iteration's first wave.
    __device__ __forceinline__ int first_cols(int cmax, int want) const {
        const int c = min(want, cmax);
        return r - c <= 2 && r <= cmax ? r : min(c, r);   // one or two rows left over: columns as well
    }

    // The score so far, or more where the killer's pair is not part of it yet.
    __device__ __forceinline__ Sum lower_bound(int k, int an) const {
        Sum lb = part[k];
        const int ke = keval[k];
        if (ke >= 0 && slot[ke] >= an) lb = sum_add(lb, sum_of(T(kc[k])));
        return lb;
    }

    // Iteration `it` goes to the tile kernels, which start it anew: this wave has removed the last root from
    // the rows and the covariance, and its statistics are the new rows'.  By variable: what is left in U, the
    // statistics, and the scores so far (the candidates' order); see k_hand_over.
    __device__ __forceinline__ void hand_over(int an) {
#pragma unroll 1
        for (int k = threadIdx.x; k < f.p; k += nt) {
            const int v = var[k];
            f.flags[v] = k < r ? kAlive : 0;
            if (k < r) {
                f.vstat[v] = st[k];
                f.hx[v] = score_out(k < an ? part[k] : lower_bound(k, an));
            }
        }
        if (threadIdx.x == 0) f.ctl->it = it;
    }

    // One pair's measure from its four sums: row slot k against slot j.
    __device__ __forceinline__ T measure(const T (&v)[4], int k, int j) const {
        T x;
        if constexpr (f32) x = measure_of(f, v, st[k], st[j]);
        else x = measure_of(f, v, *reinterpret_cast<const double*>(&st[k]), *reinterpret_cast<const double*>(&st[j]));
        if (!isfinite(x)) set_status(f.ctl, LINGAM_EDEGENERATE);
        return x;
    }

    // After a wave: scores, threshold, and the next wave (or the root and the next iteration's
    // first wave), into sh.st.
    __device__ __forceinline__ void finish_wave(const OrderWave& wv) {
        const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
        const int ncol = wv.ncol, nrow = wv.nrow, nseg = wv.nseg, nq = (ncol + Q - 1) / Q, has_k = wv.removal;
        const int RECN = 4 * Q * nq + 8 * has_k, np = ncol + has_k, own = 4 * Q * nq, ip = np | 1;   // (ip: I's pitch)
        r = sh.st.r;
        a = sh.st.a;
        it = sh.st.it;
        next_wave(0, -1, false, 0);
        const int nw = min(NW, max(4, ncol > 8 ? (r + 31) >> 5 : (r + 63) >> 6));
        nt = 32 * nw;
        const T* tot = reinterpret_cast<const T*>(static_cast<const Sum*>(f.rec) + size_t(nseg) * nrow * RECN);
        // 1. the rows' own statistics (removal: of the new rows) and I of every pair.  Units: the rows'
        //    statistics first, then row e against column c or its killer (c = ncol); a thread has four
        //    units' totals in flight.  Without a removal the workers have left the measures.
        const int stats = has_k ? nrow : 0, units = has_k ? stats + nrow * np : 0;
        if (!has_k) {
            const int w4 = measure_pitch(ncol) / 4, n4 = nrow * w4;
#pragma unroll 1
            for (int u0 = 0; u0 < n4; u0 += 4 * NT) {
                T v[4][4];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (u0 + q * NT + tid < n4) load4(v[q], tot + 4 * (u0 + q * NT + tid));
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int u = u0 + q * NT + tid;
                    if (u < n4) {
                        const int e = small_div(u, w4), c = 4 * (u - e * w4);
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            if (c + i < ncol) I[e * ip + c + i] = v[q][i];
                    }
                }
            }
        }
#pragma unroll 1
        for (int u0 = 0; u0 < units; u0 += 4 * NT) {
            T v[4][4];
            int kj[4], es[4];   // the partner's slot (-1: nothing to do), the row
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int u = u0 + q * NT + tid;
                kj[q] = -1;
                if (u0 + q * NT < units) {   // (the same for every thread)
                    int at = 0;
                    es[q] = u;
                    if (u < stats) {
                        kj[q] = 0;
                        at = u * RECN + own + 4;
                    } else if (u < units) {
                        const int e = small_div(u - stats, np), c = u - stats - e * np;
                        es[q] = e;
                        at = e * RECN + (c < ncol ? 4 * c : own);
                        if (c < ncol) {
                            if (f.reuse ? e >= ncol || c < e : e != c) kj[q] = a + c;
                        } else {
                            const int kv = keval[a + e];
                            if (kv >= 0) kj[q] = slot[kv];
                        }
                    }
                    if (kj[q] >= 0) load4(v[q], tot + at);
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int u = u0 + q * NT + tid;
                if (u0 + q * NT < stats && u < stats) {
                    const int k = a + u;
                    if constexpr (f32) {
                        // T is centred by the old offset -32 (ln 2 + m0) over the padded row
                        const float inv_n = __frcp_rn(float(f.n));
                        const float Ts = v[q][0], off = st[k].w;
                        const float m0 = -off * (1.f / kSub) - float(kLn2);
                        const float y = 2.f * ((m0 - float(kBeta)) + fmaf(float(f.ld - f.n), m0, Ts) * inv_n);
                        st[k] = make_float4(-Ts * inv_n, y, v[q][1] * (kInvScale * inv_n), off);
                    } else {
                        *reinterpret_cast<double*>(&st[k]) = hterm_inv(v[q][0] + double(f.ld - f.n) * kBeta, v[q][1], f.inv_n);
                    }
                }
            }
            if (u0 < stats && u0 + 4 * NT >= stats) __syncthreads();   // the statistics are there
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int u = u0 + q * NT + tid;
                if (u0 + q * NT < units && u >= stats && u < units)
                    I[u - stats + es[q] * (ip - np)] = kj[q] >= 0 ? measure(v[q], row_slot(es[q]), kj[q]) : T(0);
            }
        }
        __syncthreads();
        if (tid >= nt) return;
        long long best = sh.st.best;
        int bestv = sh.st.bestv;
        // 3. rows: contributions min(0, I)^2 of the columns, of the killer, and the killers to come
        int nk = 0;   // pairs besides the columns' (distinct ones: a pair may be both's killer, and a
                      // later wave may compare a killer pair again)
#pragma unroll 1
        for (int e = tid; e < nrow && f.reuse; e += nt) {
            const int k = a + e, ke = keval[k];
            if (ke >= 0) {
                const int sk = slot[ke];
                if (keval[sk] != var[k] || var[k] < ke)
                    nk += has_k ? 1 : (sk >= a && (k < a + ncol || sk < a + ncol)) ? -1 : 0;
            }
            const T* Ir = I + e * ip;
            const int cm = min(e, ncol);
            Sum acc = Sum();
            float top = 0.f;
            int topc = -1;
            int p0 = kp0[k], p1 = kp1[k];
            float w0 = kv0[k], w1 = kv1[k];
            if (has_k && ke >= 0) {   // (keval is kp0)
                const float m = toward_zero(Ir[ncol] < T(0) ? Ir[ncol] : T(0));
                w0 = __fmul_rz(m, m);   // part of a lower bound: never more than the pair contributes
                kc[k] = w0;
            }
#pragma unroll 1
            for (int c = 0; c < cm; ++c) {
                const T m = Ir[c] < T(0) ? Ir[c] : T(0);
                add_square(acc, m);
                const float ctr = float(m) * float(m);
                const int vc = var[a + c];
                if (vc == p0) {
                    w0 = ctr;
                } else if (vc == p1) {
                    w1 = ctr;
                } else if (ctr > top) {
                    top = ctr;
                    topc = vc;
                }
            }
            if (w1 > w0) {
                const float tv = w0;
                w0 = w1;
                w1 = tv;
                const int tp = p0;
                p0 = p1;
                p1 = tp;
            }
            if (top > w0) {
                w1 = w0;
                p1 = p0;
                w0 = top;
                p0 = topc;
            } else if (top > w1) {
                w1 = top;
                p1 = topc;
            }
            kp0[k] = p0;
            kp1[k] = p1;
            kv0[k] = w0;
            kv1[k] = w1;
            part[k] = sum_add(part[k], acc);
        }
        nk = __reduce_add_sync(0xffffffffu, nk);
        if (lane == 0) sh.nkill[wid] = nk;
        bar();
        // 4. columns: max(0, I)^2 over the rows below them, a warp per column
#pragma unroll 1
        for (int c = wid; c < ncol; c += nw) {
            Sum acc = Sum();
            unsigned top = 0;
            int tope = -1;
#pragma unroll 1
            for (int e = (f.reuse ? c + 1 : 0) + lane; e < nrow; e += 32) {
                const T x = I[e * ip + c];   // (0 for the column itself)
                const T m = x > T(0) ? x : T(0);
                add_square(acc, m);
                const float ctr = float(m) * float(m);
                if (__float_as_uint(ctr) > top) {
                    top = __float_as_uint(ctr);
                    tope = e;
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc = sum_add(acc, shfl_xor_sum(acc, o));
            const unsigned m = __reduce_max_sync(0xffffffffu, top);
            const unsigned who = __ballot_sync(0xffffffffu, top == m && tope >= 0);
            if (lane == (who ? __ffs(who) - 1 : 0)) {
                const int k = a + c;
                const Sum sc = sum_add(part[k], acc);
                part[k] = sc;
                sh.col[c] = score_key(sc);
                if (f.want_scores) f.rep_scores[size_t(it) * f.p + var[k]] = score_out(sc);
                const float tv = __uint_as_float(m);
                if (who && tv > kv0[k]) {
                    const int v = var[row_slot(tope)];
                    if (v != kp0[k]) {
                        kp1[k] = kp0[k];
                        kv1[k] = kv0[k];
                        kp0[k] = v;
                    }
                    kv0[k] = tv;
                }
            }
        }
        bar();
        // 5. lowest complete score of the iteration (lowest variable index on ties); every thread
#pragma unroll 1
        for (int c = 0; c < ncol; ++c) {
            const long long kk = sh.col[c];
            const int vc = var[a + c];
            if (bestv < 0 || kk < best || (kk == best && vc < bestv)) {
                best = kk;
                bestv = vc;
            }
        }
        const int an = a + ncol;   // columned so far
        // 6. threshold: the live candidates of the others
        double gamma = gmode ? sh.st.gamma : 0.0;
        int live;
        long long thr;
#pragma unroll 1
        for (int pass = 0;; ++pass) {
            thr = gmode ? score_key(sum_from(gamma)) : best;
            int n = 0;
#pragma unroll 1
            for (int k = an + tid; k < r; k += nt) {
                const Sum lb = lower_bound(k, an);
                const bool on = !(fl[k] & kNoRoot) && !(prunes && score_key(lb) > thr);
                n += on ? 1 : 0;
                row[k] = int(on ? key_bits(score_float(lb)) : kNoKey);
            }
            live = part_or(nt, n);
            // the paper's schedule: nothing can go on and nothing finished at or below gamma: raise
            // gamma by factors gamma_c until the lowest bound of a score that may be the root's is at or
            // below it
            if (!gmode || live || best <= thr || pass > 0) break;
            long long km = best;
#pragma unroll 1
            for (int k = an + tid; k < r; k += nt)
                if (!(fl[k] & kNoRoot)) km = min(km, score_key(lower_bound(k, an)));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) km = min(km, __shfl_xor_sync(0xffffffffu, km, o));
            if (lane == 0) sh.lred[wid] = km;
            bar();
#pragma unroll 1
            for (int w = 0; w < nw; ++w) km = min(km, sh.lred[w]);
            bar();
            const double target = score_out(score_of_key(km, Sum()));
            int n2 = 0;
            while (gamma < target && n2 < 4096) {   // gamma_c > 1 and target finite: a few steps
                gamma *= f.gamma_c;
                ++n2;
            }
            if (!(score_key(sum_from(gamma)) >= km)) gamma = target;
            gsteps += n2;
            if (tid == 0 && n2 > 0) sh.raised = 1;
        }
        if (tid == 0) {
            sh.rep_ncol = ncol;
            sh.rep_nrow = nrow;
            sh.rep_nw = nw;
            sh.rep_it = -1;
        }
        if (live) {
            // (the schedule's raises cost the tile kernels more: random 1000 x 2000 from a low start 387 ms
            // here, 668 there)
            if (f32 && has_k && f.handover && sh.wide >= kHandIters && sh.raised == 0) {
                hand_over(an);
                done();
                return;
            }
            a = an;
            const int nr2 = f.reuse ? r - a : r, cm = max_cols(nr2);
            if (tid == 0) {
                sh.st.a = a;
                sh.st.best = best;
                sh.st.bestv = bestv;
                sh.st.gamma = gamma;
            }
            next_wave(min(cm, r - a), -1, false, 0);
            return;
        }
        // 7. the root, its margin, and the next iteration's candidate order
        const int root = f.has_forced ? f.forced[it] : bestv;
        const int rs = slot[root];
        long long second = kMaxScore;
        int need = 0;
#pragma unroll 1
        for (int k = tid; k < r; k += nt) {
            const Sum pk = part[k];
            const Sum lb = k < an ? pk : lower_bound(k, an);
            const int v = var[k];
            if (v != bestv && !(fl[k] & kNoRoot)) second = min(second, score_key(lb));
            // a column whose strongest pair alone would not have excluded it
            if (k < an && score_key(sum_of(T(kv0[k]))) <= thr) ++need;
            // without the root's contribution, where this iteration's last wave compared the two
            float ctr = 0.f;
            if (rs >= a && rs < an && k >= a && k != rs) {
                const int c = rs - a, e = k - a;
                const float x = e > c ? fminf(float(I[e * ip + c]), 0.f) : fmaxf(float(I[c * ip + e]), 0.f);
                ctr = x * x;
            } else if (rs >= an && keval[k] == root) {
                ctr = kc[k];
            }
            if (k == rs) sh.rep_rootpt = score_key(pk);
            if (kp0[k] == root) {
                kp0[k] = kp1[k];
                kv0[k] = kv1[k];
                kp1[k] = -1;
                kv1[k] = 0.f;
            } else if (kp1[k] == root) {
                kp1[k] = -1;
                kv1[k] = 0.f;
            }
            if (f.prior && f.prior[size_t(v) * f.p + root] == 1) {   // root was a known ancestor
                const int left = f.anc_cnt[v] - 1;
                f.anc_cnt[v] = left;
                if (left == 0) fl[k] &= ~kNoRoot;
            }
            row[k] = int(k == rs || (fl[k] & kNoRoot) ? kNoKey : key_bits(fmaxf(score_float(lb) - ctr, 0.f)));
            if constexpr (f32) st[k].w = stat_offset(st[k].y);
            part[k] = Sum();
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) second = min(second, __shfl_xor_sync(0xffffffffu, second, o));
        need = __reduce_add_sync(0xffffffffu, need);
        if (lane == 0) {
            sh.lred[wid] = second;
            sh.ired[wid] = need;
        }
        if (tid == 0) {
            sh.wide = it > 0 && an >= kHandCols ? sh.wide + 1 : 0;
            sh.rep_it = it;
            sh.rep_root = root;
            sh.rep_bestv = bestv;
            sh.rep_best = best;
        }
        bar();
        ++it;
        if (it >= iters) {
            done();
            return;
        }
        need = 0;
#pragma unroll 1
        for (int w = 0; w < nw; ++w) need += sh.ired[w];
        r -= 1;
        a = 0;
        // As many columns as this iteration would have needed, had it known its strongest pairs: whole
        // quads with one to spare on the FP32 path (a column of a started quad is free), no more on the
        // FP64 path (65 x 2001: 4.0 ms, one or two to spare 4.3 and 4.9, quads 5.3).
        const int cmax = max_cols(r), want = !prunes ? kMaxCols : f32 ? (need + 4) / 4 * 4 : max(need, 1);
        new_iteration();
        if (r == 1) {
            if (tid < 32) swap_slots(rs, 1);
            bar();
            if (tid == 0) {   // the last step of the elimination
                const int v = var[0];
                const double d = __ldcg(scale + root), dv = __ldcg(scale + v);
                const double sr = __ldcg(cov + min(v, root) * f.p + max(v, root)), rho = sr * (d * dv);
                f.rmat[size_t(f.p - 2) * f.p + v] = sr;
                f.rmat[size_t(f.p - 2) * f.p + root] = __ldcg(cov + root * f.p + root);
                if (!(fma(-rho, rho, 1.0) > 0.0)) set_status(f.ctl, LINGAM_EDEGENERATE);
            }
            last_variable();
            done();
            return;
        }
        next_wave(first_cols(cmax, want), rs, true, root);
    }

    // Thread 0, once the next wave is published: the finished wave's counts, and the finished
    // iteration's results.
    __device__ __forceinline__ void report() {
        if (sh.rep_nw == 0) return;
        const int ncol = sh.rep_ncol, nrow = sh.rep_nrow;
        pairs += f.reuse ? (long long)ncol * (ncol - 1) / 2 + (long long)ncol * (nrow - ncol) : (long long)ncol * (nrow - 1);
#pragma unroll 1
        for (int w = 0; w < sh.rep_nw; ++w) pairs += sh.nkill[w];
        ++waves;
        const int i = sh.rep_it;
        if (i >= 0) {
            long long second = kMaxScore;
#pragma unroll 1
            for (int w = 0; w < sh.rep_nw; ++w) second = min(second, sh.lred[w]);
            const double bs = score_out(score_of_key(sh.rep_best, Sum()));
            f.order[i] = sh.rep_root;
            f.rep_root_score[i] = sh.rep_root == sh.rep_bestv ? bs : score_out(score_of_key(sh.rep_rootpt, Sum()));
            f.rep_margin[i] = (second == kMaxScore ? double(INFINITY) : score_out(score_of_key(second, Sum()))) - bs;
            f.rep_pairs[i] = pairs;
            total += pairs;
            pairs = 0;
        }
        sh.rep_nw = 0;
    }

    __device__ __forceinline__ static Sum sum_from(double x) {
        if constexpr (f32) {
            const float hi = float(x);
            return make_float2(hi, isfinite(hi) ? float(x - double(hi)) : 0.f);
        } else {
            return x;
        }
    }
};

// ------------------------------------------------------------------ hand-overs (bounded waits)
__device__ __forceinline__ bool give_up(Ctl* ctl, Ctl* top, unsigned long long& t0, unsigned long long tmo) {
    if (*reinterpret_cast<volatile int*>(&top->abort)) return true;
    const unsigned long long now = global_ns();
    if (t0 == 0) {
        t0 = now;
    } else if (now - t0 > tmo) {
        set_status(ctl, LINGAM_ETIMEOUT);
        set_status(top, LINGAM_ETIMEOUT);
        top->abort = 1;
        return true;
    }
    return false;
}
// Wait until the group's workers have arrived `target` times; false: gave up (recorded).
__device__ __forceinline__ bool wait_arrivals(Ctl* ctl, Ctl* top, unsigned target, unsigned long long tmo, OrderShared& sh) {
    if (threadIdx.x == 0) {
        int ok = 1;
        unsigned long long t0 = 0;
        while (int(ld_acquire(&ctl->bar_count) - target) < 0)
            if (give_up(ctl, top, t0, tmo)) {
                ok = 0;
                break;
            }
        sh.ok = ok;
    }
    __syncthreads();
    return sh.ok != 0;
}
// Wait for wave word `seq` of the group's controller.
__device__ __forceinline__ bool wait_order_wave(Ctl* ctl, Ctl* top, unsigned seq, unsigned long long tmo, OrderShared& sh,
                                                OrderWave& wv) {
    if (threadIdx.x == 0) {
        int ok = 1;
        unsigned long long w = 0, t0 = 0;
        for (;;) {
            w = ld_acquire64(&ctl->wave_word);
            if (unsigned(w >> 51) == (seq & 0x1fffu)) break;
            if (give_up(ctl, top, t0, tmo)) {
                ok = 0;
                break;
            }
        }
        sh.word = w;
        sh.ok = ok;
    }
    __syncthreads();
    wv = unpack_order_wave(sh.word);
    return sh.ok != 0;
}

// ------------------------------------------------------------------ one problem by one group
// Returns false when the launch is to end (a wait ran out here or elsewhere).
template <class T, int NT>
__device__ __forceinline__ bool run_problem(const Fit& f, Ctl* top, int rank, int size, int iters, unsigned smem_bytes,
                                            OrderShared& sh) {
    Group g;
    g.rank = rank;
    g.size = size;
    const bool dedicated = size >= kDedicated;
    g.W = dedicated ? size - 1 : size;
    g.wk = dedicated ? rank - 1 : rank;
    g.work = dedicated ? 0u : unsigned(order_state_bytes(f.p));
    g.cap = smem_bytes - g.work;
    g.tab = smem_bytes;
    const unsigned long long tmo = *reinterpret_cast<volatile unsigned long long*>(&top->timeout_ns);
    T* xb[2] = {static_cast<T*>(f.xt), static_cast<T*>(f.xalt)};
    double* sb[2] = {f.sig, f.sigalt};
    int cur = 0;   // the copy before the next removal
    if (rank != 0) {
        for (unsigned seq = 1;; ++seq) {
            OrderWave wv;
            if (!wait_order_wave(f.ctl, top, seq, tmo, sh, wv)) return false;
            if (wv.done) return true;
            worker_wave<T, NT>(f, wv, g, xb[cur], xb[cur ^ 1], sb[cur], sb[cur ^ 1], f.dscale[cur], f.dscale[cur ^ 1]);
            if (wv.removal) cur ^= 1;
            __syncthreads();
            if (threadIdx.x == 0) atom_add_release(&f.ctl->bar_count, 1u);
        }
    }
    // the controller
    Controller<T, NT> c(f, g, sh, smem_bytes, iters);
    if (threadIdx.x == 0) {
        sh.ok = *reinterpret_cast<volatile int*>(&f.ctl->status) == 0;
        sh.rep_nw = sh.wide = sh.raised = 0;
    }
    __syncthreads();
    c.next_wave(0, -1, false, 0);
    if (sh.ok != 0) c.start();
    else c.done();
    const bool timed = f.timing && threadIdx.x == 0;
    unsigned long long tit = timed ? global_ns() : 0, tph = tit;
    unsigned arrivals = 0;
    int bad = 0;
    for (unsigned seq = 1;; ++seq) {
        c.make_wave();
        bad = __syncthreads_or(bad);   // the row table and the next wave are written
        OrderWave wv = sh.st.wave;
        if (bad) wv = OrderWave{1, 0, 0, 0, 0, 0, 0};
        if (threadIdx.x == 0) {
            if (size > 1) st_release64(&f.ctl->wave_word, pack_order_wave(seq, wv));
            const int before = sh.rep_nw ? sh.rep_it : -1;
            c.report();
            if (timed) {
                const unsigned long long t = global_ns();
                f.ctl->phase_ns[1] += t - tph;
                tph = t;
                if (before >= 0) {
                    f.prev[before] = double(t - tit) * 1e-6;
                    tit = t;
                }
            }
        }
        if (wv.done) break;
        if (!dedicated) {
            __syncthreads();   // (thread 0 has reported; the worker's tables overlay the I table)
            worker_wave<T, NT>(f, wv, g, xb[cur], xb[cur ^ 1], sb[cur], sb[cur ^ 1], f.dscale[cur], f.dscale[cur ^ 1]);
            __syncthreads();
        }
        if (wv.removal) cur ^= 1;
        arrivals += unsigned(size - 1);
        if (size > 1 && !wait_arrivals(f.ctl, top, arrivals, tmo, sh)) return false;
        if (timed) {
            const unsigned long long t = global_ns();
            f.ctl->phase_ns[0] += t - tph;
            tph = t;
        }
        // a failure recorded by a worker ends the fit (the others of a batch go on): read now, looked
        // at after the wave's work
        if (threadIdx.x == 0) bad = *reinterpret_cast<volatile int*>(&f.ctl->status);
        c.cov = sb[cur];
        c.scale = f.dscale[cur];
        c.finish_wave(wv);
    }
    if (threadIdx.x == 0) {
        f.ctl->waves = c.waves;
        f.ctl->tile_pairs = c.total;
        f.ctl->gsteps = c.gsteps;
    }
    return true;
}

// ------------------------------------------------------------------ the kernel
// one problem (fits == nullptr): every CTA of the grid is the group of `one`.  Many: assign[cta] =
// {problem, rank, group size} of this CTA's first problem (problem -1: none), then the problems of
// queue[0 .. nqueue) one after another, each by a single CTA.
template <class T, int NT>
__global__ void __launch_bounds__(NT, NT == 512 ? 1 : 2)
    k_order(const __grid_constant__ Fit one, int iters, const Fit* __restrict__ fits, const int4* __restrict__ assign,
            const int* __restrict__ queue, int nqueue, unsigned* qhead, Ctl* top, unsigned smem_bytes) {
    __shared__ OrderShared sh;
    __shared__ Fit s_fit;
    // A group's CTAs leave together, when its controller says so: a single fit's status may be set by a CTA
    // that started earlier, so it is only the controller that reads it.  (A batch's: whoever sets the flag
    // has given up, and so does every CTA that waits.)
    if (fits && *reinterpret_cast<volatile int*>(&top->abort) != 0) return;
    if constexpr (sizeof(T) == 8) {   // the exponentials' table, behind everything else
        smem_bytes -= kExpTab * sizeof(double);
        double* tab = reinterpret_cast<double*>(smem_order + smem_bytes);
        for (int j = threadIdx.x; j < kExpTab; j += NT) tab[j] = exp2(double(j) / kExpTab);
    }
    int d = 0, rank = blockIdx.x, size = gridDim.x;
    if (fits) {
        const int4 as = assign[blockIdx.x];
        d = as.x;
        rank = as.y;
        size = as.z;
    }
    for (;;) {
        if (d >= 0) {
            __syncthreads();
            if (threadIdx.x == 0) s_fit = fits ? fits[d] : one;
            __syncthreads();
            if (!run_problem<T, NT>(s_fit, top, rank, size, fits ? s_fit.p : iters, smem_bytes, sh)) return;
        }
        if (!fits) return;
        __syncthreads();
        if (threadIdx.x == 0) sh.qnext = int(atomicAdd(qhead, 1u));
        __syncthreads();
        const int q = sh.qnext;
        if (q >= nqueue) return;
        d = queue[q];
        rank = 0;
        size = 1;
    }
}

// ------------------------------------------------------------------ bounded-wait self-test
// which = 1: the controller's wait for arrivals of workers that are not there; 2: a worker's wait for a
// wave word that nothing publishes.
__device__ Ctl g_order_selftest_ctl;
__global__ void k_order_wait_selftest(int which) {
    __shared__ OrderShared sh;
    Ctl* ctl = &g_order_selftest_ctl;
    const unsigned long long tmo = *reinterpret_cast<volatile unsigned long long*>(&ctl->timeout_ns);
    OrderWave wv;
    if (which == 1) wait_arrivals(ctl, ctl, 1u, tmo, sh);
    else wait_order_wave(ctl, ctl, 1u, tmo, sh, wv);
}
cudaError_t run_order_wait_selftest(int which, unsigned long long timeout_ns, int* status, cudaStream_t st) {
    Ctl h = {};
    h.timeout_ns = timeout_ns;
    cudaError_t e = cudaMemcpyToSymbolAsync(g_order_selftest_ctl, &h, sizeof(h), 0, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return e;
    k_order_wait_selftest<<<1, 32, 0, st>>>(which);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    e = cudaMemcpyFromSymbolAsync(&h, g_order_selftest_ctl, sizeof(h), 0, cudaMemcpyDeviceToHost, st);
    if (e != cudaSuccess) return e;
    e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return e;
    *status = h.status;
    return cudaSuccess;
}

// ------------------------------------------------------------------ to the tile kernels
// One CTA per variable left in U (f.flags): its row into f.xt, its covariances with the later variables,
// normalised, into both triangles of f.sig and f.sigf, its statistics by its own mean, and its sort key.
// cur: the copies that hold the current rows, covariance and scales.  Runs once, about 0.1 ms at p = 1000.
constexpr int kHandThreads = 256;
__global__ void __launch_bounds__(kHandThreads) k_hand_over(Fit f, int cur) {
    const int p = f.p, ld = f.ld, v = blockIdx.x, tid = threadIdx.x;
    if (!(f.flags[v] & kAlive)) return;
    const double* S = cur ? f.sigalt : f.sig;   // (in place when it is f.sig: each element is read here alone)
    const double* D = f.dscale[cur];
    if (cur) {
        const float4* src = reinterpret_cast<const float4*>(static_cast<const float*>(f.xalt) + size_t(v) * ld);
        float4* dst = reinterpret_cast<float4*>(static_cast<float*>(f.xt) + size_t(v) * ld);
        for (int t = tid; t < ld / 4; t += kHandThreads) dst[t] = src[t];
    }
    const double dv = D[v];
    for (int j = v + tid; j < p; j += kHandThreads) {
        if (!(f.flags[j] & kAlive)) continue;
        const double c = j == v ? 1.0 : S[size_t(v) * p + j] * (dv * D[j]);
        const float2 cf = sig_pair_f(c);
        f.sig[size_t(v) * p + j] = c;
        f.sig[size_t(j) * p + v] = c;
        f.sigf[size_t(v) * p + j] = cf;
        f.sigf[size_t(j) * p + v] = cf;
    }
    if (tid == 0) {
        // the row's sum centred by the offset -32 (ln 2 + m0) over the padded row is -corr n
        const float4 s = f.vstat[v];
        const double m0 = -double(s.w) / kSub - kLn2, m = (double(ld) * m0 - double(s.x) * f.n) * f.inv_n;
        f.vstat[v] = var_stats_inv((m - kBeta) * f.n, double(s.z) * f.n, f.n, ld, f.inv_n);
        f.prev[v] = f.hx[v];
    }
}
cudaError_t launch_hand_over(const Fit& f, int it, cudaStream_t st) {
    k_hand_over<<<f.p, kHandThreads, 0, st>>>(f, it & 1);   // (a removal per iteration, each into the other copy)
    return cudaGetLastError();
}

// ------------------------------------------------------------------ host side
constexpr size_t kOrderSmem512 = 220 * 1024;
constexpr size_t kOrderSmem256 = 108 * 1024;

// Largest p whose controller state and I table (four columns) fit.
template <class T>
static bool order_fits_smem(long long p, size_t smem, bool dedicated) {
    const size_t state = order_state_bytes(int(p));
    if (state >= smem) return false;
    return order_max_cols<T>(unsigned(smem - (dedicated ? 0 : state)), int(p), unsigned(smem - state)) >= 4;
}

bool order_supported(const Fit& f, bool batch) {
    const bool f32 = f.precision == LINGAM_MIXED;
    if (f.p > 4096 || f.ld / 256 > 0xffff) return false;
    if (f.rec_bytes < 2 * size_t(f.p) * (4 * kMaxCols + 8) * 8) return false;   // one segment of a full wave
    const size_t smem = (batch ? kOrderSmem256 : kOrderSmem512) - (f32 ? 0 : kExpTab * sizeof(double));
    // (a single fit's group is below kDedicated CTAs only when p is small)
    return f32 ? order_fits_smem<float>(f.p, smem, !batch && f.p >= 64)
               : order_fits_smem<double>(f.p, smem, !batch && f.p >= 64);
}

template <class T, int NT>
static cudaError_t launch_order_t(const Fit& f, int iters, const Fit* fits, const int4* assign, const int* queue, int nqueue,
                                  unsigned* qhead, Ctl* top, int grid, cudaStream_t st) {
    const void* fn = reinterpret_cast<const void*>(k_order<T, NT>);
    unsigned smem = unsigned(NT == 512 ? kOrderSmem512 : kOrderSmem256);
    cudaError_t e = ensure_smem_attr(fn, smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;   // all CTAs co-resident: they wait for each other
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_order<T, NT>, f, iters, fits, assign, queue, nqueue, qhead, top, smem);
}

// CTAs of a single fit: enough for four warps' units each in the first removal's wave (a row against
// four columns, and the row's own), the whole GPU at most.
int order_grid(const Fit& f, int nsm) {
    const bool f32 = f.precision == LINGAM_MIXED;
    const long long units = (long long)f.p * ((f.ld + f.unit - 1) / f.unit) * (f32 ? 2 : 5);
    return int(std::max(1ll, std::min((long long)nsm, 1 + (units + 3) / 4)));
}

cudaError_t launch_order(const Fit& f, int iters, int nsm, cudaStream_t st) {
    const int grid = order_grid(f, nsm);
    return f.precision == LINGAM_MIXED ? launch_order_t<float, 512>(f, iters, nullptr, nullptr, nullptr, 0, nullptr, f.ctl, grid, st)
                                       : launch_order_t<double, 512>(f, iters, nullptr, nullptr, nullptr, 0, nullptr, f.ctl, grid, st);
}

// Clocks (estimate) of a problem on g CTAs of 256 threads: 3 pair-samples a clock and CTA (FP64:
// 1/40 of that), about 7 pairs per row and iteration (unpruned: all), and the hand-over of a wave.
static double batch_clocks(const Fit& f, int g) {
    const double p = f.p, rate = f.precision == LINGAM_MIXED ? 3.0 : 0.075;
    const double work = (f.prune ? 3.5 * p * p : p * p * p / 6.0) * f.ld / rate;
    const int W = g >= kDedicated ? g - 1 : g;
    return work / W + p * (g > 1 ? 16000.0 : 8000.0);
}

// Groups of a batch: with fewer problems than CTA slots every problem has a group, and the slots
// left go one by one to the problem that would take longest; with more, problems of more than
// twice a slot's share of the work get groups of their own, and the others queue, longest first,
// for single CTAs.
void order_batch_plan(const Fit* fits, int count, int nsm, std::vector<int4>& assign, std::vector<int>& queue) {
    const int slots = std::min(2 * nsm, kOrderSlots);
    std::vector<int> g(static_cast<size_t>(count), 1), big;
    queue.clear();
    if (count <= slots) {
        std::priority_queue<std::pair<double, int>> longest;
        for (int d = 0; d < count; ++d) longest.push({batch_clocks(fits[d], 1), d});
        for (int left = slots - count; left > 0 && !longest.empty(); --left) {
            const int d = longest.top().second;
            longest.pop();
            ++g[size_t(d)];
            const long long most = (long long)fits[d].p * ((fits[d].ld + 1023) / 1024);   // rows x blocks
            if (g[size_t(d)] < most) longest.push({batch_clocks(fits[d], g[size_t(d)]), d});
        }
        for (int d = 0; d < count; ++d) big.push_back(d);
    } else {
        double total = 0.0;
        std::vector<std::pair<double, int>> by;
        for (int d = 0; d < count; ++d) {
            by.push_back({batch_clocks(fits[d], 1), d});
            total += by.back().first;
        }
        std::sort(by.begin(), by.end(), [](const auto& a, const auto& b) { return a.first > b.first || (a.first == b.first && a.second < b.second); });
        int left = slots - 1;   // one slot at least for the queue
        for (const auto& b : by) {
            const int want = int(std::min(double(slots), b.first / (total / slots)));
            if (want >= 2 && want <= left) {
                g[size_t(b.second)] = want;
                left -= want;
                big.push_back(b.second);
            } else {
                queue.push_back(b.second);
            }
        }
    }
    assign.clear();
    for (int d : big)
        for (int k = 0; k < g[size_t(d)]; ++k) assign.push_back(make_int4(d, k, g[size_t(d)], 0));
    while (int(assign.size()) < slots && !queue.empty()) assign.push_back(make_int4(-1, 0, 0, 0));
}

cudaError_t launch_order_batch(const Fit* fits_dev, int precision, const int4* assign, int grid, const int* queue, int nqueue,
                               unsigned* qhead, Ctl* bctl, cudaStream_t st) {
    const Fit none = {};
    return precision == LINGAM_MIXED
               ? launch_order_t<float, 256>(none, 0, fits_dev, assign, queue, nqueue, qhead, bctl, grid, st)
               : launch_order_t<double, 256>(none, 0, fits_dev, assign, queue, nqueue, qhead, bctl, grid, st);
}

}  // namespace lingam
