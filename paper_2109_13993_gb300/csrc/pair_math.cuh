// pair_math.cuh -- the FP32 per-sample arithmetic of the pair comparison (Eqs. Itest, HApp and
// var_update), float-float sums, and the release / acquire operations of the hand-overs between
// CTAs, shared by the tile kernels (k_iter.cu) and the ordering kernel (k_order.cu).
#pragma once

#include "common.cuh"

namespace lingam {

// FP32 residuals carry the scale kScale: with u' = kScale*u,
//   e^{-u^2/2} = 2^{-u'^2},   e^{-2|u|} = 2^{kC3 |u'|}.
constexpr float kScale = 0.84932180028801904272f;     // sqrt(log2(e)/2)
constexpr float kInvScale = 1.17741002251547469101f;  // 1/kScale
constexpr float kC3 = -3.39728720115207617088f;       // -2 log2(e) / kScale

// Sum of squares in float-float arithmetic: the exact square (TwoProduct) added
// with TwoSum into a (hi, lo) pair, about 48 bits of precision on the FP32 pipe.
struct FF {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add_sq(float m) {
        const float pr = m * m, pe = fmaf(m, m, -pr);
        const float s = hi + pr, bb = s - hi;
        const float err = (hi - (s - bb)) + (pr - bb);
        hi = s;
        lo += err + pe;
    }
    __device__ __forceinline__ double value() const { return double(hi) + double(lo); }
};

// gpu-scope release and acquire operations for the barrier and publication protocols: a
// CTA barrier orders every thread's writes before thread 0's release, and thread 0's
// acquire before every thread's later reads.
__device__ __forceinline__ unsigned atom_add_release(unsigned* p, unsigned v) {
    unsigned old;
    asm volatile("atom.release.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}
__device__ __forceinline__ int atom_add_acq_rel(int* p, int v) {
    int old;
    asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}
__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long ld_acquire64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release64(unsigned long long* p, unsigned long long v) {
    asm volatile("st.release.gpu.global.u64 [%0], %1;" : : "l"(p), "l"(v) : "memory");
}

// ------------------------------------------------------------------ per-sample math (FP32)
// Two consecutive samples of one residual u' (scaled by kScale).
struct Acc2 {
    float2 A, P, G;   // sum of |kC3 u'|, product of (1 + e^{-2|u|}), sum of u' e^{-u^2/2}; per half
};
__device__ __forceinline__ void acc2_add(Acc2& s, float2 u) {
    const float2 q = __fmul2_rn(u, u);
    float2 g;
    g.x = ex2_approx(-q.x);
    g.y = ex2_approx(-q.y);
    s.G = __ffma2_rn(u, g, s.G);
    // y = kC3 u' (kC3 < 0): e^{-2|u|} = 2^{-|y|}, the sign and the absolute value being
    // operand modifiers of the exponential
    const float2 y = __fmul2_rn(u, make_float2(kC3, kC3));
    float2 e;
    e.x = ex2_approx(-fabsf(y.x));
    e.y = ex2_approx(-fabsf(y.y));
    s.P = __ffma2_rn(s.P, e, s.P);
    s.A = __fadd2_rn(s.A, make_float2(fabsf(y.x), fabsf(y.y)));
}

// I(x_i, x_j, r_i^(j), r_j^(i)) of Eq. Itest on the FP32 path, from a pair's merged sums
// over the padded row: Ta, Tb the residuals' log-cosh sums centred by their variables'
// group offsets (var_stats .w), Ga, Gb their sums of u' exp(-u^2/2) (u' = kScale u), and
// the two variables' statistics si, sj.  Written as the difference of each residual's
// entropy (Eq. HApp) from its own variable's,
//   I = [H(r_i^(j)) - H(x_i)] - [H(r_j^(i)) - H(x_j)],
// each bracket -k1 d (2 (m - beta) + d) - k2 (g_r - g)(g_r + g) with d = T / n + corr the
// residual's mean log cosh minus its variable's, so that no FP32 term is larger than the
// difference it contributes to.
__device__ __forceinline__ float pair_measure_f(float Ta, float Ga, float Tb, float Gb, float4 si, float4 sj,
                                                float inv_n) {
    const float cg = kInvScale * inv_n;
    const float da = fmaf(Ta, inv_n, si.x), db = fmaf(Tb, inv_n, sj.x);
    const float ga = Ga * cg, gb = Gb * cg;
    const float Da = -float(kK1) * da * (si.y + da) - float(kK2) * (ga - si.z) * (ga + si.z);
    const float Db = -float(kK1) * db * (sj.y + db) - float(kK2) * (gb - sj.z) * (gb + sj.z);
    return Da - Db;
}

__device__ __forceinline__ void acc_pair4(Acc2& aa, Acc2& ab, float4 a4, float4 b4, float2 s2, float2 sr2) {
    const float2 vi2[2] = {make_float2(a4.x, a4.y), make_float2(a4.z, a4.w)};
    const float2 vj2[2] = {make_float2(b4.x, b4.y), make_float2(b4.z, b4.w)};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        acc2_add(aa, __ffma2_rn(s2, vi2[h], __fmul2_rn(sr2, vj2[h])));
        acc2_add(ab, __ffma2_rn(s2, vj2[h], __fmul2_rn(sr2, vi2[h])));
    }
}
__device__ __forceinline__ void acc_init(Acc2& a) {
    a.A = make_float2(0.f, 0.f);
    a.P = make_float2(1.f, 1.f);
    a.G = make_float2(0.f, 0.f);
}

}  // namespace lingam
