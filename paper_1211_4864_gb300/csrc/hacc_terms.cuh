// One-sided pair terms of the gather kernels (force, potential, adjoint): what
// a pair (i, j) adds to particle i's sums, and those sums in registers.
#pragma once

#include "hacc_pairs.cuh"

namespace hacc {
namespace {

// Sums of IPL i particles in registers: float32 partial sums, folded into
// compensated (hi, lo) pairs.
template <int IPL, int NC>
struct AccN {
    float a[IPL][NC], h[IPL][NC], l[IPL][NC];
    __device__ __forceinline__ AccN()
    {
#pragma unroll
        for (int u = 0; u < IPL; ++u)
#pragma unroll
            for (int k = 0; k < NC; ++k) a[u][k] = h[u][k] = l[u][k] = 0.f;
    }
    __device__ __forceinline__ void fold()
    {
#pragma unroll
        for (int u = 0; u < IPL; ++u)
#pragma unroll
            for (int k = 0; k < NC; ++k) {
                two_sum_acc(h[u][k], l[u][k], a[u][k]);
                a[u][k] = 0.f;
            }
    }
};

// One pair of the forward law, accumulated into acc[3] (EQ, equal masses:
// f d, the mass applied to the total).  The cutoff test is a compare whose
// predicate guards the three accumulating fma (no branch, no select): the
// paper folds the same test into the loop with fsel (Sec. III).
template <bool EQ>
__device__ __forceinline__ void pair_force(const float4 p, float oxp, float oyp, float ozp, const PairConsts &K,
                                           float *acc)
{
    float dx = p.x - oxp, dy = p.y - oyp, dz = p.z - ozp;
    float se = fmaf(dz, dz, fmaf(dy, dy, fmaf(dx, dx, K.eps)));
    float t = rsqrt_hw(se);
    float t2 = t * t;
    float q = fmaf(fmaf(fmaf(fmaf(fmaf(K.nc[5], se, K.nc[4]), se, K.nc[3]), se, K.nc[2]), se, K.nc[1]), se,
                   K.nc[0]);
    float g = EQ ? fmaf(t2, t, q) : fmaf(t2, t, q) * p.w;
    asm("{\n\t.reg .pred p;\n\tsetp.lt.f32 p, %3, %4;\n\t"
        "@p fma.rn.f32 %0, %5, %6, %0;\n\t@p fma.rn.f32 %1, %5, %7, %1;\n\t@p fma.rn.f32 %2, %5, %8, %2;\n\t}"
        : "+f"(acc[0]), "+f"(acc[1]), "+f"(acc[2])
        : "f"(se), "f"(K.rc2e), "f"(g), "f"(dx), "f"(dy), "f"(dz));
}

// The short-range pair potential V(s) = pv(se) - (s + eps)^-1/2 (se = s + eps):
// the integral of the force law, zero at the cutoff (F = -grad V).
__device__ __forceinline__ float pair_potential_of(float se, const PairConsts &K)
{
    const float h = fmaf(fmaf(fmaf(fmaf(fmaf(fmaf(K.pv[6], se, K.pv[5]), se, K.pv[4]), se, K.pv[3]), se, K.pv[2]),
                              se, K.pv[1]),
                         se, K.pv[0]);
    return h - rsqrt_hw(se);
}

__device__ __forceinline__ void pair_potential(const float4 p, float oxp, float oyp, float ozp, const PairConsts &K,
                                               float *acc)
{
    float dx = p.x - oxp, dy = p.y - oyp, dz = p.z - ozp;
    float se = fmaf(dz, dz, fmaf(dy, dy, fmaf(dx, dx, K.eps)));
    float v = pair_potential_of(se, K);
    asm("{\n\t.reg .pred p;\n\tsetp.lt.f32 p, %1, %2;\n\t@p fma.rn.f32 %0, %3, %4, %0;\n\t}"
        : "+f"(acc[0])
        : "f"(se), "f"(K.rc2e), "f"(p.w), "f"(v));
}

// One pair of the adjoint, accumulated into acc = (W, G) of one i: with f =
// f_SR(s), fp2 = 2 f_SR'(s) and mu = m_i lam_j - m_j lam_i (equal masses, EQ:
// mu / m = lam_j - lam_i),
//   W += f mu + fp2 (d.mu) d      dL/dx_i = W (equal masses: m W)
//   G += f (d.lam_j)              dL/dm_i = -G (GM only)
// Summing the antisymmetric pair term takes the cancellation between the lam_j
// and lam_i parts of a close pair out of the totals.
template <bool GM, bool EQ>
__device__ __forceinline__ void pair_adjoint(const float4 p, const float4 l, float oxp, float oyp, float ozp,
                                             float mi, float lix, float liy, float liz, const PairConsts &K,
                                             float (&acc)[ADJ_NACC])
{
    float dx = p.x - oxp, dy = p.y - oyp, dz = p.z - ozp;
    float se = fmaf(dz, dz, fmaf(dy, dy, fmaf(dx, dx, K.eps)));
    float t = rsqrt_hw(se);
    float t2 = t * t;
    float t3 = t2 * t;
    float q = fmaf(fmaf(fmaf(fmaf(fmaf(K.nc[5], se, K.nc[4]), se, K.nc[3]), se, K.nc[2]), se, K.nc[1]), se,
                   K.nc[0]);
    float f = t3 + q;
    float qp = fmaf(fmaf(fmaf(fmaf(K.kp[4], se, K.kp[3]), se, K.kp[2]), se, K.kp[1]), se, K.kp[0]);
    float fp2 = fmaf(-3.0f, t3 * t2, qp);
    float ex, ey, ez;  // mu (equal masses: mu / m)
    if constexpr (EQ) {
        ex = l.x - lix;
        ey = l.y - liy;
        ez = l.z - liz;
    } else {
        ex = fmaf(mi, l.x, -(p.w * lix));
        ey = fmaf(mi, l.y, -(p.w * liy));
        ez = fmaf(mi, l.z, -(p.w * liz));
    }
    const float r = fp2 * fmaf(dz, ez, fmaf(dy, ey, dx * ex));
    // the accumulations of this pair happen only inside the cutoff
    if constexpr (GM) {
        const float dlj = fmaf(dz, l.z, fmaf(dy, l.y, dx * l.x));
        asm("{\n\t.reg .pred p;\n\tsetp.lt.f32 p, %4, %5;\n\t"
            "@p fma.rn.f32 %0, %6, %7, %0;\n\t@p fma.rn.f32 %1, %6, %8, %1;\n\t@p fma.rn.f32 %2, %6, %9, %2;\n\t"
            "@p fma.rn.f32 %0, %10, %11, %0;\n\t@p fma.rn.f32 %1, %10, %12, %1;\n\t"
            "@p fma.rn.f32 %2, %10, %13, %2;\n\t@p fma.rn.f32 %3, %6, %14, %3;\n\t}"
            : "+f"(acc[0]), "+f"(acc[1]), "+f"(acc[2]), "+f"(acc[3])
            : "f"(se), "f"(K.rc2e), "f"(f), "f"(ex), "f"(ey), "f"(ez), "f"(r), "f"(dx), "f"(dy), "f"(dz), "f"(dlj));
    } else {
        asm("{\n\t.reg .pred p;\n\tsetp.lt.f32 p, %3, %4;\n\t"
            "@p fma.rn.f32 %0, %5, %6, %0;\n\t@p fma.rn.f32 %1, %5, %7, %1;\n\t@p fma.rn.f32 %2, %5, %8, %2;\n\t"
            "@p fma.rn.f32 %0, %9, %10, %0;\n\t@p fma.rn.f32 %1, %9, %11, %1;\n\t@p fma.rn.f32 %2, %9, %12, %2;\n\t}"
            : "+f"(acc[0]), "+f"(acc[1]), "+f"(acc[2])
            : "f"(se), "f"(K.rc2e), "f"(f), "f"(ex), "f"(ey), "f"(ez), "f"(r), "f"(dx), "f"(dy), "f"(dz));
    }
}

// What a dense gather adjoint's sum W holds of the pair of i with itself (d = 0)
// when the masses differ: f(0) times the rounding of m_i lam_i - m_i lam_i,
// some 1e-4 for the default softening, taken out of the total again.
__device__ __forceinline__ float self_term(const PairConsts &K, float m, float l)
{
    const float t = rsqrt_hw(K.eps);
    const float q = fmaf(fmaf(fmaf(fmaf(fmaf(K.nc[5], K.eps, K.nc[4]), K.eps, K.nc[3]), K.eps, K.nc[2]), K.eps, K.nc[1]),
                         K.eps, K.nc[0]);
    return (t * t * t + q) * fmaf(m, l, -(m * l));
}

// The outputs of one i from its totals, total(k), at input index o.
template <int MODE, class Total>
__device__ __forceinline__ void store_out(const KArgs &a, int o, const float4 &oi, bool eq, const Total &total)
{
    if constexpr (MODE == POTENTIAL) {
        a.out_x[o] = total(0);
    } else {
        // equal masses: the sums times m
        const float sc = eq ? oi.w : 1.0f;
        a.out_x[o] = sc * total(0);
        a.out_y[o] = sc * total(1);
        a.out_z[o] = sc * total(2);
        if constexpr (MODE == ADJOINT_GM) a.out_m[o] = -total(3);
    }
}

}  // namespace
}  // namespace hacc
