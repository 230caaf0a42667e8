// pair.cuh -- the arithmetic of physics.cuh on two cells at once, with the packed FP32 instructions
// of sm_100 and later (fma.rn.f32x2 and its kin): every operation is the scalar one in both halves,
// rounded the same way, so a cell's trajectory is bitwise that of the scalar engines.
//
// Why: the rod kernels are bound by the instruction issue of the four schedulers and by the FMA pipes
// behind them.  A packed multiply-add occupies the pipes as long as two scalar ones (measured 2.0
// scheduler cycles a warp against 1.0) but issues once: one Heun step's fields and torques take 40
// issue slots per warp and cell instead of 81, and 84 cycles instead of 93 when nothing else runs.
// Negations are written on the unpacked halves: with an exclusive-or on the packed word the same measured
// 87 cycles.
#pragma once

#include "physics.cuh"

namespace llg {

using pair_t = unsigned long long;  // two floats, cell a in the low half and cell b in the high half

__device__ __forceinline__ pair_t pack2(float a, float b)
{
    pair_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float lo2(pair_t v)
{
    float a;
    asm("{\n\t.reg .f32 t;\n\tmov.b64 {%0, t}, %1;\n\t}" : "=f"(a) : "l"(v));
    return a;
}
__device__ __forceinline__ float hi2(pair_t v)
{
    float b;
    asm("{\n\t.reg .f32 t;\n\tmov.b64 {t, %0}, %1;\n\t}" : "=f"(b) : "l"(v));
    return b;
}
__device__ __forceinline__ pair_t both(float a) { return pack2(a, a); }
__device__ __forceinline__ pair_t neg2(pair_t v) { return pack2(-lo2(v), -hi2(v)); }
__device__ __forceinline__ pair_t fma2(pair_t a, pair_t b, pair_t c)
{
    pair_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ pair_t add2(pair_t a, pair_t b)
{
    pair_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ pair_t mul2(pair_t a, pair_t b)
{
    pair_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// A vector of two cells.
struct Pair3 {
    pair_t x, y, z;
};

__device__ __forceinline__ Pair3 zero_p3() { return Pair3{0ull, 0ull, 0ull}; }
__device__ __forceinline__ Pair3 pair3(float3 a, float3 b)
{
    return Pair3{pack2(a.x, b.x), pack2(a.y, b.y), pack2(a.z, b.z)};
}
__device__ __forceinline__ float3 lo3(Pair3 v) { return make_float3(lo2(v.x), lo2(v.y), lo2(v.z)); }
__device__ __forceinline__ float3 hi3(Pair3 v) { return make_float3(hi2(v.x), hi2(v.y), hi2(v.z)); }
__device__ __forceinline__ Pair3 add_p3(Pair3 a, Pair3 b)
{
    return Pair3{add2(a.x, b.x), add2(a.y, b.y), add2(a.z, b.z)};
}
__device__ __forceinline__ Pair3 axpy_p3(pair_t a, Pair3 x, Pair3 y)
{
    return Pair3{fma2(a, x.x, y.x), fma2(a, x.y, y.y), fma2(a, x.z, y.z)};
}

// The coefficients in both halves.
struct PairCoeffs {
    pair_t c_ex, c_an, alpha, neg_dt_g1, neg_hdt_g1;
};
__device__ __forceinline__ PairCoeffs pair_coeffs(const KParams &p)
{
    return PairCoeffs{both(p.c_ex), both(p.c_an), both(p.alpha), both(p.neg_dt_g1), both(p.neg_hdt_g1)};
}

// box_muller3 for the Philox words of two cells.
__device__ __forceinline__ Pair3 box_muller_p3(uint4 a, uint4 b, float sigma_bm)
{
    const pair_t k24 = both(0x1p-24f), k25 = both(0x1p-25f), sg = both(sigma_bm);
    const pair_t u0 = fma2(pack2(bits24(a.x), bits24(b.x)), k24, k25);
    const pair_t u2 = fma2(pack2(bits24(a.z), bits24(b.z)), k24, k25);
    const pair_t r0 = mul2(sg, pack2(sqrt_fast(fabsf(log2_fast(lo2(u0)))), sqrt_fast(fabsf(log2_fast(hi2(u0))))));
    const pair_t r2 = mul2(sg, pack2(sqrt_fast(fabsf(log2_fast(lo2(u2)))), sqrt_fast(fabsf(log2_fast(hi2(u2))))));
    const pair_t step = both(kAngleStep), first = both(kAngleFirst);
    const pair_t a1 = fma2(pack2(bits24(a.y), bits24(b.y)), step, first);
    const pair_t a3 = fma2(pack2(bits24(a.w), bits24(b.w)), step, first);
    // z as a multiply-add with zero: with a plain product, to which the Zeeman field is added next, one kernel's
    // states differed from the scalar engines' in the last bit (a bitwise test found it), with this none do
    return Pair3{mul2(r0, pack2(cos_fast(lo2(a1)), cos_fast(hi2(a1)))), mul2(r0, pack2(sin_fast(lo2(a1)), sin_fast(hi2(a1)))),
                 fma2(r2, pack2(cos_fast(lo2(a3)), cos_fast(hi2(a3))), 0ull)};
}

// Thermal field of a cell (of product cell_m0 = kPhiloxM0 * cell) and the next one of the same rod.
__device__ __forceinline__ Pair3 thermal_field_p3(const PhiloxKeys &K, const PhiloxStep &S, unsigned long long cell_m0,
                                                  float sigma_bm)
{
    return box_muller_p3(philox4x32_10(K, S, cell_m0), philox4x32_10(K, S, cell_m0 + kPhiloxM0), sigma_bm);
}

// effective_field (AX = false; u unused) and effective_field_axis (AX).
template <bool AX>
__device__ __forceinline__ Pair3 effective_field_p3(Pair3 nb, Pair3 m, Pair3 h, const PairCoeffs &c, pair_t Hz, Pair3 u)
{
    if constexpr (AX) {
        const pair_t a = mul2(c.c_an, fma2(m.x, u.x, fma2(m.y, u.y, mul2(m.z, u.z))));
        return Pair3{fma2(c.c_ex, nb.x, fma2(a, u.x, h.x)), fma2(c.c_ex, nb.y, fma2(a, u.y, h.y)),
                     fma2(c.c_ex, nb.z, fma2(a, u.z, add2(h.z, Hz)))};
    } else {
        return Pair3{fma2(c.c_ex, nb.x, h.x), fma2(c.c_ex, nb.y, h.y),
                     fma2(c.c_ex, nb.z, fma2(c.c_an, m.z, add2(h.z, Hz)))};
    }
}

__device__ __forceinline__ Pair3 torque_arm_p3(Pair3 m, Pair3 H, pair_t alpha)
{
    const pair_t ax = fma2(m.y, H.z, mul2(neg2(m.z), H.y));
    const pair_t ay = fma2(m.z, H.x, mul2(neg2(m.x), H.z));
    const pair_t az = fma2(m.x, H.y, mul2(neg2(m.y), H.x));
    return Pair3{fma2(alpha, ax, H.x), fma2(alpha, ay, H.y), fma2(alpha, az, H.z)};
}

__device__ __forceinline__ Pair3 llg_torque_p3(Pair3 m, Pair3 H, pair_t alpha)
{
    const Pair3 B = torque_arm_p3(m, H, alpha);
    return Pair3{fma2(m.y, B.z, mul2(neg2(m.z), B.y)), fma2(m.z, B.x, mul2(neg2(m.x), B.z)),
                 fma2(m.x, B.y, mul2(neg2(m.y), B.x))};
}

__device__ __forceinline__ Pair3 llg_torque_add_p3(Pair3 s0, Pair3 m, Pair3 H, pair_t alpha)
{
    const Pair3 B = torque_arm_p3(m, H, alpha);
    return Pair3{fma2(m.y, B.z, fma2(neg2(m.z), B.y, s0.x)), fma2(m.z, B.x, fma2(neg2(m.x), B.z, s0.y)),
                 fma2(m.x, B.y, fma2(neg2(m.y), B.x, s0.z))};
}

__device__ __forceinline__ Pair3 normalised_p3(Pair3 v)
{
    const pair_t n = fma2(v.x, v.x, fma2(v.y, v.y, mul2(v.z, v.z)));
    const pair_t r = pack2(rsqrt_fast(lo2(n)), rsqrt_fast(hi2(n)));
    return Pair3{mul2(v.x, r), mul2(v.y, r), mul2(v.z, r)};
}

}  // namespace llg
