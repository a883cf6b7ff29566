// lb_packed.cuh — the per-site physics of lb_device.cuh for two sites at a
// time (adjacent columns x, x + 1 of one row) in packed FP32 pairs: sm_103a
// issues an add, multiply or multiply-add of two FP32 values as one
// instruction, each half rounded like the scalar operation. The step kernels
// are bound by instruction issue once their memory traffic is out of the way,
// so a pair of sites shares the instructions. Every operation below is the one
// the scalar functions compile to, in their order (products that the scalar
// code contracts into a multiply-add are written as one), so the results are
// bit-identical to theirs.
#pragma once

#include "lb_device.cuh"

namespace lbsc {
namespace dev {

__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return fma2(b, dup2(-1.f), a); }

// The arguments of a step the packed functions use, each in both halves.
struct PackedArgs {
    float2 K1, K2, K4x2, K5, K8x2;             // couplings (K4 and K8 doubled, exactly)
    float2 w0, w1, w2;
    float2 rho_ref, psi_ref, omega, omc, inv_omega;
};
template <typename T>
__host__ __device__ inline PackedArgs packed_args(const StepArgs<T>& a)
{
    auto d = [](float v) { return make_float2(v, v); };
    return PackedArgs{d(a.K1), d(a.K2), d(2.f * a.K4), d(a.K5), d(2.f * a.K8),
                      d(a.w0), d(a.w1), d(a.w2),
                      d(a.rho_ref), d(a.psi_ref), d(a.omega), d(a.omc), d(a.inv_omega)};
}

// The twelve pair differences of the force stencil for the columns x, x + 1. A[k],
// B[k], C[k] are the field's columns (x-2, x-1), (x, x+1), (x+2, x+3) in row y + k - 2: the
// stencil offsets -2, 0 and +2 are whole pairs; the differences that pair an odd offset
// are formed one half at a time from the pairs' halves.
struct Diffs2 {
    float2 d10, d01, d20, d02;   // (c) - (-c) for c = (1,0), (0,1), (2,0), (0,2)
    float2 sum1, dif1;           // (1,1) and (1,-1): sum and difference
    float2 mx, my;               // |c|^2 = 5: the x and y combinations
    float2 sum8, dif8;           // (2,2) and (2,-2)
};
__device__ __forceinline__ Diffs2 diffs2(const float2 A[5], const float2 B[5], const float2 C[5])
{
    Diffs2 r;
    r.d10 = make_float2(B[2].y - A[2].y, C[2].x - B[2].x);
    r.d01 = sub2(B[3], B[1]);
    const float2 d11 = make_float2(B[3].y - A[1].y, C[3].x - B[1].x);
    const float2 d1m = make_float2(B[1].y - A[3].y, C[1].x - B[3].x);
    r.d20 = sub2(C[2], A[2]);
    r.d02 = sub2(B[4], B[0]);
    const float2 da = sub2(C[3], A[1]);
    const float2 db = make_float2(B[4].y - A[0].y, C[4].x - B[0].x);
    const float2 dc = make_float2(A[4].y - B[0].y, B[4].x - C[0].x);
    const float2 dd = sub2(A[3], C[1]);
    const float2 e1 = sub2(C[4], A[0]);
    const float2 e2 = sub2(C[0], A[4]);
    const float2 two = dup2(2.f);
    r.sum1 = add2(d11, d1m);
    r.dif1 = sub2(d11, d1m);
    r.mx = fma2(two, sub2(da, dd), sub2(db, dc));
    r.my = fma2(two, add2(db, dc), add2(da, dd));
    r.sum8 = add2(e1, e2);
    r.dif8 = sub2(e1, e2);
    return r;
}
// The x and y force sums of force_sums / force_energy<false> from the differences
__device__ __forceinline__ float2 sum_x2(const Diffs2& r, const PackedArgs& k)
{
    const float2 s = fma2(k.K4x2, r.d20, fma2(k.K1, r.d10, mul2(k.K2, r.sum1)));
    return fma2(k.K8x2, r.sum8, fma2(k.K5, r.mx, s));
}
__device__ __forceinline__ float2 sum_y2(const Diffs2& r, const PackedArgs& k)
{
    const float2 s = fma2(k.K4x2, r.d02, fma2(k.K1, r.d01, mul2(k.K2, r.dif1)));
    return fma2(k.K8x2, r.dif8, fma2(k.K5, r.my, s));
}
__device__ __forceinline__ void force_sums2(const float2 A[5], const float2 B[5], const float2 C[5],
                                            const PackedArgs& k, float2& Sx, float2& Sy)
{
    const Diffs2 r = diffs2(A, B, C);
    Sx = sum_x2(r, k);
    Sy = sum_y2(r, k);
}

// -1/x of both halves, 1/x rounded to nearest as __frcp_rn gives it: one Newton
// step from the hardware approximation with the residual of a fused multiply-add
// (Markstein, "Computation of elementary functions on the IBM RISC System/6000
// processor", 1990). Equal to __frcp_rn for every FP32 value of magnitude 2^-125 to
// 2^125 (tests/c/rcp_check.cu compares all of them: the approximation's error decides that, not
// the theorem alone); outside (a density that has blown up) __frcp_rn itself.
__device__ __forceinline__ float2 neg_rcp2(float2 x)
{
    const float lo = fminf(fabsf(x.x), fabsf(x.y)), hi = fmaxf(fabsf(x.x), fabsf(x.y));
    if (!(lo > 0x1p-125f && hi < 0x1p125f)) return make_float2(-__frcp_rn(x.x), -__frcp_rn(x.y));
    float2 y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y.x) : "f"(-x.x));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y.y) : "f"(-x.y));
    return fma2(y, fma2(x, y, dup2(1.f)), y);
}

// The moments of two sites: d = rho - rho_ref, and the momentum negated.
struct Moments2 {
    float2 d, jx, jy;
};
__device__ __forceinline__ Moments2 moments2(const float2 f[9])
{
    Moments2 m;
    m.d = add2(add2(add2(add2(f[0], f[1]), add2(f[2], f[3])),
                    add2(add2(f[4], f[5]), add2(f[6], f[7]))),
               f[8]);
    m.jx = add2(add2(sub2(f[3], f[1]), sub2(f[6], f[5])), sub2(f[7], f[8]));
    m.jy = sub2(add2(f[7], f[8]), add2(sub2(f[2], f[4]), add2(f[5], f[6])));
    return m;
}

// collide() for two sites from their moments and minus the force (P = psi S). The
// momentum and the reciprocal are formed negated, which costs nothing and leaves
// u's bits as they are. f is read only without OM1.
template <bool OM1>
__device__ __forceinline__ void collide2(const Moments2& m, const float2 f[9], float2 Px, float2 Py,
                                         const PackedArgs& k, float2 gs[9])
{
    const float2 d = m.d, jx = m.jx, jy = m.jy;
    const float2 rho = add2(k.rho_ref, d);
    const float2 inv = neg_rcp2(rho);
    const float2 io = k.inv_omega;
    const float2 ux = mul2(OM1 ? add2(Px, jx) : fma2(Px, io, jx), inv);
    const float2 uy = mul2(OM1 ? add2(Py, jy) : fma2(Py, io, jy), inv);
    const float2 nsq = mul2(dup2(-1.5f), fma2(ux, ux, mul2(uy, uy)));   // -3/2 u^2
    const float2 orho = OM1 ? rho : mul2(k.omega, rho);
    const float2 od = OM1 ? d : mul2(k.omega, d);
    const float2 A0 = mul2(orho, k.w0), A1 = mul2(orho, k.w1), A2 = mul2(orho, k.w2);
    const float2 D0 = mul2(od, k.w0), D1 = mul2(od, k.w1), D2 = mul2(od, k.w2);
    const float2 c45 = dup2(4.5f);
    gs[0] = fma2(A0, nsq, D0);
    auto dir = [&](float2 c, float2 A, float2 D, float2& plus, float2& minus) {
        const float2 s = fma2(mul2(c45, c), c, nsq);
        plus = fma2(A, fma2(dup2(3.f), c, s), D);
        minus = fma2(A, fma2(dup2(-3.f), c, s), D);
    };
    dir(ux, A1, D1, gs[1], gs[3]);
    dir(uy, A1, D1, gs[2], gs[4]);
    dir(add2(ux, uy), A2, D2, gs[5], gs[7]);
    dir(sub2(uy, ux), A2, D2, gs[6], gs[8]);
    if (!OM1) {
#pragma unroll
        for (int i = 0; i < 9; ++i) gs[i] = fma2(k.omc, f[i], gs[i]);
    }
}

}  // namespace dev
}  // namespace lbsc
