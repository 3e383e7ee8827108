// lbm_pair.cuh -- the fused update for two nodes per thread with packed FP32x2
// arithmetic (sm_100+ FFMA2 / FADD2 / FMUL2).
//
// A thread takes nodes (x, y) and (x, y + 1): their loads and stores stay
// per node (coalesced along x, no shuffles), while every arithmetic operation
// of the collision works on both nodes at once.  The value type F2 carries the
// two nodes; a product is kept unevaluated (P2) so that a * b + c becomes one
// packed FMA, as the compiler would contract it for scalars.
#pragma once

#include <cuda_runtime.h>

#include "lbm_device.cuh"

namespace lbm {

struct F2 {
    float2 v;
    F2() = default;
    LBM_HD F2(float2 x) : v(x) {}
    LBM_HD F2(float s) : v(make_float2(s, s)) {}
    LBM_HD F2(double s) : F2(float(s)) {}
    LBM_HD F2(int s) : F2(float(s)) {}
};

__device__ __forceinline__ float2 neg2(float2 x) { return __fmul2_rn(x, make_float2(-1.f, -1.f)); }

struct P2 {  // the product a * b, not yet rounded
    float2 a, b;
    __device__ __forceinline__ operator F2() const { return F2(__fmul2_rn(a, b)); }
};

__device__ __forceinline__ P2 operator*(F2 x, F2 y) { return {x.v, y.v}; }
__device__ __forceinline__ P2 operator*(P2 p, F2 y) { return {F2(p).v, y.v}; }
__device__ __forceinline__ P2 operator*(F2 x, P2 p) { return {x.v, F2(p).v}; }
__device__ __forceinline__ P2 operator*(P2 p, P2 q) { return {F2(p).v, F2(q).v}; }

__device__ __forceinline__ F2 operator+(F2 x, F2 y) { return __fadd2_rn(x.v, y.v); }
__device__ __forceinline__ F2 operator+(P2 p, F2 y) { return __ffma2_rn(p.a, p.b, y.v); }
__device__ __forceinline__ F2 operator+(F2 y, P2 p) { return __ffma2_rn(p.a, p.b, y.v); }
__device__ __forceinline__ F2 operator+(P2 p, P2 q) { return __ffma2_rn(p.a, p.b, F2(q).v); }

// x - y = fma(y, -1, x) is exact in the product, so it rounds once like FSUB.
__device__ __forceinline__ F2 operator-(F2 x, F2 y) { return __ffma2_rn(y.v, make_float2(-1.f, -1.f), x.v); }
__device__ __forceinline__ F2 operator-(P2 p, F2 y) { return __ffma2_rn(p.a, p.b, neg2(y.v)); }
__device__ __forceinline__ F2 operator-(F2 y, P2 p) { return __ffma2_rn(neg2(p.a), p.b, y.v); }
__device__ __forceinline__ F2 operator-(P2 p, P2 q) { return __ffma2_rn(p.a, p.b, neg2(F2(q).v)); }
__device__ __forceinline__ F2 operator-(F2 x) { return neg2(x.v); }
__device__ __forceinline__ P2 operator-(P2 p) { return {neg2(p.a), p.b}; }

__device__ __forceinline__ F2& operator+=(F2& x, F2 y) { return x = x + y; }
__device__ __forceinline__ F2& operator+=(F2& x, P2 p) { return x = x + p; }
__device__ __forceinline__ F2& operator-=(F2& x, F2 y) { return x = x - y; }
__device__ __forceinline__ F2& operator-=(F2& x, P2 p) { return x = x - p; }

__device__ __forceinline__ F2 recip(F2 x) { return F2(make_float2(recip(x.v.x), recip(x.v.y))); }
__device__ __forceinline__ F2 rmul(F2 a, F2 b) { return F2(a * b); }  // rounded product (P2 -> F2)
__device__ __forceinline__ F2 fma_rn(F2 a, F2 b, F2 c) { return F2(__ffma2_rn(a.v, b.v, c.v)); }

template <>
__host__ __device__ inline F2 wgt<F2>(int q) { return F2(wgt<float>(q)); }

// ---------------------------------------------------------------- packed cascaded collision
// collide_cascaded without forcing, for two nodes, value for value the scalar
// code's results: the same sums and products in the same order, with signs
// moved by exact negation and doublings written as x + x.  The FP32x2
// instructions take register operands only, so an operation with a constant or
// a coefficient is done as two scalar instructions that take it as an immediate
// or from the constant bank: the same time on the FP32 pipe, and no register
// pairs or moves for the constants.  114 pipe operations per pair.
__device__ __forceinline__ float2 sub2(float2 x, float2 y) {
    float2 r;
    asm("{.reg .b64 a, b, c;\n mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %5};\n sub.rn.f32x2 c, a, b;\n mov.b64 {%0, %1}, c;}\n"
        : "=f"(r.x), "=f"(r.y) : "f"(x.x), "f"(x.y), "f"(y.x), "f"(y.y));
    return r;
}
__device__ __forceinline__ float2 smul(float c, float2 x) { return make_float2(__fmul_rn(c, x.x), __fmul_rn(c, x.y)); }
__device__ __forceinline__ float2 sfma(float c, float2 x, float2 y) {
    return make_float2(__fmaf_rn(c, x.x, y.x), __fmaf_rn(c, x.y, y.y));
}
__device__ __forceinline__ float2 sadd(float c, float2 x) { return make_float2(__fadd_rn(c, x.x), __fadd_rn(c, x.y)); }

__device__ __forceinline__ void collide_cascaded_pair(float2 d[9], const float* __restrict__ k) {
#define A2 __fadd2_rn
#define M2 __fmul2_rn
#define F2M __ffma2_rn
    const float2 s13 = A2(d[1], d[3]), s24 = A2(d[2], d[4]);
    const float2 s56 = A2(d[5], d[6]), s78 = A2(d[7], d[8]), s58 = A2(d[5], d[8]), s67 = A2(d[6], d[7]);
    const float2 kxxyy = A2(s56, s78);
    const float2 kxx = A2(s13, kxxyy), kyy = A2(s24, kxxyy);
    const float2 drho = A2(A2(d[0], s13), kyy);
    const float2 rho = sadd(k[K_RHO0], drho);
    const float2 kxxy = sub2(s56, s78), kxyy = sub2(s58, s67);
    const float2 jx = A2(sub2(d[1], d[3]), kxyy), jy = A2(sub2(d[2], d[4]), kxxy);
    const float2 nkxy = sub2(A2(d[6], d[8]), A2(d[5], d[7]));
    const float2 inv = make_float2(recip(rho.x), recip(rho.y));
    const float2 ux = M2(jx, inv), uy = M2(jy, inv);
    const float2 uxx = M2(ux, ux), uyy = M2(uy, uy), uxy = M2(ux, uy);
    const float nr3 = -__fmul_rn(k[K_RHO0], float(1.0 / 3.0));
    const float2 nkxxt = make_float2(__fsub_rn(nr3, kxx.x), __fsub_rn(nr3, kxx.y));
    const float2 nkyyt = make_float2(__fsub_rn(nr3, kyy.x), __fsub_rn(nr3, kyy.y));
    // Eq. (17)-(19)
    const float2 g3 = smul(k[K_C3], sub2(F2M(rho, A2(uxx, uyy), smul(float(2.0 / 3.0), drho)), A2(kxx, kyy)));
    const float2 X4 = F2M(rho, sub2(uxx, uyy), sub2(kyy, kxx));
    const float2 g4 = smul(k[K_C3 + 1], X4), ng4 = smul(-k[K_C3 + 1], X4);
    const float2 ng5 = smul(-k[K_C3 + 2], F2M(rho, uxy, nkxy));
    const float2 A = sfma(3.f, g3, g4), B = sfma(3.f, g3, ng4);
    const float2 ux2 = A2(ux, ux), uy2 = A2(uy, uy), rho2 = A2(rho, rho);
    const float2 hux = smul(-0.5f, ux), huy = smul(-0.5f, uy);
    // Eq. (20)-(21)
    const float2 X6 = F2M(uy, nkxxt, F2M(ux2, nkxy, F2M(M2(rho2, uxx), uy, kxxy)));
    const float2 h6 = M2(huy, A);
    const float2 g6 = F2M(ux2, ng5, sfma(k[K_C3 + 3], X6, h6));
    const float2 X7 = F2M(ux, nkyyt, F2M(uy2, nkxy, F2M(M2(rho2, ux), uyy, kxyy)));
    const float2 h7 = M2(hux, B);
    const float2 g7 = F2M(uy2, ng5, sfma(k[K_C3 + 4], X7, h7));
    // Eq. (22)
    const float2 uxy4 = smul(4.f, uxy);
    float2 G8 = make_float2(__fmaf_rn(float(1.0 / 9.0), drho.x, -kxxyy.x), __fmaf_rn(float(1.0 / 9.0), drho.y, -kxxyy.y));
    G8 = F2M(M2(smul(3.f, rho), uxx), uyy, G8);
    G8 = sfma(2.f, F2M(ux, kxyy, M2(uy, kxxy)), G8);
    G8 = F2M(uxx, nkyyt, G8);
    G8 = F2M(uyy, nkxxt, G8);
    G8 = F2M(uxy4, nkxy, G8);
    float2 g8 = sfma(k[K_C3 + 5], G8, smul(-2.f, g3));
    g8 = sfma(-0.5f, F2M(uyy, A, M2(uxx, B)), g8);
    g8 = F2M(uxy4, ng5, g8);
    g8 = sfma(-2.f, F2M(uy, g6, M2(ux, g7)), g8);
    // Eq. (25)
    const float2 t = sfma(2.f, g3, g8), a = sub2(g4, g3), b = sub2(ng4, g3);
    d[0] = sfma(4.f, sub2(g8, g3), d[0]);
    d[1] = A2(d[1], sfma(2.f, sub2(g7, g8), a));
    d[3] = A2(d[3], sfma(-2.f, A2(g7, g8), a));
    d[2] = A2(d[2], sfma(2.f, sub2(g6, g8), b));
    d[4] = A2(d[4], sfma(-2.f, A2(g6, g8), b));
    const float2 np = A2(ng5, g6), q = sub2(g6, ng5);
    d[5] = A2(d[5], sub2(sub2(t, np), g7));
    d[6] = A2(d[6], A2(sub2(t, q), g7));
    d[7] = A2(d[7], A2(A2(t, q), g7));
    d[8] = A2(d[8], sub2(A2(t, np), g7));
#undef A2
#undef M2
#undef F2M
}

// Coefficients of both nodes (the same lattice-wide constants).
__device__ __forceinline__ Coef<F2> pair_coef(const Args& a) {
    const Coef<float> s(a);
    Coef<F2> c;
    c.c3 = s.c3; c.c4 = s.c4; c.c5 = s.c5; c.c6 = s.c6; c.c7 = s.c7; c.c8 = s.c8;
    c.w3 = s.w3; c.w4 = s.w4; c.w5 = s.w5; c.w6 = s.w6; c.w7 = s.w7; c.w8 = s.w8;
    c.rho0 = s.rho0;
    return c;
}

// Nodes (x, y) and (x, y + 1) of an interior or periodic region (no wall
// links); `two` is false when y + 1 is past the last row (its lane is idle).
template <int MODEL, int STORE, bool ODD, int FORCE>
__device__ __forceinline__ void step_pair(const Args& a, int x, int y, bool two) {
    float d0[9], d1[9];
    load_node<STORE, ODD, false>(a, x, y, d0);
    if (two) load_node<STORE, ODD, false>(a, x, y + 1, d1);
    else {
#pragma unroll
        for (int q = 0; q < 9; ++q) d1[q] = d0[q];
    }
    float fx0, fy0, fx1 = 0.f, fy1 = 0.f;
    node_force<float, FORCE>(a, x, y, fx0, fy0);
    if (FORCE != 0) {
        if (two) node_force<float, FORCE>(a, x, y + 1, fx1, fy1);
        else { fx1 = fx0; fy1 = fy0; }
    }
    F2 d[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) d[q] = F2(make_float2(d0[q], d1[q]));
    const Coef<F2> c = pair_coef(a);
    collide<MODEL, F2, (FORCE != 0)>(d, F2(make_float2(fx0, fx1)), F2(make_float2(fy0, fy1)), c);
#pragma unroll
    for (int q = 0; q < 9; ++q) { d0[q] = d[q].v.x; d1[q] = d[q].v.y; }
    store_node<STORE, ODD, false>(a, x, y, d0, 0u);
    if (two) store_node<STORE, ODD, false>(a, x, y + 1, d1, 0u);
}

}  // namespace lbm
