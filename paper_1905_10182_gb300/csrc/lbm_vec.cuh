// The central-moment collision on one node (F1) or on a pair of nodes in packed FP32 registers (V2),
// from the same source: every operation is one explicitly rounded instruction per node (fma, add, mul;
// the compiler neither contracts nor splits them), so that a node's result is the same to the bit
// whichever kernel updates it.  Included by lbm_device.cuh.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace cmlbm {

// One node.
struct F1 {
    float v;
};
// A pair of nodes, one instruction for both (.x: first node, .y: second node).
struct V2 {
    float2 v;
};

template <typename T>
__device__ __forceinline__ T splat(float a);
template <>
__device__ __forceinline__ F1 splat<F1>(float a) { return F1{a}; }
template <>
__device__ __forceinline__ V2 splat<V2>(float a) { return V2{make_float2(a, a)}; }
__device__ __forceinline__ V2 bc(float a) { return splat<V2>(a); }

__device__ __forceinline__ F1 operator+(F1 a, F1 b) { return F1{__fadd_rn(a.v, b.v)}; }
__device__ __forceinline__ F1 operator-(F1 a, F1 b) { return F1{__fsub_rn(a.v, b.v)}; }
__device__ __forceinline__ F1 operator-(F1 a) { return F1{-a.v}; }
__device__ __forceinline__ F1 operator*(F1 a, F1 b) { return F1{__fmul_rn(a.v, b.v)}; }
__device__ __forceinline__ F1 operator*(float a, F1 b) { return F1{__fmul_rn(a, b.v)}; }
__device__ __forceinline__ F1 operator*(F1 a, float b) { return F1{__fmul_rn(a.v, b)}; }
__device__ __forceinline__ F1 operator+(F1 a, float b) { return F1{__fadd_rn(a.v, b)}; }
__device__ __forceinline__ F1& operator+=(F1& a, F1 b) {
    a = a + b;
    return a;
}
__device__ __forceinline__ F1 vfma(F1 a, F1 b, F1 c) { return F1{__fmaf_rn(a.v, b.v, c.v)}; }
__device__ __forceinline__ F1 vfma(float a, F1 b, F1 c) { return F1{__fmaf_rn(a, b.v, c.v)}; }
__device__ __forceinline__ F1 vrcp(F1 a) { return F1{__frcp_rn(a.v)}; }

__device__ __forceinline__ V2 operator+(V2 a, V2 b) { return V2{__fadd2_rn(a.v, b.v)}; }
__device__ __forceinline__ V2 operator-(V2 a, V2 b) { return V2{__ffma2_rn(b.v, make_float2(-1.0f, -1.0f), a.v)}; }
__device__ __forceinline__ V2 operator-(V2 a) { return V2{__fmul2_rn(a.v, make_float2(-1.0f, -1.0f))}; }
__device__ __forceinline__ V2 operator*(V2 a, V2 b) { return V2{__fmul2_rn(a.v, b.v)}; }
__device__ __forceinline__ V2 operator*(float a, V2 b) { return V2{__fmul2_rn(make_float2(a, a), b.v)}; }
__device__ __forceinline__ V2 operator*(V2 a, float b) { return V2{__fmul2_rn(a.v, make_float2(b, b))}; }
__device__ __forceinline__ V2 operator+(V2 a, float b) { return V2{__fadd2_rn(a.v, make_float2(b, b))}; }
__device__ __forceinline__ V2& operator+=(V2& a, V2 b) {
    a = a + b;
    return a;
}
__device__ __forceinline__ V2 vfma(V2 a, V2 b, V2 c) { return V2{__ffma2_rn(a.v, b.v, c.v)}; }
__device__ __forceinline__ V2 vfma(float a, V2 b, V2 c) { return V2{__ffma2_rn(make_float2(a, a), b.v, c.v)}; }
__device__ __forceinline__ V2 vrcp(V2 a) { return V2{make_float2(__frcp_rn(a.v.x), __frcp_rn(a.v.y))}; }

// rho and u of a node or a pair.
template <typename T>
struct MacroT {
    T rho, ux, uy, uz;
};

// Models with second-order Hermite truncations (Sec. III: M4 keeps the complete equilibrium with
// the second-order (Guo) forcing term, M5 truncates both at second order).  For any truncation
// order >= 2 the central moments of order <= 2 of f^eq and of F_i are those of the complete
// expansion (the D3Q27 quadrature is exact there), so the five omega-relaxed moments k4..k8 are
// untouched and only the moments of order >= 3, all relaxed at rate 1 (k* = k^eq + R/2), change.
// Adds to the monomial post-collision central moments K[a][b][c] (x, y, z orders):
//   ce * (kappa^eq of the 2nd-order equilibrium - kappa^eq of the complete one)
// + cf * (kappa of the 2nd-order forcing term - kappa of the complete one),
// ce = 1 for a second-order equilibrium, cf = 1/2 for a second-order forcing term, else 0.
// The differences are the central moments of the dropped Hermite terms H^(3)..H^(6) of
// Eq. eq:truncation and Eq. generalForcing, expanded about u.
// T: float, F1 or V2.
template <typename T>
__device__ __forceinline__ void hermite2_correction(T (&K)[3][3][3], T rho, T ux, T uy, T uz, T Fx, T Fy, T Fz,
                                                    float ce, float cf) {
    const T re = ce * rho;
    const T X = ux * ux, Y = uy * uy, Z = uz * uz;
    // third order, kappa with u_a squared and u_b: -rho u_a^2 u_b; -u_a (2 F_a u_b + F_b u_a)
    auto t3 = [&](T ua, T ub, T Fa, T Fb) {
        return -re * ua * ua * ub - cf * ua * (2.0f * Fa * ub + Fb * ua);
    };
    K[2][1][0] += t3(ux, uy, Fx, Fy);
    K[2][0][1] += t3(ux, uz, Fx, Fz);
    K[1][2][0] += t3(uy, ux, Fy, Fx);
    K[0][2][1] += t3(uy, uz, Fy, Fz);
    K[1][0][2] += t3(uz, ux, Fz, Fx);
    K[0][1][2] += t3(uz, uy, Fz, Fy);
    K[1][1][1] += -re * ux * uy * uz - cf * (Fx * uy * uz + Fy * ux * uz + Fz * ux * uy);
    // fourth order, a^2 b^2: 3 rho u_a^2 u_b^2; 4 u_a u_b (F_a u_b + F_b u_a)
    auto t4 = [&](T ua, T ub, T Fa, T Fb) {
        return 3.0f * re * ua * ua * ub * ub + 4.0f * cf * ua * ub * (Fa * ub + Fb * ua);
    };
    K[2][2][0] += t4(ux, uy, Fx, Fy);
    K[2][0][2] += t4(ux, uz, Fx, Fz);
    K[0][2][2] += t4(uy, uz, Fy, Fz);
    // fourth order, a^2 b c: 3 rho u_a^2 u_b u_c; 2 u_a (2 F_a u_b u_c + F_b u_a u_c + F_c u_a u_b)
    auto t4m = [&](T ua, T ub, T uc, T Fa, T Fb, T Fc) {
        return 3.0f * re * ua * ua * ub * uc + 2.0f * cf * ua * (2.0f * Fa * ub * uc + Fb * ua * uc + Fc * ua * ub);
    };
    K[2][1][1] += t4m(ux, uy, uz, Fx, Fy, Fz);
    K[1][2][1] += t4m(uy, ux, uz, Fy, Fx, Fz);
    K[1][1][2] += t4m(uz, ux, uy, Fz, Fx, Fy);
    // fifth order, a b^2 c^2: -rho u_a (18 u_b^2 u_c^2 + u_b^2 + u_c^2) / 3;
    // -(F_a (9 u_b^2 u_c^2 + u_b^2 + u_c^2) + 2 u_a (F_b u_b (9 u_c^2 + 1) + F_c u_c (9 u_b^2 + 1))) / 3
    auto t5 = [&](T ua, T ub, T uc, T Fa, T Fb, T Fc) {
        const T b2 = ub * ub, c2 = uc * uc;
        return -(re * ua * (18.0f * b2 * c2 + b2 + c2) +
                 cf * (Fa * (9.0f * b2 * c2 + b2 + c2) +
                       2.0f * ua * (Fb * ub * (9.0f * c2 + 1.0f) + Fc * uc * (9.0f * b2 + 1.0f)))) *
               (1.0f / 3.0f);
    };
    K[1][2][2] += t5(ux, uy, uz, Fx, Fy, Fz);
    K[2][1][2] += t5(uy, ux, uz, Fy, Fx, Fz);
    K[2][2][1] += t5(uz, ux, uy, Fz, Fx, Fy);
    // sixth order: rho (10 X Y Z + X Y + X Z + Y Z); (4/3) sum_a F_a u_a (6 u_b^2 u_c^2 + u_b^2 + u_c^2)
    K[2][2][2] += re * (10.0f * X * Y * Z + X * Y + X * Z + Y * Z) +
                  cf * (4.0f / 3.0f) *
                      (Fx * ux * (6.0f * Y * Z + Y + Z) + Fy * uy * (6.0f * X * Z + X + Z) +
                       Fz * uz * (6.0f * X * Y + X + Y));
}

// One D1Q3 shift from raw to central moments about u (nu = -u), in deviation form: inputs are raw
// moments minus r (1, 0, 1/3), outputs central moments minus r (1, 0, 1/3).  REST: r is not zero.
// m2 - 2 u m1 + u^2 A = m2 - u (m1 + c1), c1 = m1 - u A, A = r + m0.
template <bool REST, typename T>
__device__ __forceinline__ void d1q3_shift(T& m0, T& m1, T& m2, float r, T nu) {
    const T A = REST ? m0 + r : m0;
    const T c1 = vfma(nu, A, m1);
    m2 = vfma(nu, m1 + c1, m2);
    m1 = c1;
}

// One D1Q3 inverse (a linear map): central moments (m0, m1, m2) about u -> values at c = -1, 0, +1:
// a = m1 + u m0, t = m2 + u (a + m1); p0 = m0 - t, p(+-1) = (t +- a) / 2.
template <typename T>
__device__ __forceinline__ void d1q3_inverse(T& m0, T& m1, T& m2, T u) {
    const T a = vfma(m0, u, m1);
    const T t = vfma(u, a + m1, m2);
    const T p0 = m0 - t;
    const T ht = 0.5f * t;
    m2 = vfma(0.5f, a, ht);
    m0 = vfma(-0.5f, a, ht);
    m1 = p0;
}

// One D1Q3 raw-moment sum along an axis: values at c = -1, 0, +1 -> moments 0, 1, 2.
template <typename T>
__device__ __forceinline__ void d1q3_sums(T& pm, T& p0, T& pp) {
    const T s2 = pp + pm, d = pp - pm;
    pm = s2 + p0;
    p0 = d;
    pp = s2;
}

// The time iteration of Sec. II (steps 1-4) as an increment, so that FP32 rounding scales with the
// (small) change of each population rather than with the population:
//   k* - k = Lambda (k^eq - k) + (I - Lambda/2) R        (the post-collision CMs of Sec. II)
//   f*     = f + (T^T)^-1 (k* - k)                        (Eq. system; T^T is linear)
// In: K[x][y][z] holds the deviations g arranged by velocity (index c + 1).  Out: the increments dg
// arranged the same way.  The conserved increments are exact by construction: dk_000 = 0
// (k0* = k0 = rho) and dk_100 = F_x (k1 = -F_x/2 by Eq. macroscopic, k1* = F_x/2).
// HO: the second-order truncations of hermite2_correction (weights ce, cf).
template <bool HO, typename T>
__device__ __forceinline__ MacroT<T> collide_increment(T (&K)[3][3][3], T Fx, T Fy, T Fz, float omega, float rho0, float ce,
                                                       float cf) {
    constexpr float s[3] = {1.0f, 0.0f, 1.0f / 3.0f};
    // raw moments of the deviations: z, then y, then x
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) d1q3_sums(K[a][b][0], K[a][b][1], K[a][b][2]);
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int c = 0; c < 3; ++c) d1q3_sums(K[a][0][c], K[a][1][c], K[a][2][c]);
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int c = 0; c < 3; ++c) d1q3_sums(K[0][b][c], K[1][b][c], K[2][b][c]);

    // step 1: macroscopic variables (Eq. macroscopic)
    const T dr = K[0][0][0];
    const T rho = dr + rho0;
    const T inv = vrcp(rho);
    const T ux = vfma(0.5f, Fx, K[1][0][0]) * inv;
    const T uy = vfma(0.5f, Fy, K[0][1][0]) * inv;
    const T uz = vfma(0.5f, Fz, K[0][0][1]) * inv;

    // step 2: central moments (deviation form), x then y then z shifts; the rest moments of odd
    // order vanish
    const T nx = -ux, ny = -uy, nz = -uz;
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (b == 1 || c == 1) d1q3_shift<false>(K[0][b][c], K[1][b][c], K[2][b][c], 0.0f, nx);
            else d1q3_shift<true>(K[0][b][c], K[1][b][c], K[2][b][c], rho0 * (s[b] * s[c]), nx);
        }
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (a == 1 || c == 1) d1q3_shift<false>(K[a][0][c], K[a][1][c], K[a][2][c], 0.0f, ny);
            else d1q3_shift<true>(K[a][0][c], K[a][1][c], K[a][2][c], rho0 * (s[a] * s[c]), ny);
        }
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            if (a == 1 || b == 1) d1q3_shift<false>(K[a][b][0], K[a][b][1], K[a][b][2], 0.0f, nz);
            else d1q3_shift<true>(K[a][b][0], K[a][b][1], K[a][b][2], rho0 * (s[a] * s[b]), nz);
        }

    // step 3: increments k* - k.  k4..k6 = kappa_110, 101, 011 relax at omega; k7 = k200 - k020,
    // k8 = k200 - k002 at omega; k9 = k200 + k020 + k002 -> rho; every other moment goes to its
    // post-collision value of Eq. post_collision_central_moments_forcing (rate 1).
    const float third = 1.0f / 3.0f;
    const float nom = -omega, om1 = 1.0f - omega;
    const T k7s = om1 * (K[2][0][0] - K[0][2][0]), k8s = om1 * (K[2][0][0] - K[0][0][2]);
    K[0][0][0] = splat<T>(0.0f);
    K[1][0][0] = Fx;
    K[0][1][0] = Fy;
    K[0][0][1] = Fz;
    K[1][1][0] = nom * K[1][1][0];
    K[1][0][1] = nom * K[1][0][1];
    K[0][1][1] = nom * K[0][1][1];
    K[2][0][0] = vfma(third, k7s + k8s + dr, -K[2][0][0]);
    K[0][2][0] = vfma(third, vfma(-2.0f, k7s, k8s + dr), -K[0][2][0]);
    K[0][0][2] = vfma(third, vfma(-2.0f, k8s, k7s + dr), -K[0][0][2]);
    const float sixth = 1.0f / 6.0f, ninth = 1.0f / 9.0f, e18 = 1.0f / 18.0f;
    K[1][2][0] = vfma(sixth, Fx, -K[1][2][0]);
    K[1][0][2] = vfma(sixth, Fx, -K[1][0][2]);
    K[2][1][0] = vfma(sixth, Fy, -K[2][1][0]);
    K[0][1][2] = vfma(sixth, Fy, -K[0][1][2]);
    K[2][0][1] = vfma(sixth, Fz, -K[2][0][1]);
    K[0][2][1] = vfma(sixth, Fz, -K[0][2][1]);
    K[1][1][1] = -K[1][1][1];
    K[2][2][0] = vfma(ninth, dr, -K[2][2][0]);
    K[2][0][2] = vfma(ninth, dr, -K[2][0][2]);
    K[0][2][2] = vfma(ninth, dr, -K[0][2][2]);
    K[2][1][1] = -K[2][1][1];
    K[1][2][1] = -K[1][2][1];
    K[1][1][2] = -K[1][1][2];
    K[1][2][2] = vfma(e18, Fx, -K[1][2][2]);
    K[2][1][2] = vfma(e18, Fy, -K[2][1][2]);
    K[2][2][1] = vfma(e18, Fz, -K[2][2][1]);
    K[2][2][2] = vfma(1.0f / 27.0f, dr, -K[2][2][2]);
    if (HO) hermite2_correction(K, rho, ux, uy, uz, Fx, Fy, Fz, ce, cf);

    // step 4: dg = (T^T)^-1 dk, z then y then x inverses
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) d1q3_inverse(K[a][b][0], K[a][b][1], K[a][b][2], uz);
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int c = 0; c < 3; ++c) d1q3_inverse(K[a][0][c], K[a][1][c], K[a][2][c], uy);
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int c = 0; c < 3; ++c) d1q3_inverse(K[0][b][c], K[1][b][c], K[2][b][c], ux);
    return MacroT<T>{rho, ux, uy, uz};
}

}  // namespace cmlbm
