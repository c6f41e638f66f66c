// The increment-form collision (lbm_vec.cuh) on plain floats for the kernels of the appendices' models,
// contracted by the compiler.  The current of the magnetic field and the recolouring direction are
// small differences of the populations and amplify the last bit of a step by some hundred, so these
// kernels keep their order of operations.
#pragma once

#include "lbm_device.cuh"

namespace cmlbm {

// No change of the equilibrium.
struct NoExtra {
    __device__ __forceinline__ void operator()(float (&)[3][3][3], float, float, float, float, float) const {}
};

// One D1Q3 raw-moment sum along an axis: values at c = -1, 0, +1 -> moments 0, 1, 2.
__device__ __forceinline__ void d1q3_moments(float pm, float p0, float pp, float& m0, float& m1, float& m2) {
    const float s2 = pp + pm;
    m0 = s2 + p0;
    m1 = pp - pm;
    m2 = s2;
}

// One D1Q3 shift from raw to central moments about u, in deviation form: inputs are raw moments
// minus r*(1, 0, 1/3), outputs central moments minus r*(1, 0, 1/3).
__device__ __forceinline__ void d1q3_shift_dev(float& m0, float& m1, float& m2, float r, float u) {
    const float A = r + m0;
    const float c1 = m1 - u * A;
    const float c2 = m2 - 2.0f * u * m1 + u * u * A;
    m1 = c1;
    m2 = c2;
}

// One D1Q3 inverse without rest state (a linear map): central moments (m0, m1, m2) about u ->
// values at c = -1, 0, +1.
__device__ __forceinline__ void d1q3_inverse_lin(float m0, float m1, float m2, float u, float u2, float& pm,
                                                 float& p0, float& pp) {
    const float t = m0 * u2 + m2 + 2.0f * u * m1;
    const float a = m0 * u + m1;
    p0 = m0 - t;
    pp = 0.5f * (t + a);
    pm = 0.5f * (t - a);
}

// In: K[x][y][z] holds the deviations g arranged by velocity (index c + 1).  Out: K holds the
// increments dg arranged the same way.  Returns rho and u of the node.  extra(K, rho, ux, uy,
// uz, omega) may add further equilibrium terms to the increments before the inverse transform.
template <typename Extra>
__device__ __forceinline__ Macro model_increment(float (&K)[3][3][3], float Fx, float Fy, float Fz, float omega,
                                                   float rho0, const Extra& extra) {
    constexpr float s[3] = {1.0f, 0.0f, 1.0f / 3.0f};

    // raw moments of the deviations: z, then y, then x (index: [x][y][z], each either a velocity
    // c + 1 or a moment order)
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) d1q3_moments(K[a][b][0], K[a][b][1], K[a][b][2], K[a][b][0], K[a][b][1], K[a][b][2]);
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int c = 0; c < 3; ++c) d1q3_moments(K[a][0][c], K[a][1][c], K[a][2][c], K[a][0][c], K[a][1][c], K[a][2][c]);
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int c = 0; c < 3; ++c) d1q3_moments(K[0][b][c], K[1][b][c], K[2][b][c], K[0][b][c], K[1][b][c], K[2][b][c]);

    // step 1: macroscopic variables (Eq. macroscopic)
    const float dr = K[0][0][0];
    const float rho = rho0 + dr;
    const float inv = 1.0f / rho;
    const float ux = (K[1][0][0] + 0.5f * Fx) * inv;
    const float uy = (K[0][1][0] + 0.5f * Fy) * inv;
    const float uz = (K[0][0][1] + 0.5f * Fz) * inv;

    // step 2: central moments (deviation form), x then y then z shifts
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int c = 0; c < 3; ++c) d1q3_shift_dev(K[0][b][c], K[1][b][c], K[2][b][c], rho0 * s[b] * s[c], ux);
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int c = 0; c < 3; ++c) d1q3_shift_dev(K[a][0][c], K[a][1][c], K[a][2][c], rho0 * s[a] * s[c], uy);
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) d1q3_shift_dev(K[a][b][0], K[a][b][1], K[a][b][2], rho0 * s[a] * s[b], uz);

    // step 3: increments k* - k.  k4..k6 = kappa_110, 101, 011 relax at omega; k7 = k200 - k020,
    // k8 = k200 - k002 at omega; k9 = k200 + k020 + k002 -> rho; every other moment goes to its
    // post-collision value of Eq. post_collision_central_moments_forcing (rate 1).
    const float k7 = K[2][0][0] - K[0][2][0];
    const float k8 = K[2][0][0] - K[0][0][2];
    const float om1 = 1.0f - omega;
    const float k7s = om1 * k7, k8s = om1 * k8;
    const float third = 1.0f / 3.0f;
    K[0][0][0] = 0.0f;
    K[1][0][0] = Fx;
    K[0][1][0] = Fy;
    K[0][0][1] = Fz;
    K[1][1][0] = -omega * K[1][1][0];
    K[1][0][1] = -omega * K[1][0][1];
    K[0][1][1] = -omega * K[0][1][1];
    K[2][0][0] = (k7s + k8s + dr) * third - K[2][0][0];
    K[0][2][0] = (dr - 2.0f * k7s + k8s) * third - K[0][2][0];
    K[0][0][2] = (dr + k7s - 2.0f * k8s) * third - K[0][0][2];
    const float fx6 = Fx * (1.0f / 6.0f), fy6 = Fy * (1.0f / 6.0f), fz6 = Fz * (1.0f / 6.0f);
    K[1][2][0] = fx6 - K[1][2][0];
    K[1][0][2] = fx6 - K[1][0][2];
    K[2][1][0] = fy6 - K[2][1][0];
    K[0][1][2] = fy6 - K[0][1][2];
    K[2][0][1] = fz6 - K[2][0][1];
    K[0][2][1] = fz6 - K[0][2][1];
    K[1][1][1] = -K[1][1][1];
    const float dr9 = dr * (1.0f / 9.0f);
    K[2][2][0] = dr9 - K[2][2][0];
    K[2][0][2] = dr9 - K[2][0][2];
    K[0][2][2] = dr9 - K[0][2][2];
    K[2][1][1] = -K[2][1][1];
    K[1][2][1] = -K[1][2][1];
    K[1][1][2] = -K[1][1][2];
    K[1][2][2] = Fx * (1.0f / 18.0f) - K[1][2][2];
    K[2][1][2] = Fy * (1.0f / 18.0f) - K[2][1][2];
    K[2][2][1] = Fz * (1.0f / 18.0f) - K[2][2][1];
    K[2][2][2] = dr * (1.0f / 27.0f) - K[2][2][2];
    extra(K, rho, ux, uy, uz, omega);

    // step 4: dg = (T^T)^-1 dk, z then y then x inverses; g* = g + dg
    const float ux2 = ux * ux, uy2 = uy * uy, uz2 = uz * uz;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b)
            d1q3_inverse_lin(K[a][b][0], K[a][b][1], K[a][b][2], uz, uz2, K[a][b][0], K[a][b][1], K[a][b][2]);
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int c = 0; c < 3; ++c)
            d1q3_inverse_lin(K[a][0][c], K[a][1][c], K[a][2][c], uy, uy2, K[a][0][c], K[a][1][c], K[a][2][c]);
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int c = 0; c < 3; ++c)
            d1q3_inverse_lin(K[0][b][c], K[1][b][c], K[2][b][c], ux, ux2, K[0][b][c], K[1][b][c], K[2][b][c]);
    return Macro{rho, ux, uy, uz};
}

template <typename Extra = NoExtra>
__device__ __forceinline__ Macro model_collide(float (&g)[27], float Fx, float Fy, float Fz, float omega, float rho0,
                                               const Extra& extra = Extra()) {
    float K[3][3][3];
#pragma unroll
    for (int i = 0; i < 27; ++i) K[dir_x(i) + 1][dir_y(i) + 1][dir_z(i) + 1] = g[i];
    const Macro m = model_increment(K, Fx, Fy, Fz, omega, rho0, extra);
#pragma unroll
    for (int i = 0; i < 27; ++i) g[i] += K[dir_x(i) + 1][dir_y(i) + 1][dir_z(i) + 1];
    return m;
}

}  // namespace cmlbm
