// The Gaussian mass of one map cell as a polynomial times one base-2 exponential.
//
// A cell of half-width t (in units of sigma) whose centre lies at distance z from a first-hit
// cell's centre holds the mass G_{k,j} of Theorem 1 as
//
//   int_{-t}^{t} phi(z + v) dv = 2 t phi(z) sum_i He_2i(z) u^i / (2i + 1)!,   u = t^2
//
// (Taylor's series of phi under the integral). In the scaled variable s = z^2 / (2 ln 2), phi(z) is
// 2^-s / sqrt(2 pi) and the sum a polynomial in s whose coefficients are polynomials in u: the
// former are formed once per cell, so a pair (j, k) costs one ex2 and D + 1 multiply-adds, against
// an ex2, an rcp and a degree-4 polynomial for each Phi of the boundary form. Powers above the
// degree D kept are folded into the lower ones (minimax under the weight 2^-s, by
// csrc/fit_cell_mass.py, which prints the tables below and the errors): the mass is off by at most
// 5.3e-8 of the cell's peak for D = 3 and sigma >= 1.5 cells (5e-9 at 2), 2.9e-8 for D = 4 and
// sigma >= 1 cell, for the widest cell of a grid (sqrt 2); narrower cells are closer still.
#pragma once

#include "gauss_tail.cuh"

namespace fsmi {

constexpr int kMassOrder = 6;  // powers of u in the coefficients

// smallest sigma (cells) at which the degree-3 and the degree-4 form are used for cells of a grid
constexpr float kMassSigma3 = 1.5f, kMassSigma4 = 1.0f;

// coefficient of u^k in the polynomial's coefficient of s^i (a constant at compile time once the
// loops over i and k are unrolled)
template <int D>
__device__ __forceinline__ constexpr float mass_table(int i, int k)
{
    static_assert(D == 3 || D == 4, "degrees of the table");
    constexpr float T3[4][kMassOrder + 1] = {
        {1.000000000e+00f, -1.666666667e-01f, 2.500000000e-02f, -2.976190476e-03f, 2.676682200e-04f, -1.947783638e-05f,
         1.220020016e-06f},
        {0.000000000e+00f, 2.310490602e-01f, -6.931471806e-02f, 1.237762822e-02f, -1.373548900e-03f, 1.140179606e-04f,
         -7.807502158e-06f},
        {0.000000000e+00f, 0.000000000e+00f, 1.601510046e-02f, -5.719678737e-03f, 8.055896085e-04f, -7.624191733e-05f,
         5.674122182e-06f},
        {0.000000000e+00f, 0.000000000e+00f, 0.000000000e+00f, 5.286105587e-04f, -9.742741740e-05f, 1.046827153e-05f,
         -8.406810390e-07f}};
    constexpr float T4[5][kMassOrder + 1] = {
        {1.000000000e+00f, -1.666666667e-01f, 2.500000000e-02f, -2.976190476e-03f, 2.893518519e-04f, -2.277771230e-05f,
         1.488274530e-06f},
        {0.000000000e+00f, 2.310490602e-01f, -6.931471806e-02f, 1.237762822e-02f, -1.604507362e-03f, 1.520798211e-04f,
         -1.126854123e-05f},
        {0.000000000e+00f, 0.000000000e+00f, 1.601510046e-02f, -5.719678737e-03f, 1.112159754e-03f, -1.302253590e-04f,
         1.096989153e-05f},
        {0.000000000e+00f, 0.000000000e+00f, 0.000000000e+00f, 5.286105587e-04f, -2.055707728e-04f, 3.060835527e-05f,
         -2.929253685e-06f},
        {0.000000000e+00f, 0.000000000e+00f, 0.000000000e+00f, 0.000000000e+00f, 1.017791440e-05f, -1.988617659e-06f,
         2.152965038e-07f}};
    return D == 3 ? T3[i & 3][k] : T4[i][k];
}

// A source cell: centre x (scaled) and the coefficients of its mass as a polynomial in s = d^2
// (without its C_k), each twice for the packed operations.
template <int D>
struct MassSource {
    f32x2 x, c[D + 1];
};

// From the centre and width of a cell, both in the scaled variable.
template <int D>
__device__ __forceinline__ MassSource<D> mass_source(float x, float w)
{
    constexpr float kHalf = 0.58870501125773734f;   // sqrt(2 ln 2) / 2: scaled width -> t = half width in sigma
    constexpr float kNorm = 0.79788456080286536f;   // 2 / sqrt(2 pi)
    const float t = kHalf * w, u = t * t, a = kNorm * t;
    MassSource<D> m;
    m.x = pack2(x, x);
#pragma unroll
    for (int i = 0; i <= D; ++i) {
        float v = mass_table<D>(i, kMassOrder);
#pragma unroll
        for (int k = kMassOrder - 1; k >= (i < 1 ? 0 : i); --k) v = fmaf(v, u, mass_table<D>(i, k));
#pragma unroll
        for (int k = 0; k < i; ++k) v *= u;  // row i starts at u^i
        v *= a;
        m.c[i] = pack2(v, v);
    }
    return m;
}

// acc + (P_0 G(x_0 - x), P_1 G(x_1 - x)) for two targets at scaled positions X with weights P
template <int D>
__device__ __forceinline__ f32x2 mass_term(const MassSource<D> &m, f32x2 X, f32x2 P, f32x2 acc)
{
    const f32x2 d = sub2(X, m.x), s = mul2(d, d);
    float s0, s1;
    unpack2(s, s0, s1);
    const f32x2 t = mul2(pack2(ex2_approx(-s0), ex2_approx(-s1)), P);
    f32x2 q = m.c[D];
#pragma unroll
    for (int i = D - 1; i >= 0; --i) q = fma2(q, s, m.c[i]);
    return fma2(t, q, acc);
}

}  // namespace fsmi
