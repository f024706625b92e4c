// 2D hot path (device code shared by the 2D and mixed kernels): fixed-point ray traversal,
// first-hit probabilities, C_k and the FSMI / Approx-FSMI / Uniform-FSMI pair sums, one warp per beam.
//
// Per beam (Section 3): the traversal lists the cells the beam crosses with entry distances
// l_1 = 0 < l_2 < ... and end l_{n+1}; Algorithm 2 gives P(e_j) = o_j prod_{i<j}(1 - o_i);
// Algorithm 3 gives C_k = sum_{i<k} f(delta_emp, r_i) + f(delta_occ, r_k); the variant then sums
//   FSMI (Theorem 1):         sum_j P(e_j) sum_{k=1..n} C_k G_{k,j}
//   Approx (eq. fsmi_approx): the same with |k - j| <= Delta
//   Uniform (Algorithm 4):    sum_j P(e_j) (D_{min(n,j+H)} - D_{max(0,j-H-1)}) / (2H + 1)
//
// The exact Gaussian sum of grid cells with sigma >= 1 cell takes the mass form (cell_mass.cuh, exact_mass_sum):
// per source cell k its mass as a polynomial times one exponential, every term non-negative. Everything else
// Gaussian (smaller sigma, explicit beams and cells wider than the form's table, Approx-FSMI) is evaluated per
// first-hit cell j in boundary form (summation by parts):
//   S_j = sum_k C_k (Phi(x_{k+1}) - Phi(x_k)) = C_j + sum_{m=1}^{n+1} (C_m - C_{m-1}) sgn(x_m) T(|x_m|)
// with x_m = (l_m - mu_j) / sigma, C_0 = C_{n+1} = 0 and T the upper Gaussian tail. Every term is
// a tail mass, so no difference of two values near 1 is formed in FP32, and each (j, m) pair costs
// one tail evaluation (gauss_tail.cuh) instead of the two Phi values of G_{k,j}. The sign is taken
// from the indices (boundaries m <= j lie before the centre of cell j), not from the FP32
// difference, which is 0 for a cell shorter than the FP32 resolution of its distance.
#pragma once

#include "../../include/fsmi.h"
#include "fsmi_device.cuh"
#include "dda2d.cuh"
#include "fsmi_internal.h"
#include "gauss_tail.cuh"
#include "cell_mass.cuh"

namespace fsmi {

// ---- pair sums ------------------------------------------------------------------------------------

// per-warp shared arrays, in units of `stride` floats: l, scratch (ids / f_emp / D / dC), C, P
constexpr int kArrays2D = 4;
// Padding boundaries before index 0 and after index n + 1 of the exact sum's boundary pairs
// (l = -+3e30, dC = 0: their terms are exactly zero), so that its loops can run past a beam's ends.
constexpr int kPad2D = 32;
constexpr int kPadPairs = kPad2D / 2;

// Floats between consecutive arrays for beams of up to nmax cells (n + 2 boundaries + padding).
__host__ __device__ constexpr int stride_2d(int nmax) { return ((nmax + 2 + kPad2D) + 3) & ~3; }
// Floats of one warp's arrays: kArrays2D strides and the front padding of the boundary pairs.
__host__ __device__ constexpr int warp_floats_2d(int stride) { return kArrays2D * stride + 2 * kPad2D; }

// One warp's arrays in its region `base` (16-byte aligned): [pad | l | scratch | C | P]. The pad,
// l and scratch arrays are contiguous: the exact sum rebuilds them in place as boundary pairs.
__device__ __forceinline__ void carve_2d(float *base, int stride, float *&sl, float *&sc, float *&sp, float *&sx)
{
    sl = base + 2 * kPad2D;
    sx = sl + stride;
    sc = sx + stride;
    sp = sc + stride;
}
// Internal variant ids beside FSMI_EXACT (boundary form), FSMI_APPROX and FSMI_UNIFORM: the full
// n(n+1) sweep of the boundary form (FSMI_FLAG_FULL_SWEEP), and the exact sum in the mass form of
// degree 3 and 4.
constexpr int kExactFullSweep = 3, kExactMass3 = 4, kExactMass4 = 5;
__host__ __device__ constexpr bool mass_variant(int v) { return v == kExactMass3 || v == kExactMass4; }

// The kernel variant of a call whose cells come from the grid (widths of at most sqrt 2 cells along unit vectors;
// a beam along a shorter vector, whose cells are wider than the form's table covers, takes the boundary form by
// itself, see beam_sum).
// The exact sum takes the mass form (cell_mass.cuh) from sigma = 1 cell on; below that, and for
// explicit beams, whose cells may be any width, the boundary form. Approx-FSMI stays in boundary form:
// its band is too short to pay for the sources' polynomials (Delta = 3, 517 poses x 181 beams, R = 181.5:
// 274 us in mass form, 250 us in boundary form). The exact sum of the 2048x2048 office batch (1024
// poses x 360 beams, R = 256, sigma = 2) took 1.69 ms in mass form, 1.86 ms in boundary form, both before the
// traversal in closed form and with a cut of 4.58 for the masses (1.72 ms with both and the present cuts).
// From sigma = 1 to 1.5 the degree-4 form is kept for its error, not its time: 512 poses on the same map at sigma 1.0 /
// 1.2 / 1.45 take 759 / 796 / 850 us, in boundary form 688 / 743 / 801 us, but on random cells at 1.49 its largest error is
// 7.1e-7 against 1.8e-6. At sigma 1.5 and 2 the degree-3 form takes 777 and 875 us (boundary form 819 and 943, before the
// traversal in closed form).
inline int grid_variant(const DevParams &p)
{
    if (p.variant != FSMI_EXACT) return p.variant;
    if (p.sigma < kMassSigma4) return p.flags & FSMI_FLAG_FULL_SWEEP ? kExactFullSweep : FSMI_EXACT;
    return p.sigma >= kMassSigma3 ? kExactMass3 : kExactMass4;
}

enum { kSrcMap = 0, kSrcBeams = 1, kSrcSets = 2, kSrcTraj = 3 };

struct Src2D {
    // map source (kSrcMap, kSrcSets)
    const float *map;
    int W, H;
    const int32_t *poses;
    int P;
    const int32_t *dirs;
    int B;
    const float4 *gains;  // optional per-map-cell (o, f_occ, f_emp, 0)
    // explicit-beam source (kSrcBeams)
    const int32_t *off;
    const float *o;
    const float *l;
    const float *lend;
    // candidate sets (kSrcSets): device array of nsets descriptors
    const fsmi_set_2d *sets;
    int nsets;
    // trajectories (kSrcTraj, poses and beams as kSrcMap): states traj_off[t] .. traj_off[t+1]-1,
    // stamp[t][cell] = first state of trajectory t whose beams visit the cell
    const int32_t *traj_off;
    int T;
    const int32_t *stamp;
};

// Largest scaled distance whose tail is not flushed to zero: beyond |d| = 11.3 the factor
// 2^(-d^2) <= 2^(-127.69) is subnormal and ex2.approx.ftz returns exactly 0, so the term is +-0.
constexpr float kTailCut = 11.3f;
// Default window of the boundary form: T(4.81) = 7.4e-9 < 2^-27. Boundaries come at most two per
// major-axis crossing interval (scaled length >= cs = sqrt(log2 e) / (sigma sqrt 2)), so the terms
// skipped on one side weigh at most 2 T(4.81) / (1 - 2^(-9.62 cs)) times max |C_m - C_{m-1}|:
// at most 2^-24 of it (one FP32 ulp) for sigma up to 19 cells (1.01 x 2^-24 at 20), below 2^-25
// for sigma <= 2.
constexpr float kTailCutDefault = 4.81f;

// ---- the exact pair sum over boundary pairs ------------------------------------------------------
//
// Boundary pairs: Q[P] = (l_{2P}, l_{2P+1}, dC_{2P}, dC_{2P+1}) with scaled distances l and
// dC_m = C_m - C_{m-1} (C_{-1} = C_n = 0), for P in [-kPadPairs, n / 2 + 1 + kPadPairs); pairs
// past either end of the beam are padding (l = -+3e30, dC = 0). One 16-byte shared load gives a
// pair's two distances and two weights.
//
// Built in place over the traversal's distances sl and the scratch array after them (ids, then
// f_emp, both dead by now), from the top pair down: writing Q[P] overwrites l_{4P} .. l_{4P+3},
// which only Q[2P] and Q[2P+1] read, and those lie higher (P >= 1) or in the same step of 32 pairs,
// whose reads all come before its writes.
__device__ __forceinline__ void build_pairs(float *sl, const float *sc, int n, float cs)
{
    const int lane = lane_id();
    float4 *Q = reinterpret_cast<float4 *>(sl);
    const int pend = (n >> 1) + 1 + kPadPairs;  // pairs 0 .. pend - 1 (the last kPadPairs all padding)
    for (int top = pend; top > 0; top -= 32) {
        const int P = top - 32 + lane;
        float4 v = make_float4(3.0e30f, 3.0e30f, 0.0f, 0.0f);
        if (P >= 0) {
            const int m = 2 * P;
            if (m <= n) {  // l_m, l_{m+1} and C_m, C_{m+1} as 8-byte loads (m even); sc[n] = C_n = 0
                const float2 l2 = *reinterpret_cast<const float2 *>(sl + m);
                const float2 c2 = *reinterpret_cast<const float2 *>(sc + m);
                const float cm = m > 0 ? sc[m - 1] : 0.0f;
                v.x = l2.x * cs;
                v.z = c2.x - cm;
                if (m + 1 <= n) {
                    v.y = l2.y * cs;
                    v.w = c2.y - c2.x;
                }
            }
        }
        __syncwarp();
        if (P >= 0) Q[P] = v;
        __syncwarp();
    }
    if (lane < kPadPairs) Q[-1 - lane] = make_float4(-3.0e30f, -3.0e30f, 0.0f, 0.0f);
    __syncwarp();
}

// Boundary terms of the pairs (m, m + 1), m even, for the first-hit centre mu: below it (NEG)
// -dC_m T(mu - l_m), above it +dC_m T(l_m - mu), two terms per packed operation.
#ifndef FSMI_PAIR_UNROLL
#define FSMI_PAIR_UNROLL 4
#endif
#ifndef FSMI_PAIR2_UNROLL
#define FSMI_PAIR2_UNROLL 2
#endif
constexpr int kPairUnroll = FSMI_PAIR_UNROLL;    // boundary pairs in flight per lane, one slot per lane
constexpr int kPair2Unroll = FSMI_PAIR2_UNROLL;  // the same, two slots per lane (twice the work per pair)

template <bool NEG>
__device__ __forceinline__ f32x2 pair_term(const float4 &q, f32x2 mu2, f32x2 acc)
{
    const f32x2 L = pack2(q.x, q.y), dc = pack2(q.z, q.w);
    return fma2(dc, gauss_tail2p<NEG>(NEG ? sub2(mu2, L) : sub2(L, mu2)), acc);
}

// the pair (m, m + 1) that straddles the centre: m below it, m + 1 above
__device__ __forceinline__ f32x2 straddle_term(const float4 &q, float mu, f32x2 acc)
{
    return fma2(pack2(-q.z, q.w), gauss_tail2p<false>(pack2(mu - q.x, q.y - mu)), acc);
}

// Exact pair sum (Theorem 1) of one beam over the boundary pairs Q: for every first-hit slot j at
// least the boundaries with |l_m - mu_j| < cut (scaled) are visited, in increasing m, even and odd
// m in the two halves of a packed accumulator. With cut = kTailCut every non-zero term of the full
// sweep is added, in the same order, so the FP32 result equals the full sweep (cut = +inf) bit for
// bit; with kTailCutDefault the terms skipped are below 2^-27 of their weights.
//
// Slots go in rounds of 64 while more than 32 remain: lane i takes the adjacent slots A = jb + 2i
// and B = A + 1 and evaluates both against each pair it loads. Pairs below A (m < A) lie below both
// centres, the pair at m = A straddles A's centre and lies below B's, pairs from A + 2 on lie above
// both. The last <= 32 slots (and the no-return slot n when e0 is set: centre mu0 before l_0, every
// boundary above it) go one per lane. In every round all lanes run the same number of pairs below
// and above (the fewest that cover every window of the round), so that no lane leaves the unrolled
// loops early; a lane whose window is shorter adds boundaries beyond it, which are terms of the
// full sum as well (or padding). The counts come from coverage trials that start from the previous
// round's: below, a count G covers a slot when the boundary just before the loop's first pair lies
// below mu - cut; above, when the boundary just after its last pair lies at or beyond mu + cut.
__device__ __forceinline__ float exact_pairs_sum(const float4 *Q, const float *sc, const float *sp, int n, bool e0,
                                                 float pe0, float mu0, float cut)
{
    const int lane = lane_id();
    const float *Qf = reinterpret_cast<const float *>(Q);
    auto lq = [&](int m) { return Qf[4 * (m >> 1) + (m & 1)]; };  // l_m (m >> 1 floors negative m)
    const int nslots = n + (e0 ? 1 : 0);
    const int mtop = ((n >> 1) + 1 + kPadPairs) * 2;  // pairs (m, m + 1) stay below this m
    // first trial: about cut x (boundaries per unit of scaled distance) boundaries on each side
    const float span = lq(n) - lq(0);
    const float per = span > 0.0f ? __fdividef((float)n, span) : 0.0f;
    int GN = (int)fminf(cut * per, (float)(n + 1)) >> 1, GP = GN;
    float r = 0.0f;
    int jb = 0;
    // ---- two adjacent slots per lane ----
    for (; n - jb > 32; jb += 64) {
        const int j = jb + 2 * lane;
        const bool actA = j < n, actB = j + 1 < n;
        const int a = actA ? j : jb;  // an idle lane shadows slot jb with zero weight
        const float4 q0 = Q[a >> 1];  // l_a, l_{a+1}, dC_a, dC_{a+1}
        const float muA = 0.5f * (q0.x + q0.y), muB = 0.5f * (q0.y + Qf[4 * ((a >> 1) + 1)]);
        const float2 Cs = *reinterpret_cast<const float2 *>(sc + a);
        const float2 Ps = *reinterpret_cast<const float2 *>(sp + a);
        const float below = muA - cut, above = (actB ? muB : muA) + cut;
        auto neg_ok = [&](int G) {
            const int m = a - 2 * G;
            return !actA || m <= 0 || lq(m - 1) < below;
        };
        auto pos_ok = [&](int G) {
            const int e = a + 2 + 2 * G;
            return !actA || e > n || lq(e) >= above;
        };
        if (__all_sync(kFull, neg_ok(GN))) {
            while (GN > 0 && __all_sync(kFull, neg_ok(GN - 1))) --GN;
        } else {
            do ++GN;
            while (!__all_sync(kFull, neg_ok(GN)));
        }
        if (__all_sync(kFull, pos_ok(GP))) {
            while (GP > 0 && __all_sync(kFull, pos_ok(GP - 1))) --GP;
        } else {
            do ++GP;
            while (!__all_sync(kFull, pos_ok(GP)));
        }
        const f32x2 muA2 = pack2(muA, muA), muB2 = pack2(muB, muB);
        f32x2 accA = pack2(0.0f, 0.0f), accB = pack2(0.0f, 0.0f);
        int m = max(a - 2 * GN, -kPad2D);
#pragma unroll kPair2Unroll
        for (; m < a; m += 2) {
            const float4 q = Q[m >> 1];
            accA = pair_term<true>(q, muA2, accA);
            accB = pair_term<true>(q, muB2, accB);
        }
        accA = straddle_term(q0, muA, accA);
        accB = pair_term<true>(q0, muB2, accB);
        const int end = min(a + 2 + 2 * GP, mtop);
#pragma unroll kPair2Unroll
        for (m = a + 2; m < end; m += 2) {
            const float4 q = Q[m >> 1];
            accA = pair_term<false>(q, muA2, accA);
            accB = pair_term<false>(q, muB2, accB);
        }
        float a0, a1, b0, b1;
        unpack2(accA, a0, a1);
        unpack2(accB, b0, b1);
        r = fmaf(actA ? Ps.x : 0.0f, Cs.x + (a0 + a1), r);
        r = fmaf(actB ? Ps.y : 0.0f, Cs.y + (b0 + b1), r);
    }
    // ---- one slot per lane ----
    for (; jb < nslots; jb += 32) {
        const int j = jb + lane;
        const bool act = j < nslots;
        float mu = 0.0f, Cj = 0.0f, Pj = 0.0f;
        int mid = 0;
        if (act && j < n) {
            mu = 0.5f * (lq(j) + lq(j + 1));
            Cj = sc[j];
            Pj = sp[j];
            mid = j + 1;
        } else if (act) {  // the no-return slot: centre before l_0, every boundary above it
            mu = mu0;
            Pj = pe0;
        }
        const int nb = mid & ~1;  // pairs (m, m + 1) with m + 1 < mid end here
        const float below = mu - cut, above = mu + cut;
        auto neg_ok = [&](int G) {
            const int m = nb - 2 * G;
            return !act || m <= 0 || lq(m - 1) < below;
        };
        auto pos_ok = [&](int G) {
            const int e = nb + 2 + 2 * G;
            return !act || e > n || lq(e) >= above;
        };
        if (__all_sync(kFull, neg_ok(GN))) {
            while (GN > 0 && __all_sync(kFull, neg_ok(GN - 1))) --GN;
        } else {
            do ++GN;
            while (!__all_sync(kFull, neg_ok(GN)));
        }
        if (__all_sync(kFull, pos_ok(GP))) {
            while (GP > 0 && __all_sync(kFull, pos_ok(GP - 1))) --GP;
        } else {
            do ++GP;
            while (!__all_sync(kFull, pos_ok(GP)));
        }
        const f32x2 mu2 = pack2(mu, mu);
        f32x2 acc = pack2(0.0f, 0.0f);
        int m = act ? max(nb - 2 * GN, -kPad2D) : 0;
        const int nbe = act ? nb : 0;
#pragma unroll kPairUnroll
        for (; m < nbe; m += 2) acc = pair_term<true>(Q[m >> 1], mu2, acc);
        const int end = act ? min(nb + 2 + 2 * GP, mtop) : 0;
        if (m < end) {  // the pair at nb: it straddles the centre when mid is odd, else lies above it
            const float4 q = Q[m >> 1];
            acc = (m == mid - 1) ? straddle_term(q, mu, acc) : pair_term<false>(q, mu2, acc);
            m += 2;
        }
#pragma unroll kPairUnroll
        for (; m < end; m += 2) acc = pair_term<false>(Q[m >> 1], mu2, acc);
        float a0, a1;
        unpack2(acc, a0, a1);
        r = fmaf(Pj, Cj + (a0 + a1), r);
    }
    return r;
}

// ---- the Approx-FSMI pair sum over mirrored boundary pairs -------------------------------------
//
// Interleaved boundaries for Approx-FSMI: LW[m] = (l_m, dC_m) (scaled distance, C_m - C_{m-1})
// for m in [-kPad2D, n + kPad2D], padding (l = -+3e30, dC = 0) beyond the beam. Built in place over
// sl and the scratch array after it from the top down, as build_pairs does (writing LW[m]
// overwrites l_{2m}, l_{2m+1}, which only LW[2m], LW[2m+1] read).
__device__ __forceinline__ void build_lw(float *sl, const float *sc, int n, float cs)
{
    const int lane = lane_id();
    float2 *LW = reinterpret_cast<float2 *>(sl);
    const int mend = n + 1 + kPad2D;  // boundaries 0 .. mend - 1 (those above n padding)
    for (int top = mend; top > 0; top -= 32) {
        const int m = top - 32 + lane;
        float2 v = make_float2(3.0e30f, 0.0f);
        if (m >= 0 && m <= n) v = make_float2(sl[m] * cs, sc[m] - (m > 0 ? sc[m - 1] : 0.0f));  // sc[n] = 0
        __syncwarp();
        if (m >= 0) LW[m] = v;
        __syncwarp();
    }
    LW[-1 - lane] = make_float2(-3.0e30f, 0.0f);  // kPad2D = 32 padding boundaries below 0
    __syncwarp();
}

// Approx-FSMI (eq. fsmi_approx): for first-hit slot j the band k in [klo, khi] = [j - Delta,
// j + Delta] n [0, n - 1], i.e. boundaries m in [klo, khi + 1] with C' = C on the band and 0 outside
// it. In boundary form the interior boundaries weigh dC_m, the band edges C_klo (at m = klo) and
// -C_khi (at m = khi + 1). The boundaries below the centre, j - i, and above it, j + 1 + i, are
// taken as mirrored pairs (j - i, j + 1 + i), i = 0 .. Delta, so that every pair has the signs
// (-, +), which the tail's coefficients carry, and every lane runs exactly Delta + 1 pairs: an edge
// clamped at the beam's end lands on a padding boundary (its term is 0, and dC_0 = C_0, dC_n =
// -C_{n-1} are already the clamped edges' weights), and an unclamped edge is the last pair, whose
// weights are C_{j-Delta} and -C_{j+Delta}. The no-return slot (e0) is j = -1 with centre mu0: the
// paper's band k in [1, Delta], every boundary above it. Delta beyond n changes nothing (every band
// is the whole beam), so it is capped at n; past the padding (Delta > kPad2D - 1) the indices are
// clamped to it.
template <bool CLAMP>
__device__ __forceinline__ float approx_pairs_sum(const float2 *LW, const float *sc, const float *sp, int n, bool e0,
                                                  float pe0, float mu0, int D)
{
    const int lane = lane_id();
    float r = 0.0f;
    for (int jb = e0 ? -1 : 0; jb < n; jb += 32) {
        const int j = jb + lane;
        const bool act = j < n;
        const int jj = act ? j : n - 1;  // an idle lane shadows the last slot with zero weight
        float mu, Cj, Pj;
        if (jj >= 0) {
            mu = 0.5f * (LW[jj].x + LW[jj + 1].x);
            Cj = sc[jj];
            Pj = act ? sp[jj] : 0.0f;
        } else {
            mu = mu0;
            Cj = 0.0f;
            Pj = pe0;
        }
        f32x2 acc = pack2(0.0f, 0.0f);
        int i = 0;
#pragma unroll 2
        for (; i < D; ++i) {
            const int mb = jj - i, ma = jj + 1 + i;
            const float2 b = LW[CLAMP ? max(mb, -kPad2D) : mb], a = LW[CLAMP ? min(ma, n + kPad2D) : ma];
            acc = fma2(pack2(b.y, a.y), gauss_tail2p<true, false>(pack2(mu - b.x, a.x - mu)), acc);
        }
        {  // i = D: the band edges
            const int mb = jj - D, ma = jj + 1 + D;
            const float2 b = LW[CLAMP ? max(mb, -kPad2D) : mb], a = LW[CLAMP ? min(ma, n + kPad2D) : ma];
            const float wb = mb >= 0 ? sc[mb] : 0.0f, wa = (ma >= 1 && ma <= n) ? -sc[ma - 1] : 0.0f;
            acc = fma2(pack2(wb, wa), gauss_tail2p<true, false>(pack2(mu - b.x, a.x - mu)), acc);
        }
        float a0, a1;
        unpack2(acc, a0, a1);
        r = fmaf(Pj, Cj + (a0 + a1), r);
    }
    return r;
}

// ---- the exact pair sum in mass form ---------------------------------------------------------
//
// I = sum_k C_k sum_j P(e_j) G_{k,j}, the lanes holding source cells k (their mass polynomials in
// registers, cell_mass.cuh) and running over the targets j, which shared memory gives in pairs:
// Tg[p] = (x_2p, x_2p+1, P_2p, P_2p+1) with x the scaled cell centres, one 16-byte load per pair of
// targets and two sources. Every term is a product of non-negative factors (C_k of known cells may
// round below zero), so nothing cancels. Target -1 is the no-return event (P = 0 unless e0 is set);
// a slot past the last cell has P = 0.
//
// A pair of terms costs 7 packed FP32 operations and two ex2 (14 FMA-pipe cycles and 8 SFU cycles per
// warp at D = 3) where the boundary form costs 10 and two ex2 and two rcp (20 and 24).
//
// Windows: a cell whose centre lies beyond a cut plus half its width holds, together with all the cells behind
// it, less Gaussian mass than the tail at the cut. Its weight is C_k itself, a running sum that grows along the
// beam, not the difference of two neighbours as in the boundary form, and what is left out has one sign;
// so the cells after the first hit, whose C_k is the larger, need a wider cut than the boundary form's:
// T(kMassCut) = 4.6e-10 < 2^-31; for those before it (C_k about C_j at most) T(kTailCutDefault) = 7.4e-9 < 2^-27
// does. Largest relative change of a beam's MI, sigma 2 / 5 / 20, on the office map and on random cells: 1.2e-7 /
// 2.1e-7 / 5.2e-7 with both cuts at 4.58, 1.5e-9 / 3.7e-9 / 7.6e-9 here for 6 % more terms and 5 % more time on the
// 2048x2048 office batch (both cuts at 5.2: the same, 11 % more terms; 5.0: 3.7e-9 / 1.1e-8 / 2.8e-8, 9 %). (FSMI_FLAG_FULL_WINDOW: kTailCut, beyond which
// 2^(-d^2) is exactly 0; FSMI_FLAG_FULL_SWEEP: no cut. Both add the same non-zero terms in the same order.)
constexpr float kMassCut = 5.2f, kMassCutStep = kMassCut - kTailCutDefault;

// Builds Tg in place over sl and the scratch array after it, from the top pair down (writing Tg[p]
// overwrites l_4p .. l_4p+3, which only Tg[2p - 1], Tg[2p] and Tg[2p + 1] read: they lie higher, or
// at p <= 1 in the same step of 32 pairs, whose reads all come before its writes), and replaces P
// in sp by the cells' scaled widths.
__device__ __forceinline__ void build_targets(float *sl, float *sp, int n, float cs, float pe0, float mu0)
{
    const int lane = lane_id();
    float4 *Tg = reinterpret_cast<float4 *>(sl);
    const int pend = (n >> 1) + 1;  // pairs 0 .. n / 2
    for (int top = (pend + 31) & ~31; top > 0; top -= 32) {
        const int p = top - 32 + lane;
        float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        float2 w = make_float2(0.0f, 0.0f);
        const int m = 2 * p;
        if (m < n) {  // l_m, l_{m+1}, l_{m+2}: m + 2 <= n + 1, inside the array
            const float2 l2 = *reinterpret_cast<const float2 *>(sl + m);
            const float2 p2 = *reinterpret_cast<const float2 *>(sp + m);
            const float l0 = l2.x * cs, l1 = l2.y * cs;
            v.x = 0.5f * (l0 + l1);
            v.z = p2.x;
            w.x = l1 - l0;
            if (m + 1 < n) {
                const float l3 = sl[m + 2] * cs;
                v.y = 0.5f * (l1 + l3);
                v.w = p2.y;
                w.y = l3 - l1;
            }
        }
        __syncwarp();
        if (p < pend) {
            Tg[p] = v;
            if (m < n) *reinterpret_cast<float2 *>(sp + m) = w;
        }
        __syncwarp();
    }
    if (lane == 0) Tg[-1] = make_float4(mu0, mu0, 0.0f, pe0);
    __syncwarp();
}

// Exact sum. Sources in rounds of 64 while more than 32 remain, lane i the adjacent cells A = 2i and
// B = A + 1 of the round, then one per lane. In every round all lanes run over the same number of
// pairs below and above their own (the fewest that cover every window of the round, by coverage
// trials from the previous round's counts), clamped to the beam. `cut` bounds the targets below a
// source, cut - kMassCutStep those above it.
template <int D>
__device__ __forceinline__ float exact_mass_sum(const float4 *Tg, const float *sc, const float *sw, int n, bool e0, float cut)
{
    const int lane = lane_id();
    const float *Tf = reinterpret_cast<const float *>(Tg);
    auto xq = [&](int m) { return Tf[4 * (m >> 1) + (m & 1)]; };  // x_m (m >> 1 floors m = -1)
    const int mlo = e0 ? -1 : 0, plast = (n - 1) >> 1;
    const float span = xq(n - 1) - xq(0);
    const float per = span > 0.0f ? __fdividef((float)n, span) : 0.0f;
    int GN = (int)fminf(cut * per, (float)(n + 1)) >> 1, GP = GN;  // first trial
    float r = 0.0f;
    int kb = 0;
    for (; kb < n; kb += 64) {
        const bool two = n - kb > 32;  // one source per lane in the last round of at most 32
        const int k = kb + (two ? 2 * lane : lane);
        const bool act = k < n, actB = two && k + 1 < n;
        const int a = act ? k : kb;  // an idle lane shadows the round's first source with weight 0
        const int b = actB ? a + 1 : a;
        const int pa = a >> 1;
        const float xa = xq(a), xb = xq(b);
        const float below = xa - cut, above = xb + (cut - kMassCutStep);
        auto neg_ok = [&](int G) {
            const int m = 2 * (pa - G) - 1;
            return !act || m < mlo || xq(m) < below;
        };
        auto pos_ok = [&](int G) {
            const int m = 2 * (pa + G) + 2;
            return !act || m >= n || xq(m) >= above;
        };
        if (__all_sync(kFull, neg_ok(GN))) {
            while (GN > 0 && __all_sync(kFull, neg_ok(GN - 1))) --GN;
        } else {
            do ++GN;
            while (!__all_sync(kFull, neg_ok(GN)));
        }
        if (__all_sync(kFull, pos_ok(GP))) {
            while (GP > 0 && __all_sync(kFull, pos_ok(GP - 1))) --GP;
        } else {
            do ++GP;
            while (!__all_sync(kFull, pos_ok(GP)));
        }
        int p = max(pa - GN, -1);
        const int end = min(pa + GP, plast);
        const MassSource<D> A = mass_source<D>(xa, sw[a]);
        f32x2 accA = pack2(0.0f, 0.0f);
        float a0, a1;
        if (two) {
            const MassSource<D> B = mass_source<D>(xb, sw[b]);
            f32x2 accB = pack2(0.0f, 0.0f);
#pragma unroll kPair2Unroll
            for (; p <= end; ++p) {
                const float4 q = Tg[p];
                const f32x2 X = pack2(q.x, q.y), P = pack2(q.z, q.w);
                accA = mass_term<D>(A, X, P, accA);
                accB = mass_term<D>(B, X, P, accB);
            }
            float b0, b1;
            unpack2(accB, b0, b1);
            r = fmaf(actB ? sc[b] : 0.0f, b0 + b1, r);
        } else {
#pragma unroll kPairUnroll
            for (; p <= end; ++p) {
                const float4 q = Tg[p];
                accA = mass_term<D>(A, pack2(q.x, q.y), pack2(q.z, q.w), accA);
            }
        }
        unpack2(accA, a0, a1);
        r = fmaf(act ? sc[a] : 0.0f, a0 + a1, r);
        if (!two) break;
    }
    return r;
}

// Widest cell (scaled) that the mass form's table of degree D covers: sqrt 2 cells at the smallest sigma of the
// degree, and 1 / 1000 more for rounded direction vectors.
template <int D>
constexpr float kMassWidth = (float)(1.001 * kSqrtLog2e / (D == 3 ? kMassSigma3 : kMassSigma4));

// The boundary form for a beam of a mass kernel whose cells are wider than that, all n (n + 1) terms: no beam
// along a unit vector gets here, so it is kept small (a call of exact_pairs_sum costs the mass kernels' other
// beams 44 bytes of spilled registers each).
__device__ __forceinline__ float wide_beam_sum(const float *sl, const float *sc, const float *sp, int n, bool e0, float pe0,
                                               float cs)
{
    float r = 0.0f;
#pragma unroll 1
    for (int j = lane_id() - (e0 ? 1 : 0); j < n; j += 32) {
        const float mu = j < 0 ? sl[0] * cs - 0.5f * cs : 0.5f * (sl[j] * cs + sl[j + 1] * cs);
        float acc = j < 0 ? 0.0f : sc[j], c = 0.0f;
#pragma unroll 1
        for (int m = 0; m <= n; ++m) {  // sc[n] = 0
            const float dc = sc[m] - c, t = gauss_tail(sl[m] * cs - mu);
            c = sc[m];
            acc = fmaf(m <= j ? -dc : dc, t, acc);
        }
        r = fmaf(j < 0 ? pe0 : sp[j], acc, r);
    }
    return r;
}

// Uniform-FSMI (Algorithm 4) from D = inclusive prefix of C (sd), with Algorithm 4's clamps.
__device__ __forceinline__ float uniform_sum(const float *sd, const float *sp, int n, bool e0, float pe0, int H,
                                             float inv_2h1)
{
    float r = 0.0f;
    for (int j = lane_id(); j < n; j += 32) {
        const int hi = min(n - 1, j + H);
        const int lo = j - H - 1;
        const float S = (sd[hi] - (lo >= 0 ? sd[lo] : 0.0f)) * inv_2h1;
        r = fmaf(sp[j], S, r);
    }
    if (e0 && lane_id() == 0) {
        const int hi = min(n - 1, H - 1);
        if (hi >= 0) r = fmaf(pe0, sd[hi] * inv_2h1, r);
    }
    return r;
}

#ifndef FSMI_MIN_BLOCKS_2D
#define FSMI_MIN_BLOCKS_2D 4  // resident 8-warp blocks per SM requested from the register allocator (64 registers)
#endif

// the candidate set holding flat beam index `beam` (sets sorted by beam_offset)
__device__ __forceinline__ int set_of(const fsmi_set_2d *sets, int nsets, long long beam)
{
    int lo = 0, len = nsets;
    while (len > 0) {
        const int half = len >> 1;
        if (__ldg(&sets[lo + half].beam_offset) <= beam) {
            lo += half + 1;
            len -= half + 1;
        } else {
            len = half;
        }
    }
    return lo - 1;
}

// the trajectory holding pose p: t with traj_off[t] <= p < traj_off[t+1], or -1
__device__ __forceinline__ int traj_of(const int32_t *traj_off, int T, int p)
{
    int lo = 0, len = T + 1;  // last index with traj_off[idx] <= p
    while (len > 0) {
        const int half = len >> 1;
        if (__ldg(traj_off + lo + half) <= p) {
            lo += half + 1;
            len -= half + 1;
        } else {
            len = half;
        }
    }
    const int t = lo - 1;
    return (t >= 0 && t < T && p < __ldg(traj_off + t + 1)) ? t : -1;
}

// Cells of one beam on the map: traversal from `pose` along the sensor-frame direction (ux, uy)
// up to rfix (Q16) / rend, then per cell o (sp), f(delta_occ, o) (sc), f(delta_emp, o) (sx) and
// the entry distances (sl). With TRAJ, cells whose visit stamp is below `state` keep o but lose
// their gains (Section 2.4). Returns n, or -1 if the beam has more than cap cells; `wmax` is at least the width
// of its widest cell (the distance between two crossings along its major axis).
template <bool TRAJ>
__device__ __forceinline__ int beam_cells(const float *__restrict__ map, int W, int H, const float4 *__restrict__ gains,
                                          const int32_t *pose, int ux, int uy, long long rfix, float rend, int cap,
                                          const DevParams &p, int state, const int32_t *stamps, float *sl, float *sc,
                                          float *sp, float *sx, int *status, float &wmax)
{
    const int lane = lane_id();
    int dx, dy;
    beam_dir(pose, ux, uy, dx, dy);
    const unsigned ncell = (unsigned)W * (unsigned)H;
    Geo g;
    int K;
    wmax = 0.0f;
    if (!beam_geo(W, H, pose[0], pose[1], dx, dy, rfix, rend, g, K)) return 0;
    wmax = 65536.0f * g.rM;
    float lend = 0.0f;
    bool by_range, bad = false;
    int n = -1;
    Fixed f;
    const bool fixed = fixed_setup(g, f) && fixed_cells(f, K) <= cap;
    if (gains && fixed) {
        // traversal and gather in one pass, two chunks of intervals (up to four cells per lane) in
        // flight: the gathers go out before any of their results is stored
        const int stepm = g.xmaj ? g.sm * g.W : g.sm;
        n = fixed_run<2>(g, f, K,
                         [&](const Interval(&v)[2]) {
                             float4 a[2], b[2];
#pragma unroll
                             for (int u = 0; u < 2; ++u) {
                                 const unsigned i1 = v[u].ok1 ? (unsigned)v[u].id : ncell;
                                 const unsigned i2 = v[u].ok2 ? (unsigned)(v[u].id + stepm) : ncell;
                                 bad |= (v[u].ok1 && i1 >= ncell) || (v[u].ok2 && i2 >= ncell);
                                 a[u] = b[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                                 if (i1 < ncell) a[u] = __ldg(gains + i1);
                                 if (i2 < ncell) b[u] = __ldg(gains + i2);
                                 if (TRAJ && i1 < ncell && __ldg(stamps + i1) < state) a[u].y = a[u].z = 0.0f;
                                 if (TRAJ && i2 < ncell && __ldg(stamps + i2) < state) b[u].y = b[u].z = 0.0f;
                             }
#pragma unroll
                             for (int u = 0; u < 2; ++u) {
                                 if (v[u].ok1) {
                                     const int i = v[u].pos;
                                     sl[i] = v[u].lam1;
                                     sp[i] = a[u].x;
                                     sc[i] = a[u].y;
                                     sx[i] = a[u].z;
                                 }
                                 if (v[u].ok2) {
                                     const int i = v[u].pos + 1;
                                     sl[i] = v[u].lam2;
                                     sp[i] = b[u].x;
                                     sc[i] = b[u].y;
                                     sx[i] = b[u].z;
                                 }
                             }
                         },
                         lend, by_range);
        __syncwarp();
    }
    if (n < 0) {  // ids first, then per cell
        bad = false;
        int *ids = (int *)sx;
        if (fixed && !gains) {
            const int stepm = g.xmaj ? g.sm * g.W : g.sm;
            n = fixed_run<1>(g, f, K,
                             [&](const Interval(&v)[1]) {
                                 if (v[0].ok1) {
                                     ids[v[0].pos] = v[0].id;
                                     sl[v[0].pos] = v[0].lam1;
                                 }
                                 if (v[0].ok2) {
                                     ids[v[0].pos + 1] = v[0].id + stepm;
                                     sl[v[0].pos + 1] = v[0].lam2;
                                 }
                             },
                             lend, by_range);
            __syncwarp();
        }
        if (n < 0) n = dda_walk(g, K, cap, ids, sl, lend, by_range);
        if (n < 0) return -1;
        for (int i = lane; i < n; i += 32) {
            const unsigned id = (unsigned)ids[i];
            bad |= id >= ncell;  // cannot happen for a consistent traversal; never read out of bounds
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (id < ncell) {
                if (gains) {
                    v = __ldg(gains + id);
                } else {
                    const float o = __ldg(map + id);
                    v = make_float4(o, cell_gain(p.docc, o), cell_gain(p.demp, o), 0.0f);
                }
                // a cell already counted by an earlier state of the trajectory (Section 2.4) still
                // stops the beam with probability o but adds no information
                if (TRAJ && __ldg(stamps + id) < state) v.y = v.z = 0.0f;
            }
            sp[i] = v.x;
            sc[i] = v.y;
            sx[i] = v.z;
        }
    }
    if (__any_sync(kFull, bad) && lane == 0) set_status(status, FSMI_STATUS_INTERNAL);
    if (lane == 0) sl[n] = lend;
    __syncwarp();
    return n;
}

// The variant's mutual information of one beam of n cells held in shared memory (sl: n + 1
// distances, sp: o, sc: f_occ, sx: f_emp; no cell wider than wmax, which only the mass form asks for):
// Algorithm 2, Algorithm 3 (4), then the pair sum.
template <int VAR>
__device__ __forceinline__ float beam_sum(const DevParams &p, int n, float wmax, float *sl, float *sc, float *sp, float *sx)
{
    const int lane = lane_id();
    const bool e0 = p.e0 != 0;
    const float cs = p.inv_s2 * (float)kSqrtLog2e;  // distance -> tail variable
    float I = 0.0f;
    if (n > 0) {
        const float pe0 = cell_prefixes(sp, sc, sx, n, VAR == FSMI_UNIFORM);
        if (VAR == FSMI_EXACT || VAR == kExactFullSweep) {
            const float mu0 = sl[0] * cs - 0.5f * cs;  // e_0 centre, l_1 - 1/2 (scaled)
            build_pairs(sl, sc, n, cs);
            float cut = VAR == kExactFullSweep ? __int_as_float(0x7f800000) : kTailCutDefault;
            if (VAR == FSMI_EXACT && (p.flags & FSMI_FLAG_FULL_WINDOW)) cut = kTailCut;
            I = exact_pairs_sum(reinterpret_cast<const float4 *>(sl), sc, sp, n, e0, pe0, mu0, cut);
        }
        if (VAR == FSMI_APPROX) {
            const float mu0 = sl[0] * cs - 0.5f * cs;  // e_0 centre, l_1 - 1/2 (scaled)
            build_lw(sl, sc, n, cs);
            const int D = min(p.trunc, n);
            const float2 *LW = reinterpret_cast<const float2 *>(sl);
            I = D < kPad2D ? approx_pairs_sum<false>(LW, sc, sp, n, e0, pe0, mu0, D)
                           : approx_pairs_sum<true>(LW, sc, sp, n, e0, pe0, mu0, D);
        }
        if (mass_variant(VAR)) {
            constexpr int D = VAR == kExactMass3 ? 3 : 4;
            if (wmax * cs > kMassWidth<D>) {
                I = wide_beam_sum(sl, sc, sp, n, e0, pe0, cs);
            } else {
                const float mu0 = sl[0] * cs - 0.5f * cs;  // e_0 centre, l_1 - 1/2 (scaled)
                build_targets(sl, sp, n, cs, e0 ? pe0 : 0.0f, mu0);
                float cut = fmaf(0.5f * wmax, cs, kMassCut);
                if (p.flags & FSMI_FLAG_FULL_WINDOW) cut = kTailCut + kMassCutStep;
                if (p.flags & FSMI_FLAG_FULL_SWEEP) cut = __int_as_float(0x7f800000);
                I = exact_mass_sum<D>(reinterpret_cast<const float4 *>(sl), sc, sp, n, e0, cut);
            }
        }
        if (VAR == FSMI_UNIFORM) I = uniform_sum(sx, sp, n, e0, pe0, p.H, p.inv_2h1);
        I = warp_sum(I);
    }
    return I;
}

__device__ __forceinline__ void store_nan(float *out, long long i, int *status, int bits)
{
    if (lane_id() == 0) {
        out[i] = __int_as_float(0x7fc00000);
        set_status(status, bits);
    }
    __syncwarp();
}

// One beam: traversal (or explicit cells), gains, prefixes, the variant's pair sum, store.
template <int VAR, int SRC>
__device__ __forceinline__ void eval_beam(const Src2D &src, const DevParams &p, long long beam, float *sl, float *sc,
                                          float *sp, float *sx, float *__restrict__ out, int *status)
{
    const int lane = lane_id();
    int n;
    float wmax = 0.0f;
    if (SRC != kSrcBeams) {
        const int32_t *pose;
        int ux, uy;
        int state = 0;                   // kSrcTraj: state index within the trajectory
        const int32_t *stamps = nullptr;  // kSrcTraj: the trajectory's visit stamps
        long long rfix = p.rfix;
        float rend = p.rend;
        if (SRC == kSrcMap || SRC == kSrcTraj) {
            int pi, bi;
            if (beam <= 0x7fffffffLL) {  // 32-bit division (the common case; the 64-bit one is far longer)
                pi = (int)((unsigned)beam / (unsigned)src.B);
                bi = (int)((unsigned)beam - (unsigned)pi * (unsigned)src.B);
            } else {
                pi = (int)(beam / src.B);
                bi = (int)(beam % src.B);
            }
            pose = src.poses + 4 * (size_t)pi;
            ux = src.dirs[2 * bi];
            uy = src.dirs[2 * bi + 1];
            if (SRC == kSrcTraj) {
                const int t = traj_of(src.traj_off, src.T, pi);
                if (t < 0) return store_nan(out, beam, status, FSMI_STATUS_BAD_BEAM);  // pose outside every trajectory
                state = pi - __ldg(src.traj_off + t);
                stamps = src.stamp + (size_t)t * src.W * src.H;
            }
        } else {
            const int si = set_of(src.sets, src.nsets, beam);
            bool ok = si >= 0;
            fsmi_set_2d st{};
            if (ok) st = src.sets[si];
            const long long k = beam - st.beam_offset;
            const long long nb = (long long)st.npose * st.nbeam;
            ok = ok && st.npose >= 0 && st.nbeam > 0 && k >= 0 && k < nb;
            long long pi = 0, bi = 0;
            if (ok) {
                pi = st.pose_offset + k / st.nbeam;
                bi = st.dir_offset + k % st.nbeam;
                ok = st.pose_offset >= 0 && st.dir_offset >= 0 && pi < src.P && bi < src.B;
            }
            if (ok) {
                ok = st.max_range > 0.0f && st.max_range <= p.rmax;
                rfix = __double2ll_rn((double)st.max_range * 65536.0);
                rend = (float)((double)rfix * (1.0 / 65536.0));
            }
            if (!ok) return store_nan(out, beam, status, FSMI_STATUS_BAD_BEAM);  // never index with it
            pose = src.poses + 4 * (size_t)pi;
            ux = src.dirs[2 * bi];
            uy = src.dirs[2 * bi + 1];
        }
        n = beam_cells<SRC == kSrcTraj>(src.map, src.W, src.H, src.gains, pose, ux, uy, rfix, rend, p.nmax, p, state,
                                        stamps, sl, sc, sp, sx, status, wmax);
        if (n < 0) return store_nan(out, beam, status, FSMI_STATUS_BEAM_OVERFLOW);
    } else {
        const int base = src.off[beam];
        n = src.off[beam + 1] - base;
        if (n < 0 || n > p.nmax) return store_nan(out, beam, status, FSMI_STATUS_BAD_BEAM);
        for (int i = lane; i < n; i += 32) {
            const float o = __ldg(src.o + base + i);
            sl[i] = __ldg(src.l + base + i);
            sp[i] = o;
            sc[i] = cell_gain(p.docc, o);
            sx[i] = cell_gain(p.demp, o);
        }
        if (lane == 0) sl[n] = __ldg(src.lend + beam);
        __syncwarp();
    }
    const float I = beam_sum<VAR>(p, n, wmax, sl, sc, sp, sx);
    if (lane == 0) out[beam] = I;
    __syncwarp();
}

}  // namespace fsmi
