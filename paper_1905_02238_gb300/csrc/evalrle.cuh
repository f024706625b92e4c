// 3D hot path (Section 4): virtual-cell sampling of each ray, run-length encoding (eq.
// occup_rle), run prefixes P_E(u), D_E(v), and the run-pair sums of FSMI-RLE (Theorem 3),
// Approx-FSMI-RLE (Theorem 5) and Uniform-FSMI-RLE (Theorem 6). One warp per ray.
//
// Run-pair terms. With x = 1 - o_u and a shift-invariant noise kernel g between virtual cells,
//   A[x, Lu, Lv, t] = sum_{j<Lu} sum_{k<Lv} x^j g(j + t - k),  B = same with weight k.
// The k-sum is a window of g: W0(m) = sum_{k<Lv} g(m - k) = Psi(m) - Psi(m - Lv) and
// W1(m) = sum_{k<Lv} k g(m - k) = m W0(m) - (Psi1(m) - Psi1(m - Lv)), with the prefix tables
// Psi(m) = sum_{d<=m} g(d), Psi1(m) = sum_{d<=m} d g(d) held in shared memory. Then
// A = sum_j x^j W0(j + t), B = sum_j x^j W1(j + t), summed only where W0 can be non-zero
// (j + t in [-K, Lv - 1 + K], K the kernel's support radius). No power x^{-t} is ever formed,
// which avoids the instability the paper notes for its alpha/beta tables (Section 4.1).
//
// Short runs. The run-pair sum is Theorem 3's regrouping of the cell-level double sum
// sum_j sum_k P(e_j) C_k g(k - j) over the virtual cells (eq. eqn_from_fsmi). When a ray's runs
// are short (mean length below kCellRunLen) that cell-level form, a banded convolution of width
// 2K + 1, costs less than the run pairs, so the ray is decompressed in shared memory and
// evaluated that way -- the switch Section 5.4 recommends between the RLE algorithm and the
// algorithm on the decompressed sequence. Both forms give the same value (pinned in the tests).
#pragma once


#include "../../include/fsmi.h"
#include "fsmi_device.cuh"
#include "gauss_tail.cuh"
#include "fsmi_internal.h"

namespace fsmi {

// Gains f(delta_occ, o) and f(delta_emp, o) of one cell: the host-fitted polynomials of h(o) = f / (o (1 - o)),
// both together in packed FP32, Horner's rule (TERMS agrees with p.gain_fit).
template <int TERMS>
__device__ __forceinline__ void poly_gains(const DevParams &p, float o, float &fo, float &fe)
{
    const float x = __fmaf_rn(2.0f, o, -1.0f);
    const f32x2 X = pack2(x, x);
    f32x2 h = pack2(p.gfit2[TERMS - 1][0], p.gfit2[TERMS - 1][1]);
#pragma unroll
    for (int k = TERMS - 2; k >= 0; --k) h = fma2(h, X, pack2(p.gfit2[k][0], p.gfit2[k][1]));
    const float w = __fmul_rn(o, __fsub_rn(1.0f, o));
    unpack2(mul2(pack2(w, w), h), fo, fe);
}

// The polynomials where they are accurate for these deltas, else the closed forms.
__device__ __forceinline__ void rle_gains(const DevParams &p, float o, float &fo, float &fe)
{
    if (p.gain_fit == 2) {
        poly_gains<kGainShortTerms>(p, o, fo, fe);
    } else if (p.gain_fit) {
        poly_gains<kGainFitTerms>(p, o, fo, fe);
    } else {
        fo = cell_gain(p.docc, o);
        fe = cell_gain(p.demp, o);
    }
}

// C keeps its first cell at a 16-byte boundary, conv_pad(K) >= K floats after its array's start; four outputs
// read conv_quads(K) groups of four of it
__host__ __device__ constexpr int conv_pad(int K) { return (K + 3) & ~3; }
__host__ __device__ constexpr int conv_quads(int K) { return (conv_pad(K) + K + 7) / 4; }

// ---- noise-kernel prefix tables --------------------------------------------------------------

// tab[i] = (Psi(m), Psi1(m)) for m = i - K - 1, i in [0, 2K + 1]; Psi(-K-1) = 0, Psi(K) = total;
// gtab[K + d] = g(d). The host builds both once per launch (fill_rle_table: kind 0 Gaussian
// density (Theorem 3), 1 Gaussian cell mass, 2 box 1[|d| <= H] (Theorem 6); band >= 0 zeroes
// |d| > band, the strict-band reading of Approx-FSMI-RLE; normalisation folded into g; in double,
// stored as float); each block copies them from the launch's parameters into shared memory.
// gz (for band_conv_any) is g with zeros around it: gz[4 + (conv_pad(K) - K) + d] = g(d - K), d = 0 .. 2K.
static __device__ void load_table(float2 *tab, float *gtab, float *gz, int K, const RleTable &t)
{
    for (int i = threadIdx.x; i < 2 * K + 2; i += blockDim.x) tab[i] = t.tab[i];
    for (int i = threadIdx.x; i < 2 * K + 1; i += blockDim.x) gtab[i] = t.gtab[i];
    for (int i = threadIdx.x; i < 4 * (conv_quads(K) + 1); i += blockDim.x) {
        const int d = i - 4 - (conv_pad(K) - K);
        gz[i] = d >= 0 && d <= 2 * K ? t.gtab[d] : 0.0f;
    }
    __syncthreads();
}

__device__ __forceinline__ float2 tab_at(const float2 *tab, int K, int m)
{
    return tab[min(max(m, -K - 1), K) + K + 1];
}

// A and B of one run pair (see the file comment).
__device__ __forceinline__ void pair_AB(float x, int Lu, int Lv, int t, const float2 *tab, int K, float &A,
                                        float &B)
{
    A = 0.0f;
    B = 0.0f;
    const int jlo = max(0, -K - t);
    const int jhi = min(Lu - 1, Lv - 1 + K - t);
    if (jlo > jhi) return;
    float xp = ipowf(x, jlo);
    for (int j = jlo; j <= jhi; ++j) {
        const int m = j + t;
        const float2 a = tab_at(tab, K, m);
        const float2 b = tab_at(tab, K, m - Lv);
        const float w0 = a.x - b.x;
        const float w1 = fmaf((float)m, w0, -(a.y - b.y));
        A = fmaf(xp, w0, A);
        B = fmaf(xp, w1, B);
        xp *= x;
    }
}

// ---- per-ray run arrays in shared memory ----------------------------------------------------

struct RunSmem {
    float *O;  // o_u, then P_E(u) o_u
    float *X;  // 1 - o_u
    float *A;  // D_E(u) + f(delta_occ, r_u)
    float *F;  // f(delta_emp, r_u)
    int *S;    // s_u (first virtual cell of run u); S[nr] = n
    int *L;    // L_u
};

__device__ __forceinline__ RunSmem run_smem(float *base, int stride)
{
    RunSmem r;
    r.O = base;
    r.X = base + stride;
    r.A = base + 2 * stride;
    r.F = base + 3 * stride;
    r.S = (int *)(base + 4 * stride);
    r.L = (int *)(base + 5 * stride);
    return r;
}

// Run starts s_u = sum_{i<u} L_i (and S[nr] = n) from the lengths, or lengths from the starts.
static __device__ void run_starts(const RunSmem &r, int nr, bool have_s)
{
    const int lane = lane_id();
    const int K = (nr + 31) >> 5;
    const int lo = min(nr, lane * K), hi = min(nr, lo + K);
    if (!have_s) {
        int cs = 0;
        for (int u = lo; u < hi; ++u) cs += r.L[u];
        const int ic = warp_incl_add_int(cs);
        int s = __shfl_up_sync(kFull, ic, 1);
        if (lane == 0) s = 0;
        for (int u = lo; u < hi; ++u) {
            r.S[u] = s;
            s += r.L[u];
        }
        if (lane == 31) r.S[nr] = ic;
    } else {
        for (int u = lo; u < hi; ++u) r.L[u] = r.S[u + 1] - r.S[u];
    }
    __syncwarp();
}

// Run prefixes (Algorithms for P_E(u) and D_E(v)): P_E(u) = prod_{i<u} (1 - o_i)^{L_i},
// D_E(u) = sum_{i<u} L_i f(delta_emp, r_i). On entry O, L and S are set. (A run's gains are formed once and wait in A
// and F for the second pass.)
static __device__ void run_prefixes(const RunSmem &r, int nr, const DevParams &p)
{
    const int lane = lane_id();
    const int K = (nr + 31) >> 5;
    const int lo = min(nr, lane * K), hi = min(nr, lo + K);
    float prod = 1.0f, sum = 0.0f;
    for (int u = lo; u < hi; ++u) {
        const float o = r.O[u];
        const int L = r.L[u];
        float fo, fe;
        rle_gains(p, o, fo, fe);
        r.A[u] = fo;
        r.F[u] = fe;
        prod *= ipowf(1.0f - o, L);
        sum = fmaf((float)L, fe, sum);
    }
    const float ip = warp_incl_mul(prod);
    const float is = warp_incl_add(sum);
    float E = __shfl_up_sync(kFull, ip, 1);
    float D = __shfl_up_sync(kFull, is, 1);
    if (lane == 0) {
        E = 1.0f;
        D = 0.0f;
    }
    for (int u = lo; u < hi; ++u) {
        const float o = r.O[u];
        const int L = r.L[u];
        const float x = 1.0f - o, fe = r.F[u];
        r.X[u] = x;
        r.A[u] += D;
        r.O[u] = E * o;
        E *= ipowf(x, L);
        D = fmaf((float)L, fe, D);
    }
    __syncwarp();
}

// Eq. (group_fsmi_rle_exact) over every run pair whose A, B can be non-zero (FSMI-RLE,
// Uniform-FSMI-RLE, strict-band Approx-FSMI-RLE); returns this lane's partial sum.
static __device__ float pairs_all(const RunSmem &r, int nr, const float2 *tab, int K)
{
    float tot = 0.0f;
    for (int u = lane_id(); u < nr; u += 32) {
        const float Pu = r.O[u];
        if (Pu == 0.0f) continue;
        const float x = r.X[u];
        const int su = r.S[u], Lu = r.L[u];
        float acc = 0.0f;
        for (int v = 0; v < nr; ++v) {
            const int t = su - r.S[v];
            const int Lv = r.L[v];
            if (t + Lu - 1 < -K || t > Lv - 1 + K) continue;
            float A, B;
            pair_AB(x, Lu, Lv, t, tab, K, A, B);
            acc = fmaf(r.A[v], A, fmaf(r.F[v], B, acc));
        }
        tot = fmaf(Pu, acc, tot);
    }
    return tot;
}

// Theorem 5 as printed: the full diagonal block (theta, gamma) plus, for runs within Delta of
// each other, the sub-blocks s', L' of eqs. (su')-(Lv') with shift t = s_u' - s_v', weighted by
// (1 - o_u)^{s_u' - s_u} (u < v) or with D_E(v) + (s_v' - s_v) f(delta_emp, r_v) (u > v).
static __device__ float pairs_thm5(const RunSmem &r, int nr, const float2 *tab, int K, int D)
{
    float tot = 0.0f;
    for (int u = lane_id(); u < nr; u += 32) {
        const float Pu = r.O[u];
        if (Pu == 0.0f) continue;
        const float x = r.X[u];
        const int su = r.S[u], Lu = r.L[u];
        float A, B;
        pair_AB(x, Lu, Lu, 0, tab, K, A, B);
        float acc = fmaf(r.A[u], A, r.F[u] * B);
        for (int v = u + 1; v < nr; ++v) {
            const int sv = r.S[v];
            if (!(sv < su + Lu + D)) break;
            const int Lv = r.L[v];
            const int su2 = max(su, sv - D);
            const int Lu2 = su + Lu - su2;
            const int Lv2 = min(Lv, su + Lu + D - sv);
            pair_AB(x, Lu2, Lv2, su2 - sv, tab, K, A, B);
            acc = fmaf(ipowf(x, su2 - su), fmaf(r.A[v], A, r.F[v] * B), acc);
        }
        for (int v = u - 1; v >= 0; --v) {
            const int sv = r.S[v], Lv = r.L[v];
            if (!(su < sv + Lv + D)) break;
            const int Lu2 = min(Lu, sv + Lv + D - su);
            const int sv2 = max(sv, su - D);
            const int Lv2 = sv + Lv - sv2;
            pair_AB(x, Lu2, Lv2, su - sv2, tab, K, A, B);
            acc = fmaf(fmaf((float)(sv2 - sv), r.F[v], r.A[v]), A, fmaf(r.F[v], B, acc));
        }
        tot = fmaf(Pu, acc, tot);
    }
    return tot;
}

constexpr int kArraysRLE = 7;                  // per-warp shared arrays (each `stride` floats)

// ---- the cell form ---------------------------------------------------------------------------------
//
// A ray's cells go through in blocks of 128, four consecutive cells per lane: the gains, Algorithm 2's and 3's
// prefixes within the lane, one warp scan per block for the lanes' totals, and P(e_j) and C_k stored once, 16
// bytes per lane. The fused kernel runs it on the samples as they arrive (no o, f_occ or f_emp array is
// written and read back), the run-input kernel on the decompressed runs; the same operations in the
// same order, so the two give the same floats.

// 16 or 8 bytes of consecutive cells
__device__ __forceinline__ void store_cells(float *p, const float (&v)[4])
{
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void store_cells(float *p, const float (&v)[2])
{
    *reinterpret_cast<float2 *>(p) = make_float2(v[0], v[1]);
}
__device__ __forceinline__ void store_cells(int *p, const int (&v)[4])
{
    *reinterpret_cast<int4 *>(p) = make_int4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void store_cells(int *p, const int (&v)[2]) { *reinterpret_cast<int2 *>(p) = make_int2(v[0], v[1]); }

// prefixes carried from block to block
struct CellScan {
    float E, q;  // prod (1 - o) and sum f_emp of the cells before the block
};

// cells per lane: rays of at most 64 samples go in one block of 64, so that half the lanes' work is not idle
constexpr int kShortRay = 64;

// Closed-form gains of a block's cells, once per span of equal values: the spans' values are listed in the block's
// part of CP, one lane evaluates each, and the cells read their span's pair back (CP, CB: scan_block writes there
// next). Two logarithms and a division per gain cost too much to repeat per cell (256x256x64 voxels without noise,
// 16 x 64x64 rays of 200 samples, delta 40 and 0.02: 196 us per cell, 159 us so; with noise 103 and 80 us).
template <int CPL>
__device__ __forceinline__ void closed_gains(const DevParams &p, const float (&o)[CPL], int i0, int n, float *CP, float *CB,
                                             float (&fo)[CPL], float (&fe)[CPL])
{
    const int lane = lane_id(), b0 = i0 - CPL * lane;
    const unsigned left = __shfl_up_sync(kFull, __float_as_uint(o[CPL - 1]), 1);
    int id[CPL], cnt = 0;
#pragma unroll
    for (int t = 0; t < CPL; ++t) {
        const unsigned before = t ? __float_as_uint(o[t > 0 ? t - 1 : 0]) : left;
        id[t] = i0 + t < n && (__float_as_uint(o[t]) != before || (t == 0 && lane == 0));
        cnt += id[t];
    }
    const int incl = warp_incl_add_int(cnt), total = __shfl_sync(kFull, incl, 31);
    int k = incl - cnt - 1;
#pragma unroll
    for (int t = 0; t < CPL; ++t) {
        if (id[t]) CP[b0 + ++k] = o[t];
        id[t] = k;
    }
    __syncwarp();
    for (int j = b0 + lane; j < b0 + total; j += 32) {
        const float v = CP[j];
        CP[j] = cell_gain(p.docc, v);
        CB[j] = cell_gain(p.demp, v);
    }
    __syncwarp();
#pragma unroll
    for (int t = 0; t < CPL; ++t) {
        fo[t] = i0 + t < n ? CP[b0 + id[t]] : 0.0f;
        fe[t] = i0 + t < n ? CB[b0 + id[t]] : 0.0f;
    }
    __syncwarp();
}

// One block of 32 CPL cells (CPL = 4, or 2 on short rays): o of this lane's cells i0 .. i0 + CPL - 1 (zero from
// the ray's end on); stores P in CP and C in CB where i0 < n. POLY: only for deltas with polynomial gains.
template <int CPL, bool POLY>
__device__ __forceinline__ void scan_block(const DevParams &p, const float (&o)[CPL], int i0, int n, CellScan &s, float *CP,
                                           float *CB)
{
    float fo[CPL], fe[CPL];
    if (p.gain_fit == 2) {
#pragma unroll
        for (int t = 0; t < CPL; ++t) poly_gains<kGainShortTerms>(p, o[t], fo[t], fe[t]);
    } else if (POLY || p.gain_fit) {
#pragma unroll
        for (int t = 0; t < CPL; ++t) poly_gains<kGainFitTerms>(p, o[t], fo[t], fe[t]);
    } else {
        closed_gains<CPL>(p, o, i0, n, CP, CB, fo, fe);
    }
    float prod = (1.0f - o[0]) * (1.0f - o[1]), sum = fe[0] + fe[1];
    if (CPL == 4) {
        prod = (prod * (1.0f - o[CPL - 2])) * (1.0f - o[CPL - 1]);  // cell by cell, see cell_prefixes
        sum += fe[CPL - 2] + fe[CPL - 1];
    }
    prod = warp_incl_mul(prod);
    sum = warp_incl_add(sum);
    float E = __shfl_up_sync(kFull, prod, 1), q = __shfl_up_sync(kFull, sum, 1);
    const int lane = lane_id();
    E = lane == 0 ? s.E : s.E * E;
    q = lane == 0 ? s.q : s.q + q;
    s.E *= __shfl_sync(kFull, prod, 31);
    s.q += __shfl_sync(kFull, sum, 31);
    float P[CPL], C[CPL];
#pragma unroll
    for (int t = 0; t < CPL; ++t) {
        P[t] = E * o[t];  // Algorithm 2
        E *= 1.0f - o[t];
        C[t] = q + fo[t];  // Algorithm 3
        q += fe[t];
    }
    if (i0 < n) {
        store_cells(CP + i0, P);
        store_cells(CB + i0, C);
    }
}

// conv_pad(K) zeros before C_0 and K + 8 from C_n on (scan_block leaves up to three entries past C_{n-1}
// undefined)
__device__ __forceinline__ void pad_conv(float *CB, int K, int n)
{
    for (int i = lane_id(); i < K + 8; i += 32) {
        if (i < conv_pad(K)) CB[-1 - i] = 0.0f;
        CB[n + i] = 0.0f;
    }
    __syncwarp();
}

// sum_j P(e_j) sum_{|d| <= K} g(d) C_{j+d} (P in CP, C at CB, zero-padded on both sides). With a compile-time
// radius KK a lane takes V consecutive j: C comes in 16-byte loads, (V + 2 KK) / 4 of them for V outputs
// instead of one load per tap and output, and every loaded pair (C_k, C_{k+1}) meets all the output pairs it
// belongs to in packed FP32 operations: outputs (j, j + 1) for one parity of the tap, (j - 1, j) for the
// other, each in accumulators of its own. The kernel values are operands from the launch parameters. On the
// 512x512x128 batch one output per lane and one load per tap took 329 of 1,741 warp instructions per ray
// and a third of the shared-memory wavefronts.
template <int KK, int V>
__device__ __forceinline__ float band_conv_v(const float *CP, const float *CB, const RleTable &t, int n)
{
    constexpr int kPad = conv_pad(KK), kSh = kPad - KK;  // inputs from j0 - kPad: input k meets output j with tap k - j - kSh
    constexpr int kQuads = (kPad + KK + V + 3) / 4;
    static_assert(V % 4 == 0 && KK <= kConvMaxRadius, "outputs per lane");
    float v = 0.0f;
    for (int j0 = V * lane_id(); j0 < n; j0 += 32 * V) {
        f32x2 ev[V / 2], od[V / 2 + 1];
#pragma unroll
        for (int q = 0; q < V / 2; ++q) ev[q] = pack2(0.0f, 0.0f);
#pragma unroll
        for (int q = 0; q <= V / 2; ++q) od[q] = pack2(0.0f, 0.0f);
        const float4 *c4 = reinterpret_cast<const float4 *>(CB + j0 - kPad);
#pragma unroll
        for (int m = 0; m < kQuads; ++m) {
            const float4 c = c4[m];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const f32x2 x = h ? pack2(c.z, c.w) : pack2(c.x, c.y);
                const int k = 4 * m + 2 * h - kSh;
#pragma unroll
                for (int q = 0; q < V / 2; ++q) {
                    const int d = k - 2 * q;  // taps of outputs 2q, 2q + 1
                    if (d >= 0 && d <= 2 * KK) ev[q] = fma2(x, pack2(t.gdup[d].x, t.gdup[d].y), ev[q]);
                }
#pragma unroll
                for (int q = 0; q <= V / 2; ++q) {
                    const int d = k - 2 * q + 1;  // of outputs 2q - 1, 2q
                    if (d >= 0 && d <= 2 * KK) od[q] = fma2(x, pack2(t.gdup[d].x, t.gdup[d].y), od[q]);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < V / 2; q += 2) {
            const float4 P = *reinterpret_cast<const float4 *>(CP + j0 + 2 * q);
            float a0, a1, a2, a3, b0, b1, b2, b3, x;
            unpack2(ev[q], a0, a1);
            unpack2(ev[q + 1], a2, a3);
            unpack2(od[q], x, b0);
            unpack2(od[q + 1], b1, b2);
            unpack2(od[q + 2], b3, x);
            const int j = j0 + 2 * q;
            if (j < n) v = fmaf(P.x, a0 + b0, v);
            if (j + 1 < n) v = fmaf(P.y, a1 + b1, v);
            if (j + 2 < n) v = fmaf(P.z, a2 + b2, v);
            if (j + 3 < n) v = fmaf(P.w, a3 + b3, v);
        }
    }
    return v;
}

template <int KK>
__device__ __forceinline__ float band_conv_k(const float *CP, const float *CB, const RleTable &t, int n)
{
    // 8 outputs per lane need half the passes of 4 on a longer ray and waste half a pass on a shorter one
    return n > 128 ? band_conv_v<KK, 8>(CP, CB, t, n) : band_conv_v<KK, 4>(CP, CB, t, n);
}

// The same for any radius: four outputs per lane, and per group of four inputs one 16-byte load of C and one
// (the same for all lanes) of the zero-padded kernel, for 16 products, where one of each went with every
// product before.
__device__ __forceinline__ float band_conv_any(const float *CP, const float *CB, const float *gz, int K, int n)
{
    const int quads = conv_quads(K);
    float v = 0.0f;
    for (int j0 = 4 * lane_id(); j0 < n; j0 += 128) {
        const float4 *c4 = reinterpret_cast<const float4 *>(CB + j0 - conv_pad(K)), *g4 = reinterpret_cast<const float4 *>(gz);
        float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        float4 a = g4[0];
        for (int m = 0; m < quads; ++m) {
            const float4 c = c4[m], b = g4[m + 1];
            const float x[4] = {c.x, c.y, c.z, c.w}, g[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
            for (int h = 0; h < 4; ++h)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[q] = fmaf(x[h], g[4 + h - q], acc[q]);
            a = b;
        }
        const float4 P = *reinterpret_cast<const float4 *>(CP + j0);
        v = fmaf(P.x, acc[0], v);
        if (j0 + 1 < n) v = fmaf(P.y, acc[1], v);
        if (j0 + 2 < n) v = fmaf(P.z, acc[2], v);
        if (j0 + 3 < n) v = fmaf(P.w, acc[3], v);
    }
    return v;
}

// radii with a compiled-in convolution: Gaussian kernels at sigma = 1.88 .. 2.01 cells, the strict band of Delta = 6,
// the box of H = 4. A neighbouring radius in the general form costs 0 to 7 % more, 512x512x128 voxels, 64 x
// 128x128 rays: sigma 1.0 / 1.5 / 1.9 / 2.0 / 2.1 / 3.0 in 1,066 / 1,126 / 1,114 / 1,114 / 1,189 / 1,307 us (one
// output per lane and one load per tap, before: 1,700 / 1,811 / 1,701 / 1,703 / 1,941 / 2,245); box of H 3 / 4 / 5
// in 1,008 / 1,006 / 1,066 us.
__host__ __device__ constexpr bool conv_fixed(int K) { return K == 15 || K == 6 || K == 4; }

// FIXED / ANY: whether the kernel holds the compiled-in radii and the general form
template <bool FIXED, bool ANY>
__device__ __forceinline__ float band_conv(const float *CP, const float *CB, const float *gz, const RleTable &t, int K, int n)
{
    if (FIXED) {
        if (K == 15) return band_conv_k<15>(CP, CB, t, n);
        if (K == 6) return band_conv_k<6>(CP, CB, t, n);
        if (K == 4 || !ANY) return band_conv_k<4>(CP, CB, t, n);
    }
    return band_conv_any(CP, CB, gz, K, n);
}

// Theorem 5 at the cell level. The pairs (j, k) its sub-blocks keep (the whole diagonal block of
// each run, and for runs u < v the cells j >= s_v - Delta of run u with the cells k < e_u + Delta
// of run v, and the mirror image) are, for a first-hit cell j of run u, the contiguous cells
// [lo_j, hi_j) with lo_j = max(s of the run holding j - Delta, s_u - Delta) and
// hi_j = min(e_u + Delta, e of the run holding j + Delta) (cells clamped to [0, n); s, e a run's
// first cell and one past its last). So Theorem 5 is sum_j P(e_j) sum_{k in [lo_j, hi_j)} g(k - j)
// C_k, taken here with the taps |k - j| <= K of the banded convolution, in increasing k. RI holds
// each cell's run index, S the run starts (S[nr] = n).
__device__ __forceinline__ void kept_window(const int *S, const int *RI, int n, int D, int j, int &lo, int &hi)
{
    const int u = RI[j], a = max(j - D, 0), b = min(j + D, n - 1);
    lo = max(S[RI[a]], S[u] - D);
    hi = min(S[u + 1] + D, S[RI[b] + 1]);
}

__device__ __forceinline__ float window_conv(const float *CP, const float *CB, const float *gtab, int K, int n,
                                             const int *S, const int *RI, int D)
{
    float v = 0.0f;
    for (int j = lane_id(); j < n; j += 32) {
        int lo, hi;
        kept_window(S, RI, n, D, j, lo, hi);
        const int d0 = max(lo - j, -K), d1 = min(hi - j, K + 1);
        float acc = 0.0f;
        for (int d = d0; d < d1; ++d) acc = fmaf(gtab[K + d], CB[j + d], acc);
        v = fmaf(CP[j], acc, v);
    }
    return v;
}

// window_conv with a compile-time radius KK: the 2 KK + 1 kernel values in registers and every tap
// predicated on the window, so that no lane waits for another's longer window; the same products
// added in the same order (bit-identical). (Four cells per lane with 16-byte loads of C and a mask of taps per
// cell: 161 against 158 us on the 301x253x77 batch.)
template <int KK>
__device__ __forceinline__ float window_conv_k(const float *CP, const float *CB, const float *gtab, int n, const int *S,
                                               const int *RI, int D)
{
    float g[2 * KK + 1];
#pragma unroll
    for (int d = 0; d <= 2 * KK; ++d) g[d] = gtab[d];
    float v = 0.0f;
    for (int j = lane_id(); j < n; j += 32) {
        int lo, hi;
        kept_window(S, RI, n, D, j, lo, hi);
        const int d0 = lo - j + KK, w = hi - lo;  // taps d0 .. d0 + w - 1 of 0 .. 2 KK
        float acc = 0.0f;
#pragma unroll
        for (int d = 0; d <= 2 * KK; ++d)
            if ((unsigned)(d - d0) < (unsigned)w) acc = fmaf(g[d], CB[j + d - KK], acc);
        v = fmaf(CP[j], acc, v);
    }
    return v;
}

__host__ __device__ inline bool thm5_of(const DevParams &p) { return p.variant == FSMI_APPROX && p.approx_reading == 0; }
// Which evaluation paths a 3D kernel is compiled with (each kernel holds as little as it can, for its registers and
// the instruction cache): everything, with the variant and the ray's length read at run time; Theorem 5's sub-blocks;
// the others (cell-level convolution and all run pairs) with a general or with a compiled-in radius
// (conv_fixed).
enum { kRay3dAny = 0, kRay3dThm5 = 1, kRay3dOther = 2, kRay3dFixed = 3 };
__host__ __device__ inline int ray3d_mode(const DevParams &p)
{
    return thm5_of(p) ? kRay3dThm5 : conv_fixed(p.K) ? kRay3dFixed : kRay3dOther;
}

// The cells of a ray given as runs through scan_block: RI holds run u's index at its first cell and 0
// elsewhere; with keep it receives every cell's run index.
template <int CPL, bool POLY>
__device__ __forceinline__ void decompress(const DevParams &p, const float *O, int *RI, int n, float *CP, float *CB, bool keep)
{
    const int lane = lane_id();
    CellScan s{1.0f, 0.0f};
    int last = 0;  // run of the last cell before the block
    for (int base = 0; base < n; base += 32 * CPL) {
        const int i0 = base + CPL * lane;
        int u[CPL];
#pragma unroll
        for (int t = 0; t < CPL; ++t) u[t] = max(t ? u[t > 0 ? t - 1 : 0] : 0, i0 + t < n ? RI[i0 + t] : 0);
        int m = u[CPL - 1];  // running maximum over the lanes
#pragma unroll
        for (int k = 1; k < 32; k <<= 1) {
            const int v = __shfl_up_sync(kFull, m, k);
            if (lane >= k) m = max(m, v);
        }
        int before = __shfl_up_sync(kFull, m, 1);
        before = lane == 0 ? last : max(before, last);
        last = max(last, __shfl_sync(kFull, m, 31));
        float o[CPL];
#pragma unroll
        for (int t = 0; t < CPL; ++t) {
            u[t] = max(u[t], before);
            o[t] = i0 + t < n ? O[u[t]] : 0.0f;
        }
        if (keep && i0 < n) store_cells(RI + i0, u);
        scan_block<CPL, POLY>(p, o, i0, n, s, CP, CB);
    }
}

// Cell-level evaluation (eq. eqn_from_fsmi) of one ray given as runs: decompress the runs into the n virtual
// cells, form P(e_j) and C_k (Algorithms 2 and 3), then I = sum_j P(e_j) sum_{|d| <= K} g(d) C_{j+d}
// (FSMI-RLE, Uniform-FSMI-RLE, strict-band Approx-FSMI-RLE), or for Theorem 5 the same sum over each
// first-hit cell's window of kept pairs (window_conv). Each run's index is put at its first cell and
// spread by a running maximum. Arrays: 0 run o, 3 P, 4 run starts S, 5 the cells' run indices, 6 C.
template <int MODE, int CPL>
static __device__ float ray_mi_cells(float *base, int stride, int nr, int n, const DevParams &p, const float *gtab,
                                     const float *gz, const RleTable &t, int K)
{
    const int lane = lane_id();
    const float *O = base;
    float *CP = base + 3 * stride, *CB = base + 6 * stride + conv_pad(K);
    const int *S = (const int *)(base + 4 * stride);
    int *RI = (int *)(base + 5 * stride);
    for (int i = 4 * lane; i < n; i += 128) *reinterpret_cast<int4 *>(RI + i) = make_int4(0, 0, 0, 0);
    __syncwarp();
    for (int u = lane; u < nr; u += 32) RI[S[u]] = u;  // every run has a cell, so no two share one
    __syncwarp();
    if (CPL == 4 || (CPL == 0 && p.nmax > kShortRay))
        decompress<4, CPL != 0>(p, O, RI, n, CP, CB, MODE == kRay3dThm5);
    else
        decompress<2, CPL != 0>(p, O, RI, n, CP, CB, MODE == kRay3dThm5);
    __syncwarp();
    if (MODE == kRay3dThm5) return window_conv(CP, CB, gtab, K, n, S, RI, p.trunc);
    pad_conv(CB, K, n);
    return band_conv<MODE == kRay3dFixed, MODE == kRay3dOther>(CP, CB, gz, t, K, n);
}

template <int MODE, int CPL>
__device__ __forceinline__ float ray_mi(float *base, int stride, int nr, const DevParams &p, const float2 *tab,
                                        const float *gtab, const float *gz, const RleTable &t, int K, bool have_s)
{
    if (nr <= 0) return 0.0f;
    const RunSmem r = run_smem(base, stride);
    run_starts(r, nr, have_s);
    const int n = r.S[nr];
    float v;
    if (n < p.cell_runlen * nr) {
        v = ray_mi_cells<MODE, CPL>(base, stride, nr, n, p, gtab, gz, t, K);
    } else {
        run_prefixes(r, nr, p);
        if (MODE == kRay3dThm5)
            v = pairs_thm5(r, nr, tab, K, p.trunc);
        else
            v = pairs_all(r, nr, tab, K);
    }
    return warp_sum(v);
}

// ---- sampling and encoding -------------------------------------------------------------------

// Virtual cells of a ray: sample i is the voxel holding o + (i + 1/2) d, i.e. floor of the Q31 position
// (o << 15) + (2i + 1) d, for i < nsamp until the first sample outside the grid. Runs are maximal spans of
// bit-identical values split every `cap` cells from the span's start.

// Q31 position of sample 0, less d, and the direction (Q30) of a ray
__device__ __forceinline__ void ray_dir(const int32_t *pose, const int32_t *u, long long (&o)[3], long long (&d)[3])
{
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const long long acc = (long long)pose[3 + 3 * a] * u[0] + (long long)pose[4 + 3 * a] * u[1] +
                              (long long)pose[5 + 3 * a] * u[2];
        d[a] = (acc + (1LL << 29)) >> 30;
        o[a] = (long long)pose[a] << 15;
    }
}

// The encoder's form: writes O[u] = value, S[u] = first cell, S[nr] = n; returns nr.
static __device__ int sample_encode_ray(const float *__restrict__ vox, int X, int Y, int Z, const int32_t *pose,
                                        const int32_t *u, int nsamp, int cap, float *O, int *S)
{
    const int lane = lane_id();
    long long d[3], o[3];
    ray_dir(pose, u, o, d);
    int nrun = 0, carried = 0, n = 0;
    unsigned prev_bits = 0u;
    // Q31 position o + (2i + 1) d of this lane's sample, advanced by 64 d per chunk of 32
    long long q[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) q[a] = o[a] + (2LL * lane + 1) * d[a];
    const float inv_cap = 1.0f / (float)cap;
    const unsigned lane_le = 0xffffffffu >> (31 - lane);  // lanes 0 .. lane
    // this lane's sample of the chunk at `base`: whether it lies in the grid, and its voxel value
    auto fetch = [&](int i, bool &inb, float &val) {
        inb = false;
        val = 0.0f;
        if (i < nsamp) {
            // voxel = position >> 31; positions stay far below 2^62, so the low 32 bits of the
            // shifted value are the voxel when it is in the grid and a value >= the extent (as
            // unsigned) when it is not, negative positions included
            const unsigned px = (unsigned)(q[0] >> 31), py = (unsigned)(q[1] >> 31), pz = (unsigned)(q[2] >> 31);
            inb = px < (unsigned)X && py < (unsigned)Y && pz < (unsigned)Z;
            if (inb) val = __ldg(vox + ((size_t)(pz * (unsigned)Y + py) * (unsigned)X + px));
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) q[a] += 64 * d[a];
    };
    // the next chunk's gathers are issued before the current chunk is encoded
    bool inb_next;
    float val_next;
    fetch(lane, inb_next, val_next);
    for (int base = 0; base < nsamp; base += 32) {
        const int i = base + lane;
        const bool inb = inb_next;
        const float val = val_next;
        if (__all_sync(kFull, inb)) fetch(i + 32, inb_next, val_next);  // a chunk with a sample outside is the last
        const unsigned m_in = __ballot_sync(kFull, inb);
        const int nvalid = (m_in == kFull) ? 32 : (__ffs(~m_in) - 1);
        const bool valid = lane < nvalid;
        const unsigned bits = __float_as_uint(val);
        unsigned pbits = __shfl_up_sync(kFull, bits, 1);
        if (lane == 0) pbits = prev_bits;
        const bool newval = valid && (i == 0 || bits != pbits);
        // start of this cell's span of equal values: the last lane at or before this one where a new
        // value begins, else the span carried over from the previous chunk
        const unsigned mnew = __ballot_sync(kFull, newval);
        const unsigned nle = mnew & lane_le;
        const int st = nle ? base + 31 - __clz(nle) : carried;
        // a run of equal values splits every cap samples: (i - st) a multiple of cap, found with a
        // rounded quotient (exact: i - st < 2^20 and cap <= 255) instead of an integer remainder
        const int rel = i - st;
        const bool brk = valid && rel - __float2int_rn((float)rel * inv_cap) * cap == 0;
        const unsigned mb = __ballot_sync(kFull, brk);
        if (brk) {
            const int k = nrun + __popc(mb & ((1u << lane) - 1u));
            O[k] = val;
            S[k] = i;
        }
        nrun += __popc(mb);
        n += nvalid;
        if (nvalid < 32) break;
        carried = __shfl_sync(kFull, st, 31);
        prev_bits = __shfl_sync(kFull, bits, 31);
    }
    if (lane == 0) S[nrun] = n;
    __syncwarp();
    return nrun;
}

// Runs of a block of cells, CPL consecutive ones per lane (nw: a new value begins at the cell): O[k], S[k] of
// the runs below nrcap, and with RI every cell's run index.
struct RunScan {
    int nrun, carried;  // runs so far, start of the span that reaches into the block
};
template <int CPL>
__device__ __forceinline__ void encode_block(const float (&o)[CPL], const bool (&nw)[CPL], int i0, int n, int cap, float inv_cap,
                                             RunScan &s, float *O, int *S, int nrcap, int *RI)
{
    const int lane = lane_id();
    // start of each cell's span: the last cell at or before it where a new value begins
    int st[CPL], own = -1;
#pragma unroll
    for (int t = 0; t < CPL; ++t) {
        if (nw[t]) own = i0 + t;
        st[t] = own;
    }
    int m = own;
#pragma unroll
    for (int k = 1; k < 32; k <<= 1) {
        const int w = __shfl_up_sync(kFull, m, k);
        if (lane >= k) m = max(m, w);
    }
    int from = __shfl_up_sync(kFull, m, 1);
    from = lane == 0 ? s.carried : max(from, s.carried);
    s.carried = max(s.carried, __shfl_sync(kFull, m, 31));
    bool brk[CPL];
    int cnt = 0;
#pragma unroll
    for (int t = 0; t < CPL; ++t) {
        const int rel = i0 + t - max(st[t], from);  // a multiple of cap starts a run (exact, see sample_encode_ray)
        brk[t] = i0 + t < n && rel - __float2int_rn((float)rel * inv_cap) * cap == 0;
        cnt += brk[t];
    }
    const int incl = warp_incl_add_int(cnt);
    int k = s.nrun + incl - cnt, r[CPL];
    s.nrun += __shfl_sync(kFull, incl, 31);
#pragma unroll
    for (int t = 0; t < CPL; ++t) {
        if (brk[t]) {
            if (k < nrcap) {
                O[k] = o[t];
                S[k] = i0 + t;
            }
            ++k;
        }
        r[t] = k - 1;
    }
    if (RI && i0 < n) store_cells(RI + i0, r);
}

// The fused kernel's form: blocks of 128 samples, four consecutive ones per lane, straight through scan_block into
// P (CP) and C (CB). Returns n. With ENC the runs are formed on the way (O, S, RI; count = their number), else the
// values go to CO (for encode_cells) and count = the number of spans of equal values.
//
// What bounds it is instructions per sample. One sample per lane and chunk of 32 took, per chunk, a ballot and
// a scan step for each of the range end, the spans, the run splits and the two prefixes, the gains spread
// from the spans through shared memory, and six array accesses; a block of 128 pays the warp-wide steps
// once and stores three 16-byte words. 512x512x128 voxels, 64 poses x 128x128 rays: 1,741 to 1,068 warp
// instructions per ray and 1,690 to 1,136 us, with the convolution below (73 registers, 28 warps per SM; held
// to 64: 1,152 - 1,172 us), then 1,103 us with a kernel per path and ray length (80 registers, 24 warps); Theorem 5
// on 301x253x77 voxels, 23 x 80x61 rays: 162 to 150 us in all.
template <int CPL, bool ENC, bool POLY>
__device__ __forceinline__ int sample_cells(const float *__restrict__ vox, int X, int Y, int Z, const int32_t *pose,
                                            const int32_t *u, int nsamp, const DevParams &p, float *CP, float *CB, float *CO,
                                            float *O, int *S, int nrcap, int *RI, int &count)
{
    const int lane = lane_id();
    long long d[3], q[3];
    ray_dir(pose, u, q, d);
#pragma unroll
    for (int a = 0; a < 3; ++a) q[a] += (2LL * CPL * lane + 1) * d[a];  // sample CPL lane
    CellScan s{1.0f, 0.0f};
    RunScan rs{0, 0};
    const float inv_cap = 1.0f / (float)p.run_cap;
    unsigned prev = 0u;
    int n = 0, spans = 0;
    for (int base = 0; base < nsamp; base += 32 * CPL) {
        const int i0 = base + CPL * lane;
        float o[CPL];
        bool in[CPL];
#pragma unroll
        for (int t = 0; t < CPL; ++t) {
            // as in sample_encode_ray
            const unsigned px = (unsigned)(q[0] >> 31), py = (unsigned)(q[1] >> 31), pz = (unsigned)(q[2] >> 31);
            in[t] = px < (unsigned)X && py < (unsigned)Y && pz < (unsigned)Z && i0 + t < nsamp;
            o[t] = in[t] ? __ldg(vox + ((size_t)(pz * (unsigned)Y + py) * (unsigned)X + px)) : 0.0f;
#pragma unroll
            for (int a = 0; a < 3; ++a) q[a] += (t < CPL - 1 ? 2 : 64 * CPL - 2 * CPL + 2) * d[a];
        }
        // the ray ends at its first sample outside
        const int c = !in[0] ? 0 : !in[1] ? 1 : CPL == 2 || !in[CPL - 2] ? 2 : !in[CPL - 1] ? 3 : 4;
        const unsigned m = __ballot_sync(kFull, c == CPL);
        const int L = m == kFull ? 31 : __ffs(~m) - 1;
        n = base + CPL * L + __shfl_sync(kFull, c, L);
        const unsigned left = __shfl_up_sync(kFull, __float_as_uint(o[CPL - 1]), 1);
        unsigned before = lane == 0 ? prev : left;
        prev = __shfl_sync(kFull, __float_as_uint(o[CPL - 1]), 31);
        bool nw[CPL];
#pragma unroll
        for (int t = 0; t < CPL; ++t) {
            const unsigned bits = __float_as_uint(o[t]);
            const bool valid = i0 + t < n;
            nw[t] = valid && (bits != before || i0 + t == 0);
            spans += nw[t];
            before = bits;
            if (!valid) o[t] = 0.0f;
        }
        if (ENC)
            encode_block<CPL>(o, nw, i0, n, p.run_cap, inv_cap, rs, O, S, nrcap, RI);
        else if (i0 < n)
            store_cells(CO + i0, o);
        scan_block<CPL, POLY>(p, o, i0, n, s, CP, CB);
        if (m != kFull) break;
    }
    if (ENC) {
        if (lane == 0 && rs.nrun <= nrcap) S[rs.nrun] = n;
        count = rs.nrun;
    } else {
        count = __reduce_add_sync(kFull, spans);
    }
    __syncwarp();
    return n;
}

// Run-length encoding of the n cells in CO; returns the number of runs (S[nr] = n if nr <= nrcap).
static __device__ int encode_cells(const float *CO, int n, int cap, float *O, int *S, int nrcap)
{
    const int lane = lane_id();
    const float inv_cap = 1.0f / (float)cap;
    RunScan rs{0, 0};
    unsigned prev = 0u;
    for (int base = 0; base < n; base += 128) {
        const int i0 = base + 4 * lane;
        float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (i0 < n) v = *reinterpret_cast<const float4 *>(CO + i0);
        const float o[4] = {v.x, v.y, v.z, v.w};
        const unsigned left = __shfl_up_sync(kFull, __float_as_uint(o[3]), 1);
        unsigned before = lane == 0 ? prev : left;
        prev = __shfl_sync(kFull, __float_as_uint(o[3]), 31);
        bool nw[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const unsigned bits = __float_as_uint(o[t]);
            nw[t] = i0 + t < n && (bits != before || i0 + t == 0);
            before = bits;
        }
        encode_block<4>(o, nw, i0, n, cap, inv_cap, rs, O, S, nrcap, nullptr);
    }
    if (lane == 0 && rs.nrun <= nrcap) S[rs.nrun] = n;
    __syncwarp();
    return rs.nrun;
}

// ---- the fused 3D ray (sampling and evaluation in one warp) --------------------------------------
//
// Per-warp layout: per-cell P (CP), o (CO) and C padded by zeros on both sides (CB), each
// cell_stride floats (absent for Theorem 5's sub-blocks, which always use the runs), then the six
// run arrays sized for the runs the run-pair path can see: a ray takes that path only when
// n >= cell_runlen * n_r, so n_r <= nmax / cell_runlen.

__host__ __device__ inline int ray3d_cell_stride(const DevParams &p) { return (p.nmax + conv_pad(p.K) + p.K + 12 + 3) & ~3; }
__host__ __device__ inline int ray3d_nrcap(const DevParams &p)
{
    const int T = p.cell_runlen > 0 ? p.cell_runlen : 1;
    return thm5_of(p) ? p.nmax : min(p.nmax, p.nmax / T + 2);
}
__host__ __device__ inline int ray3d_run_stride(const DevParams &p) { return ((ray3d_nrcap(p) + 2) + 3) & ~3; }
// Per-warp floats of the fused 3D path. The others: [CP | CO | CB | six run arrays]. Theorem 5 (all
// runs stored): [S | O | four cell-stride arrays], the four holding CP, CO, CB and the cells' run
// indices for the cell form, or the run arrays X, A, F, L for the run pairs.
__host__ __device__ inline int ray3d_warp_floats(const DevParams &p)
{
    return thm5_of(p) ? 2 * ray3d_run_stride(p) + 4 * ray3d_cell_stride(p)
                      : 3 * ray3d_cell_stride(p) + 6 * ray3d_run_stride(p);
}

// Samples and evaluates one ray in the warp's region `w` (ray3d_warp_floats floats); returns the MI
// (warp-reduced) and, with nr_out, the run count. MODE must agree with ray3d_mode(p). Outside Theorem 5 the runs are
// formed (from the sampled values in shared memory) only where they are needed: for a caller who asks for
// their number, or on a ray whose spans of equal values do not already show that its mean run is short.
// CPL: cells per lane of a block, 2 for rays of at most kShortRay samples, else 4, both for polynomial gains only (the
// closed forms' code takes registers from every ray); 0: ray length and gains read at run time.
template <int MODE, int CPL>
__device__ __forceinline__ float ray_mi_fused(const float *vox, int X, int Y, int Z, const int32_t *pose,
                                              const int32_t *u, int nsamp, const DevParams &p, const float2 *tab,
                                              const float *gtab, const float *gz, const RleTable &t, int K, float *w,
                                              int *nr_out)
{
    const bool thm5 = MODE == kRay3dAny ? thm5_of(p) : MODE == kRay3dThm5;
    const int cst = ray3d_cell_stride(p), rst = ray3d_run_stride(p);
    float *CP, *CO, *CB;
    int *RI = nullptr;
    RunSmem r;
    if (thm5) {
        float *c4 = w + 2 * rst;
        CP = c4;
        CO = c4 + cst;
        CB = c4 + 2 * cst + conv_pad(K);
        RI = (int *)(c4 + 3 * cst);
        r.S = (int *)w;
        r.O = w + rst;
        r.X = CP;
        r.A = CO;
        r.F = c4 + 2 * cst;
        r.L = RI;
    } else {
        CP = w;
        CO = w + cst;
        CB = w + 2 * cst + conv_pad(K);
        r = run_smem(w + 3 * cst, rst);
    }
    int n, nr = 0;
    bool cells;
    if (thm5) {
        n = CPL == 4 || (CPL == 0 && nsamp > kShortRay)
                ? sample_cells<4, true, CPL != 0>(vox, X, Y, Z, pose, u, nsamp, p, CP, CB, CO, r.O, r.S, ray3d_nrcap(p), RI, nr)
                : sample_cells<2, true, CPL != 0>(vox, X, Y, Z, pose, u, nsamp, p, CP, CB, CO, r.O, r.S, ray3d_nrcap(p), RI, nr);
        cells = n < p.cell_runlen * nr;
    } else {
        int nspan;
        n = CPL == 4 || (CPL == 0 && nsamp > kShortRay)
                ? sample_cells<4, false, CPL != 0>(vox, X, Y, Z, pose, u, nsamp, p, CP, CB, CO, nullptr, nullptr, 0, nullptr, nspan)
                : sample_cells<2, false, CPL != 0>(vox, X, Y, Z, pose, u, nsamp, p, CP, CB, CO, nullptr, nullptr, 0, nullptr, nspan);
        cells = n < p.cell_runlen * nspan;  // at least one run per span
        if (n > 0 && (nr_out || !cells)) {
            nr = encode_cells(CO, n, p.run_cap, r.O, r.S, ray3d_nrcap(p));
            cells = n < p.cell_runlen * nr;
        }
    }
    if (nr_out) *nr_out = nr;
    if (n == 0) return 0.0f;
    float v;
    if (cells) {
        // eq. eqn_from_fsmi on the virtual cells: the banded convolution (Theorem 5: over each first-hit
        // cell's window of kept pairs)
        if (thm5) {
            v = MODE == kRay3dThm5 && K == 15 ? window_conv_k<15>(CP, CB, gtab, n, r.S, RI, p.trunc)
                                               : window_conv(CP, CB, gtab, K, n, r.S, RI, p.trunc);
        } else {
            pad_conv(CB, K, n);
            v = band_conv<MODE == kRay3dAny || MODE == kRay3dFixed, MODE == kRay3dAny || MODE == kRay3dOther>(CP, CB, gz, t, K, n);
        }
    } else {  // here n_r <= nrcap, so every run was stored
        run_starts(r, nr, true);
        run_prefixes(r, nr, p);
        v = thm5 ? pairs_thm5(r, nr, tab, K, p.trunc) : pairs_all(r, nr, tab, K);
    }
    return warp_sum(v);
}

// pose and ray of batch item `ray` = pose * R + r (a 32-bit division when ray fits, the common case)
__device__ __forceinline__ void split_ray(long long ray, int R, int &pi, int &ri)
{
    if (ray <= 0x7fffffffLL) {
        pi = (int)((unsigned)ray / (unsigned)R);
        ri = (int)((unsigned)ray - (unsigned)pi * (unsigned)R);
    } else {
        pi = (int)(ray / R);
        ri = (int)(ray % R);
    }
}

// ray = pose * R + r of a batch
__device__ __forceinline__ int sample_encode(const Vox3D &v, long long ray, int nsamp, int cap, float *O, int *S)
{
    int pi, ri;
    split_ray(ray, v.R, pi, ri);
    return sample_encode_ray(v.vox, v.X, v.Y, v.Z, v.poses + 12 * (size_t)pi, v.dirs + 3 * (size_t)ri, nsamp, cap, O,
                             S);
}

// ---- kernels -----------------------------------------------------------------------------------

struct TabSpec {
    int kind, H, band, K;
    double sigma;
};

__host__ __device__ inline TabSpec table_spec(const DevParams &p)
{
    TabSpec t;
    t.sigma = p.sigma;
    t.H = p.H;
    t.band = -1;
    t.K = p.K;
    if (p.variant == FSMI_UNIFORM) {
        t.kind = 2;
    } else {
        t.kind = p.g_kernel == FSMI_G_ERF ? 1 : 0;
        if (p.variant == FSMI_APPROX && p.approx_reading == 1) t.band = p.trunc;
    }
    return t;
}

// shared memory: [tab float2 (2K+2)] [gtab float (2K+1)] [gz float 4 (conv_quads + 1)] [per-warp arrays]
__host__ __device__ inline size_t rle_gz_at(int K)
{
    return ((size_t)(2 * K + 2) * sizeof(float2) + (size_t)(2 * K + 1) * sizeof(float) + 15) & ~(size_t)15;
}
__host__ __device__ inline size_t rle_table_bytes(int K) { return rle_gz_at(K) + 16 * (size_t)(conv_quads(K) + 1); }

// Shared-memory layout of the RLE evaluation kernels: the block's kernel table, then each warp's arrays.
struct RleBlock {
    TabSpec ts;
    float2 *tab;
    float *gtab, *gz;
    float *base;
};

// the tables at the front of the block's shared memory, loaded
__device__ __forceinline__ RleBlock rle_tables(unsigned char *smem_raw, const DevParams &p, const RleTable &t, bool load)
{
    RleBlock rb;
    rb.ts = table_spec(p);
    rb.tab = (float2 *)smem_raw;
    rb.gtab = (float *)(smem_raw + (size_t)(2 * rb.ts.K + 2) * sizeof(float2));
    rb.gz = (float *)(smem_raw + rle_gz_at(rb.ts.K));
    if (load) load_table(rb.tab, rb.gtab, rb.gz, rb.ts.K, t);
    return rb;
}

__device__ __forceinline__ RleBlock rle_block(unsigned char *smem_raw, const DevParams &p, const RleTable &t,
                                              int warp_floats)
{
    RleBlock rb = rle_tables(smem_raw, p, t, true);
    rb.base = (float *)(smem_raw + rle_table_bytes(rb.ts.K)) + (size_t)(threadIdx.x >> 5) * warp_floats;
    return rb;
}

// sampling, encoding and evaluation of one 3D ray (= pose * R + r), fused layout; WIDE: the batch
// has more than 2^31 - 1 rays (64-bit index division), else a 32-bit one
template <int MODE, int CPL, bool WIDE>
__device__ __forceinline__ void eval_ray_3d(const Vox3D &vx, const DevParams &p, const RleBlock &rb, const RleTable &t,
                                            long long ray, float *__restrict__ out, int32_t *__restrict__ nruns)
{
    int pi, ri;
    if (WIDE) {
        pi = (int)(ray / vx.R);
        ri = (int)(ray % vx.R);
    } else {
        pi = (int)((unsigned)ray / (unsigned)vx.R);
        ri = (int)((unsigned)ray - (unsigned)pi * (unsigned)vx.R);
    }
    int nr = 0;
    const float I = ray_mi_fused<MODE, CPL>(vx.vox, vx.X, vx.Y, vx.Z, vx.poses + 12 * (size_t)pi, vx.dirs + 3 * (size_t)ri, p.nmax,
                                 p, rb.tab, rb.gtab, rb.gz, t, rb.ts.K, rb.base, nruns ? &nr : nullptr);
    if (lane_id() == 0) {
        out[ray] = I;
        if (nruns) nruns[ray] = nr;
    }
    __syncwarp();
}

// evaluation of one run-length-encoded ray given in CSR form (MODE, CPL as ray_mi_fused's, CPL by p.nmax)
template <int MODE, int CPL>
__device__ __forceinline__ void eval_ray_rle(const int32_t *__restrict__ off, const float *__restrict__ ro,
                                             const uint8_t *__restrict__ rl, const DevParams &p, const RleBlock &rb,
                                             const RleTable &t, int stride, long long ray, float *__restrict__ out, int *status)
{
    const int lane = lane_id();
    const RunSmem r = run_smem(rb.base, stride);
    const int b = off[ray];
    const int nr = off[ray + 1] - b;
    bool bad = b < 0 || nr < 0 || nr > p.nmax;
    int cells = 0;
    if (!bad) {
        for (int u = lane; u < nr; u += 32) {
            const int L = rl[b + u];
            r.O[u] = __ldg(ro + b + u);
            r.L[u] = L;
            cells += L;
            bad |= (L == 0);
        }
        cells = __reduce_add_sync(kFull, cells);
        bad = __any_sync(kFull, bad) || cells > p.nmax;
    }
    __syncwarp();
    if (bad) {
        if (lane == 0) {
            out[ray] = __int_as_float(0x7fc00000);
            set_status(status, FSMI_STATUS_BAD_BEAM);
        }
        __syncwarp();
        return;
    }
    const float I = ray_mi<MODE, CPL>(rb.base, stride, nr, p, rb.tab, rb.gtab, rb.gz, t, rb.ts.K, false);
    if (lane == 0) out[ray] = I;
    __syncwarp();
}

}  // namespace fsmi
