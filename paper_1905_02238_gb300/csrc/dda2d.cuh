// Fixed-point 2D ray traversal shared by the evaluation, visit-stamp and map-update kernels: the
// cells a beam crosses (Section 2.2 lists them in ascending distance) with their entry distances.
#pragma once

#include <stdint.h>

#include "fsmi_device.cuh"

namespace fsmi {

// Beam direction: the sensor-frame unit vector u rotated by the pose's (cos, sin), rounded half
// up: d = floor((Rot u + 2^29) / 2^30). Arithmetic right shift is a floor division by 2^30.
__device__ __forceinline__ void beam_dir(const int32_t *pose, int32_t ux, int32_t uy, int &dx, int &dy)
{
    const long long c = pose[2], s = pose[3];
    dx = (int)((c * ux - s * uy + (1LL << 29)) >> 30);
    dy = (int)((s * ux + c * uy + (1LL << 29)) >> 30);
}

// ---- traversal ----------------------------------------------------------------------------------
//
// The beam is o + lambda * d / 2^30 (o in Q16 cell units, d in Q30); lambda is its distance. Cells
// change at x crossings lambda_x(a) = (nx0 + a 2^16) 2^14 / |dx| and y crossings likewise, with
// nx0, ny0 the Q16 distances from o to the far side of the first cell (the cell entered by
// o + eps d). Crossings are ordered by exact int64 comparison; coinciding crossings are one
// diagonal step. A cell is entered while its entry lambda < R and it lies inside the grid.
//
// Parallel form: along the major axis M (|d_M| >= |d_m|) consecutive M-crossings split the beam
// into intervals [lambda_M(k), lambda_M(k+1)), k = -1, 0, 1, ... (lambda_M(-1) = 0). Minor
// crossings are at least as far apart as major ones, so each interval holds the cell entered at
// its start plus at most one cell entered at a minor crossing strictly inside it. Lane L walks a
// contiguous block of intervals k0..k1; its starting minor coordinate is the number of minor
// crossings at or before lambda_M(k0) (one integer division). Its cell count, unless the beam
// ends inside the block, is (k1 - k0 + 1) + (minor crossings in (lambda_M(k0), lambda_M(k1+1)])
// minus the crossings among those that coincide with a major crossing (diagonal steps, which
// enter one cell, not two). The lanes write their cells at offsets from a warp scan of that count
// taken without the coincidences, and count the coincidences as they walk; if a lane before the
// one where the beam ends met any, the offsets were too large and the lanes walk again at the
// exact offsets (beams along a lattice diagonal through cell centres; rare otherwise). The first
// lane that meets the range limit or the grid boundary ends the beam.

struct Geo {
    int sM, sm, cM0, cm0, dimM, dimm, xmaj, W;
    unsigned nM0, nm0;  // Q16 distances to the first major / minor boundary (< 2^31 + 2^16 with k)
    unsigned aM, am;    // |d| along the major / minor axis (Q30, <= 2^31)
    unsigned LM, Lm;    // crossing numerators below these have entry distance < R
    float rM, rm, R;
};

__device__ __forceinline__ unsigned long long mulw(unsigned a, unsigned b) { return (unsigned long long)a * b; }

// Number of minor crossings at or before the major crossing k: #{i >= 0 : nm(i) aM <= nM(k) am}
// = floor((nM(k) am - nm0 aM) / (2^16 aM)) + 1 when that numerator is >= 0. The quotient (< 2^11
// for ranges up to 1024 cells) is estimated in FP32 and corrected exactly in integers.
__device__ __forceinline__ int minor_before(const Geo &g, int k)
{
    if (g.am == 0 || k < 0) return 0;
    const long long num = (long long)mulw(g.nM0 + (unsigned)k * 65536u, g.am) - (long long)mulw(g.nm0, g.aM);
    if (num < 0) return 0;
    const long long hi = num >> 16;  // floor(num / 2^16); floor(hi / aM) = floor(num / (2^16 aM))
    long long q = (long long)((float)hi * (1.0f / (float)g.aM));
    q -= (q * (long long)g.aM > hi);
    q -= (q * (long long)g.aM > hi);
    q += ((q + 1) * (long long)g.aM <= hi);
    q += ((q + 1) * (long long)g.aM <= hi);
    return (int)q + 1;
}

// Walks intervals k0..k1 from minor crossing i0 = minor_before(k0), writing (WRITE) its cells
// from index `base`; cnt = cells entered, ties = minor crossings that coincided with a major one
// (diagonal steps) before the walk ended. CHECK: skip writes at indices >= cap (not needed when
// every index the walk can reach is below cap). The current cell's id advances with its
// coordinates (by stepM per major step, stepm per minor step) rather than being recomputed.
template <bool WRITE, bool CHECK = true>
__device__ __forceinline__ void walk(const Geo &g, int k0, int k1, int i0, int base, int cap, int *ids, float *l,
                                     int &cnt, int &ties, bool &ended, float &endl, bool &by_range)
{
    int cM = g.cM0 + g.sM * (k0 + 1);
    int i = i0;
    int cm = g.cm0 + g.sm * i;
    const int stepM = g.xmaj ? g.sM : g.sM * g.W, stepm = g.xmaj ? g.sm * g.W : g.sm;
    int id = g.xmaj ? (cm * g.W + cM) : (cM * g.W + cm);
    int *ip = ids + base;
    float *lp = l + base;
    cnt = 0;
    ties = 0;
    ended = false;
    endl = 0.0f;
    by_range = false;
#define FSMI_EMIT(lam_)                                                              \
    do {                                                                             \
        if (WRITE && (!CHECK || base + cnt < cap)) {                                 \
            *ip = id;                                                                \
            *lp = (lam_);                                                            \
        }                                                                            \
        ++ip;                                                                        \
        ++lp;                                                                        \
        ++cnt;                                                                       \
    } while (0)
    // crossings are compared as nm(i) aM against nM(k + 1) am; both products advance by constant
    // steps (aM 2^16 per minor crossing, am 2^16 per interval), so the loop multiplies nothing
    unsigned nMn = g.nM0 + (unsigned)(k0 + 1) * 65536u;  // next major crossing
    unsigned nmi = g.nm0 + (unsigned)i * 65536u;         // next minor crossing
    unsigned long long pm = mulw(nmi, g.aM), pM = mulw(nMn, g.am);
    const unsigned long long dm = (unsigned long long)g.aM << 16, dM = (unsigned long long)g.am << 16;
    for (int k = k0; k <= k1; ++k, nMn += 65536u, pM += dM) {
        FSMI_EMIT(k < 0 ? 0.0f : (float)(nMn - 65536u) * g.rM);
        const bool minor = g.am && pm < pM;  // a minor crossing inside the interval
        if (minor && (nmi >= g.Lm || (unsigned)(cm + g.sm) >= (unsigned)g.dimm)) {  // the beam ends there
            ended = true;
            by_range = nmi >= g.Lm;
            endl = by_range ? g.R : (float)nmi * g.rm;
            break;
        }
        if (minor) {  // no branch inside: the lanes stay together whichever of them cross
            cm += g.sm;
            id += stepm;
            FSMI_EMIT((float)nmi * g.rm);
            ++i;
            nmi += 65536u;
            pm += dm;
        }
        if (nMn >= g.LM) {
            ended = true;
            endl = g.R;
            by_range = true;
            break;
        }
        const bool tie = g.am && pm == pM;
        cM += g.sM;
        id += stepM;
        if (tie) {
            cm += g.sm;
            id += stepm;
            ++i;
            nmi += 65536u;
            pm += dm;
            ++ties;
        }
        if ((unsigned)cM >= (unsigned)g.dimM || (unsigned)cm >= (unsigned)g.dimm) {
            ended = true;
            endl = (float)nMn * g.rM;
            break;
        }
    }
#undef FSMI_EMIT
}

// ---- closed form ----------------------------------------------------------------------------------
//
// Without diagonal steps everything about interval k follows from i_k, the number of minor crossings
// at or before major crossing k: its first cell is (cM0 + sM (k + 1), cm0 + sm i_k), at list index
// k + 1 + i_k, and it holds a second cell when i_{k+1} > i_k. i_k is the floor of
// V_k = (nM(k) am - nm0 aM) / (2^16 aM) + 1 = V_0 + k am / aM, which fixed point gives for one
// interval per lane with an addition per chunk of 32 intervals; no walk, no division per lane and no
// scan. V is kept with 32 fractional bits and is off by less than kSlack of its last bits, so the
// floor is exact unless V lies within kSlack of an integer; a coinciding crossing (diagonal step) has
// V_k an integer and is caught the same way. Such beams (lattice directions, and about one in a
// thousand others) take the walk below. The two forms give the same cells and the same floats.
//
// On the 2048x2048 office batch (R = 256) the walk took 743 of the 1,717 warp instructions of a
// Uniform-FSMI beam; with the closed form, gathering as it goes, and 16-byte prefix scans it issues
// 1,381 (702 -> 660 us; exact 1,688 -> 1,621 us). What bounds it now is the gathers: 16 bytes each from
// 32 different lines, half of the shared-memory and L1 wavefronts.

constexpr unsigned kSlack = 4096;  // >= 1.5 (K + 2) + 2 for K <= 2048 major crossings

struct Fixed {
    unsigned long long V;     // V_{k+1} of this lane's interval (32 fractional bits)
    unsigned R;               // am / aM
    unsigned long long V0;
    int I;                    // minor crossings 0 .. I - 1 are in range and inside the grid
    bool amb;                 // a floor on the way was not certain
};

// V_0 and the slope, or false where the closed form does not apply (am = aM: a diagonal)
__device__ __forceinline__ bool fixed_setup(const Geo &g, Fixed &f)
{
    if (g.am == g.aM) return false;
    f.amb = false;
    if (g.am == 0) {
        f.R = 0;
        f.V0 = 1ull << 31;
        f.I = 1 << 20;
    } else {
        const float inv = __fdividef(1.0f, (float)g.aM);
        f.R = (unsigned)fminf((float)g.am * inv * 4294967296.0f, 4294966784.0f);
        // the estimate is off by 2^-21 of itself at most; the remainder gives the rest to 1.5 units
        const long long rem = ((long long)g.am << 32) - (long long)mulw(f.R, g.aM);
        f.R += (unsigned)__float2int_rn((float)rem * inv);
        f.V0 = (1ull << 32) + (mulw(g.nM0, f.R) >> 16) - ((unsigned long long)g.nm0 << 16);
        const int IR = g.Lm > g.nm0 ? (int)((g.Lm - g.nm0 + 65535u) >> 16) : 0;
        const int IG = g.sm > 0 ? g.dimm - 1 - g.cm0 : g.cm0;
        f.I = min(IR, IG);
    }
    f.V = f.V0 + mulw(lane_id(), f.R);
    return true;
}

// One interval of a chunk: whether its first and second cells belong to the beam, the first cell's
// list index and id (the second's are pos + 1 and id + stepm), and their entry distances.
struct Interval {
    bool ok1, ok2;
    int pos, id;
    float lam1, lam2;
};

// The interval k = base + lane - 1 of the chunk at `base` (advances f to the next chunk).
__device__ __forceinline__ Interval fixed_interval(const Geo &g, Fixed &f, int K, int base, int id0, int stepM, int stepm)
{
    Interval v;
    const int k1 = base + lane_id();  // k + 1
    const int in = (int)(f.V >> 32);
    const int i = k1 == 0 ? 0 : (int)((f.V - f.R) >> 32);
    v.ok1 = k1 <= K && i <= f.I;
    v.ok2 = v.ok1 && in > i && i < f.I;
    f.amb |= k1 <= K && (unsigned)f.V + kSlack < 2u * kSlack;
    v.pos = k1 + i;
    v.id = id0 + k1 * stepM + i * stepm;
    v.lam1 = k1 == 0 ? 0.0f : (float)(g.nM0 + (unsigned)(k1 - 1) * 65536u) * g.rM;
    v.lam2 = (float)(g.nm0 + (unsigned)i * 65536u) * g.rm;
    f.V += 32ull * f.R;
    return v;
}

// Runs the chunks of a beam of K major crossings in groups of UN: use(Interval (&)[UN]) is called by
// all lanes; then the cell count, the end distance and whether the beam ended by range. Returns -1
// if the beam has to be walked instead (what `use` saw is then void: ids may lie outside the grid,
// list indices below fixed_cells).
template <int UN, class F>
__device__ __forceinline__ int fixed_run(const Geo &g, Fixed &f, int K, F &&use, float &lend, bool &by_range)
{
    const int stepM = g.xmaj ? g.sM : g.sM * g.W, stepm = g.xmaj ? g.sm * g.W : g.sm;
    const int id0 = g.xmaj ? g.cm0 * g.W + g.cM0 : g.cM0 * g.W + g.cm0;
    int nint = 0;  // intervals of the beam
    for (int base = 0; base <= K; base += 32 * UN) {
        Interval v[UN];
#pragma unroll
        for (int u = 0; u < UN; ++u) v[u] = fixed_interval(g, f, K, base + 32 * u, id0, stepM, stepm);
        use(v);
        unsigned m = 0;
#pragma unroll
        for (int u = 0; u < UN; ++u) {
            m = __ballot_sync(kFull, v[u].ok1);
            nint += __popc(m);
        }
        if (m != kFull) break;
    }
    if (__any_sync(kFull, f.amb)) return -1;
    // the last interval, k = nint - 2, ends at its minor crossing if that is not allowed, else at major K
    const unsigned long long Ve = f.V0 + mulw((unsigned)(nint - 1), f.R);
    const int in = (int)(Ve >> 32), i = nint == 1 ? 0 : (int)((Ve - f.R) >> 32);
    const bool inner = in > i;
    if (inner && i == f.I) {
        const unsigned nm = g.nm0 + (unsigned)i * 65536u;
        by_range = nm >= g.Lm;
        lend = by_range ? g.R : (float)nm * g.rm;
    } else {
        const unsigned nM = g.nM0 + (unsigned)K * 65536u;
        by_range = nM >= g.LM;
        lend = by_range ? g.R : (float)nM * g.rM;
    }
    return nint + i + (inner && i < f.I ? 1 : 0);
}

// ---- a beam ----------------------------------------------------------------------------------------

// Geometry of a beam; false if it crosses no cell. K = major crossings in range and inside the grid.
__device__ __forceinline__ bool beam_geo(int W, int H, int ox, int oy, int dx, int dy, long long rfix, float rend, Geo &g,
                                         int &K)
{
    if ((dx | dy) == 0) return false;
    int cx = ox >> 16, cy = oy >> 16;
    if (dx < 0 && (ox & 0xFFFF) == 0) --cx;
    if (dy < 0 && (oy & 0xFFFF) == 0) --cy;
    if ((unsigned)cx >= (unsigned)W || (unsigned)cy >= (unsigned)H) return false;
    const unsigned adx = dx < 0 ? 0u - (unsigned)dx : (unsigned)dx, ady = dy < 0 ? 0u - (unsigned)dy : (unsigned)dy;
    g.xmaj = adx >= ady;
    g.W = W;
    g.aM = g.xmaj ? adx : ady;
    g.am = g.xmaj ? ady : adx;
    const int dM = g.xmaj ? dx : dy, dm = g.xmaj ? dy : dx;
    g.sM = dM > 0 ? 1 : -1;
    g.sm = dm > 0 ? 1 : -1;
    g.cM0 = g.xmaj ? cx : cy;
    g.cm0 = g.xmaj ? cy : cx;
    g.dimM = g.xmaj ? W : H;
    g.dimm = g.xmaj ? H : W;
    // distances to the first boundaries, in (0, 2^16] (32-bit arithmetic modulo 2^32 is exact)
    const unsigned oM = (unsigned)(g.xmaj ? ox : oy), om = (unsigned)(g.xmaj ? oy : ox);
    g.nM0 = g.sM > 0 ? ((unsigned)(g.cM0 + 1) << 16) - oM : oM - ((unsigned)g.cM0 << 16);
    g.nm0 = g.am == 0 ? 0u : g.sm > 0 ? ((unsigned)(g.cm0 + 1) << 16) - om : om - ((unsigned)g.cm0 << 16);
    // crossing numerators below these limits have entry lambda < R:
    //   num * 2^30 < rfix * a  <=>  num < floor((rfix * a - 1) / 2^30) + 1
    g.LM = (unsigned)((((unsigned long long)rfix * g.aM - 1) >> 30) + 1);
    g.Lm = g.am ? (unsigned)((((unsigned long long)rfix * g.am - 1) >> 30) + 1) : 0u;
    g.rM = __fdividef(16384.0f, (float)g.aM);  // distances need not be correctly rounded (< 2 ulp)
    g.rm = g.am ? __fdividef(16384.0f, (float)g.am) : 0.0f;
    g.R = rend;
    // major crossings that stay in range and inside the grid along M
    const long long KR = g.LM > g.nM0 ? ((long long)g.LM - g.nM0 + 65535) >> 16 : 0;
    const long long KG = g.sM > 0 ? (g.dimM - 1 - g.cM0) : g.cM0;
    K = (int)(KR < KG ? KR : KG);
    return true;
}

// cells the closed form may place: every list index lies below this
__device__ __forceinline__ int fixed_cells(const Fixed &f, int K)
{
    return K + 1 + min(f.I, (int)((f.V0 + mulw((unsigned)K, f.R)) >> 32));
}

// The beam walked by blocks of intervals (see the top of this file); all 32 lanes. Writes
// ids[0..n-1] and l[0..n-1] and returns n, or -1 if the beam has more than cap cells.
static __device__ int dda_walk(const Geo &g, int K, int cap, int *ids, float *l, float &lend, bool &by_range)
{
    const int lane = lane_id();
    const int NI = K + 1;  // intervals k = -1 .. K-1
    const int q = (NI + 31) >> 5;
    const int k0 = -1 + lane * q;
    const int k1 = min(K - 1, k0 + q - 1);
    int cnt = 0, ties = 0;
    bool ended = false, rng = false;
    float endl = 0.0f;
    // minor crossings before each lane's first interval: lane L's block ends where lane L + 1's
    // begins, so one count per lane (at the end of its block) serves both
    const int iend = k0 <= k1 ? minor_before(g, k1 + 1) : 0;
    int i0 = __shfl_up_sync(kFull, iend, 1);
    if (lane == 0) i0 = 0;  // k0 = -1: no minor crossing before the start
    int pred = 0;
    if (k0 <= k1) pred = (k1 - k0 + 1) + iend - i0;
    const int pinc = warp_incl_add_int(pred);
    // a lane writes at most its predicted count from its offset, so every index stays below the
    // predicted total: within cap, the writes need no check
    const bool fits = __shfl_sync(kFull, pinc, 31) <= cap;
    if (k0 <= k1) {
        if (fits)
            walk<true, false>(g, k0, k1, i0, pinc - pred, cap, ids, l, cnt, ties, ended, endl, rng);
        else
            walk<true, true>(g, k0, k1, i0, pinc - pred, cap, ids, l, cnt, ties, ended, endl, rng);
    }
    const unsigned eb = __ballot_sync(kFull, ended);
    const int first = eb ? __ffs(eb) - 1 : 31;
    lend = __shfl_sync(kFull, endl, first);
    const unsigned rb = __ballot_sync(kFull, rng);
    by_range = (rb >> first) & 1u;
    int n;
    if (__any_sync(kFull, lane < first && ties > 0)) {
        // offsets of lanes after a diagonal step were too large: count exactly, place the cells again
        const int c = lane <= first ? cnt : 0;
        const int inc = warp_incl_add_int(c);
        n = __shfl_sync(kFull, inc, 31);
        if (n > cap) return -1;
        __syncwarp();
        if (lane <= first && k0 <= k1) walk<true, false>(g, k0, k1, i0, inc - c, cap, ids, l, cnt, ties, ended, endl, rng);
    } else {
        // every lane before the first that ended walked its whole block without a diagonal step,
        // so its predicted count was exact: n = that lane's offset + its count
        n = __shfl_sync(kFull, pinc - pred + cnt, first);
        if (n > cap) return -1;
    }
    __syncwarp();
    return n;
}

// All 32 lanes call this. Writes ids[0..n-1] (cell y*W + x) and l[0..n] (entry distances, then
// the end distance) and returns n; returns -1 if the beam has more than cap cells. rend = R as
// float. *end_by_range (optional) = whether the beam ended at the range limit inside the grid (false
// when it left the grid first or crossed no cell).
static __device__ int dda_warp(int W, int H, int ox, int oy, int dx, int dy, long long rfix, float rend, int cap, int *ids,
                               float *l, bool *end_by_range = nullptr)
{
    if (end_by_range) *end_by_range = false;
    Geo g;
    int K;
    if (!beam_geo(W, H, ox, oy, dx, dy, rfix, rend, g, K)) return 0;
    float lend = 0.0f;
    bool by_range = false;
    int n = -1;
    Fixed f;
    if (fixed_setup(g, f) && fixed_cells(f, K) <= cap) {
        const int stepm = g.xmaj ? g.sm * g.W : g.sm;
        n = fixed_run<1>(g, f, K,
                         [&](const Interval(&v)[1]) {
                             if (v[0].ok1) {
                                 ids[v[0].pos] = v[0].id;
                                 l[v[0].pos] = v[0].lam1;
                             }
                             if (v[0].ok2) {
                                 ids[v[0].pos + 1] = v[0].id + stepm;
                                 l[v[0].pos + 1] = v[0].lam2;
                             }
                         },
                         lend, by_range);
        __syncwarp();
    }
    if (n < 0) n = dda_walk(g, K, cap, ids, l, lend, by_range);
    if (n < 0) return -1;
    if (end_by_range) *end_by_range = by_range;
    if (lane_id() == 0) l[n] = lend;
    __syncwarp();
    return n;
}

}  // namespace fsmi
