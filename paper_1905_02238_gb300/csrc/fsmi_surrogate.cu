// Learned surrogate of the 2D beam FSMI (not part of the paper): a 1D conv + MLP that predicts a
// beam's mutual information from its occupancy profile, trained on beams that exact FSMI labels,
// used to prescreen candidate poses before exact FSMI reranks the best of them.
//
//   input  x[256][2]: sample i of the beam at distance i + 1/2 cells; (o, 1) inside the map, (0, 0)
//          beyond it
//   conv1  2 -> 32, kernel 3, stride 2, zero padding 1, ReLU        256 -> 128 positions
//   conv2  32 -> 32, same                                           128 -> 64
//   conv3  32 -> 32, same                                           64 -> 32
//   fc1    1024 -> 256 (input index t * 32 + c), ReLU;  fc2 256 -> 1
//   conv:  z[t][c] = b[c] + sum_{k<3} sum_ci W[c][k][ci] a[2t + k - 1][ci]
//
// Parameters are one flat FP32 vector (master copy, layout below); the weights are used as a BF16
// copy of the same vector, accumulation is FP32. Training keeps FP32 activations and splits them into
// BF16 terms for the tensor cores; every sum is taken in a fixed order, so a training step gives
// the same floats on every run.
#include <cuda.h>  // CUtensorMap and its enums (the encoder is fetched through the runtime, no -lcuda)
#include <cuda_bf16.h>
#include <cudaTypedefs.h>
#include <float.h>

#include <algorithm>

#include <mutex>

#include "../../include/fsmi.h"
#include "fsmi_device.cuh"
#include "fsmi_internal.h"

namespace fsmi {

namespace {

constexpr int kL = 256, kCin = 2, kCh = 32, kK = 3, kHid = 256, kFlat = kCh * (kL / 8);
// flat parameter layout
constexpr int oW1 = 0, oB1 = oW1 + kCh * kK * kCin, oW2 = oB1 + kCh, oB2 = oW2 + kCh * kK * kCh, oW3 = oB2 + kCh,
              oB3 = oW3 + kCh * kK * kCh, oW4 = oB3 + kCh, oB4 = oW4 + kHid * kFlat, oW5 = oB4 + kHid,
              oB5 = oW5 + kHid, kNParams = oB5 + 1;
static_assert(kNParams == FSMI_SURR_NPARAMS, "parameter layout");

using bf16 = __nv_bfloat16;

__device__ __forceinline__ float bf(const bf16 *p, long long i) { return __bfloat162float(p[i]); }

// ---- profiles ---------------------------------------------------------------------------------

// Sample i of a beam: the cell holding o + (i + 1/2) d, the floor of the Q31 position
// (o << 15) + (2i + 1) d (d the Q30 beam direction).
// sample i (of the first `keep`; later ones read as outside the map)
__device__ __forceinline__ void sample_2d(const float *map, int W, int H, long long ox, long long oy, int dx, int dy,
                                          int i, int keep, float &o, float &in)
{
    const long long px = ((ox << 15) + (long long)(2 * i + 1) * dx) >> 31;
    const long long py = ((oy << 15) + (long long)(2 * i + 1) * dy) >> 31;
    const bool inside = i < keep && px >= 0 && px < W && py >= 0 && py < H;
    o = inside ? __ldg(map + py * W + px) : 0.0f;
    in = inside ? 1.0f : 0.0f;
}

__device__ __forceinline__ void beam_dir_2d(const int32_t *pose, const int32_t *u, int &dx, int &dy)
{
    const long long c = pose[2], s = pose[3], ux = u[0], uy = u[1];
    dx = (int)((c * ux - s * uy + (1LL << 29)) >> 30);
    dy = (int)((s * ux + c * uy + (1LL << 29)) >> 30);
}

// one warp per beam: out[n][i] = (o, inside) as BF16 pairs
__global__ void __launch_bounds__(256)
    k_profiles(const float *__restrict__ map, int W, int H, const int32_t *__restrict__ poses,
               const int32_t *__restrict__ dirs, int B, int keep, long long nbeams,
               const int32_t *__restrict__ beam_ids, long long N, __nv_bfloat162 *__restrict__ out, int *status)
{
    const int lane = lane_id();
    const long long wpb = blockDim.x >> 5;
    for (long long n = blockIdx.x * wpb + (threadIdx.x >> 5); n < N; n += (long long)gridDim.x * wpb) {
        const long long id = beam_ids ? (long long)__ldg(beam_ids + n) : n;
        if (id < 0 || id >= nbeams) {  // no such beam: an empty profile
            for (int i = lane; i < kL; i += 32) out[n * kL + i] = __floats2bfloat162_rn(0.0f, 0.0f);
            if (lane == 0) set_status(status, FSMI_STATUS_BAD_BEAM);
            continue;
        }
        const int32_t *pose = poses + 4 * (id / B);
        int dx, dy;
        beam_dir_2d(pose, dirs + 2 * (id % B), dx, dy);
        for (int i = lane; i < kL; i += 32) {
            float o, in;
            sample_2d(map, W, H, pose[0], pose[1], dx, dy, i, keep, o, in);
            out[n * kL + i] = __floats2bfloat162_rn(o, in);
        }
    }
}

int grid_cap(long long want)
{
    const long long cap = (long long)sm_count() * 32;
    return (int)(want < 1 ? 1 : (want > cap ? cap : want));
}

__device__ __forceinline__ float relu(float v) { return v > 0.0f ? v : 0.0f; }

// ---- Adam --------------------------------------------------------------------------------------

// Adam (Kingma and Ba, Algorithm 1) with bias correction; also refreshes the BF16 copy.
__global__ void k_adam(float *__restrict__ p, float *__restrict__ m, float *__restrict__ v, const float *__restrict__ g,
                       long long n, float lr, float b1, float b2, float eps, float c1, float c2, bf16 *__restrict__ wb)
{
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.0f - b1) * gi;
        const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        p[i] = pi;
        wb[i] = __float2bfloat16_rn(pi);
    }
}

__global__ void k_cast(const float *__restrict__ p, long long n, bf16 *__restrict__ wb)
{
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        wb[i] = __float2bfloat16_rn(p[i]);
}

// ---- inference on the tensor cores (mma.sync m16n8k16, BF16 operands, FP32 accumulation) --------

__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void ldsm_x4(unsigned addr, unsigned &r0, unsigned &r1, unsigned &r2, unsigned &r3)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}

__device__ __forceinline__ void mma_bf16(float (&c)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0,
                                         unsigned b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ unsigned pack_bf16x2(float lo, float hi)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const unsigned *>(&v);
}


__device__ __forceinline__ void mma_bf16_k8(float (&c)[4], unsigned a0, unsigned a1, unsigned b0)
{
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a0), "r"(a1), "r"(b0));
}

constexpr int kS2 = 104;  // W2 / W3 row stride (bf16): 208 B, eight rows in eight bank groups

// Weight fragments of k-step ks (16 of the K = 96 inputs) of a conv layer for the four n8 tiles
__device__ __forceinline__ void load_wfrag(const bf16 *Wt, int ks, unsigned (&bw)[4][2])
{
    const int lane = lane_id();
#pragma unroll
    for (int np = 0; np < 2; ++np) {
        const int row = np * 16 + (lane & 7) + 8 * (lane >> 4);
        ldsm_x4(smem_u32(Wt + row * kS2 + ks * 16 + 8 * ((lane >> 3) & 1)), bw[2 * np][0], bw[2 * np][1],
                bw[2 * np + 1][0], bw[2 * np + 1][1]);
    }
}

// ---- training ---------------------------------------------------------------------------------------
//
// Activations (FP32, pre-ReLU) per batch of N beams: z1 [N][128][32], z2 [N][64][32], z3 [N][32][32],
// z4 [N][256]. All products run on the tensor cores (mma.sync m16n8k16, BF16 operands, FP32
// accumulation) with each FP32 operand split into BF16 terms, a_1 = bf16(a), a_2 = bf16(a - a_1),
// a_3 = bf16(a - a_1 - a_2), whose sum is a (1 + d) with |d| <= 2^-18 for two terms and 2^-27 for three
// (the split-BF16 products of Henry, Tang and Heinecke, "Leveraging the bfloat16 artificial
// intelligence datatype for higher-precision computations", 2019). The forward pass, whose outputs feed
// the loss and its derivative, takes three terms (weights are exact in one); the data gradients and
// fc1's weight gradient take two, A_1 B_1 + A_2 B_1 + A_1 B_2 where both operands are FP32 (the A_2 B_2 term is
// below 2^-18 of the product); the convolutions' weight gradients take three and all products above 2^-26, as
// accurate as FP32 multiply-adds (strip_outer).
//
// The convolutions work on strips of 16 output positions per warp whose MMA fragments are formed in
// registers: nothing is staged, and the im2col matrix exists nowhere. A step of 4096 beams with its sampling
// takes 268 us; 754 us with every layer an index-function GEMM (operands gathered element by element through
// shared memory) and the reductions in 21 launches.

// (v.x, v.y) as T BF16 pairs
template <int T>
__device__ __forceinline__ void split(float2 v, unsigned (&t)[T])
{
#pragma unroll
    for (int i = 0; i < T; ++i) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(v.x, v.y);
        t[i] = *reinterpret_cast<const unsigned *>(&h);
        v.x -= __low2float(h);
        v.y -= __high2float(h);
    }
}

// Channels and fragment columns: column s = 8 nt + 2w + e of an MMA tile holds channel 16 (nt / 2) + 4w +
// 2 (nt % 2) + e, so that lane w's pairs of the tiles 0, 1 and 2, 3 are 4 consecutive channels each and a
// warp's 16-byte access covers whole sectors, 64 bytes of each of 8 rows. (With the columns' own order an
// access is 8 bytes per lane and meets 8 lines for 256 bytes; the L1 wavefronts of that bound these kernels.)
// The weights are staged in the same order; as a sum over channels runs over all columns, nothing else changes.
__device__ __forceinline__ int chan(int s) { return 16 * (s >> 4) + 4 * ((s >> 1) & 3) + 2 * ((s >> 3) & 1) + (s & 1); }

// channels 0 .. 3 and 16 .. 19 from p as the pairs of the four n8 tiles
__device__ __forceinline__ void load8(const float *p, float2 (&v)[4])
{
    const float4 a = *reinterpret_cast<const float4 *>(p), b = *reinterpret_cast<const float4 *>(p + 16);
    v[0] = make_float2(a.x, a.y);
    v[1] = make_float2(a.z, a.w);
    v[2] = make_float2(b.x, b.y);
    v[3] = make_float2(b.z, b.w);
}

__device__ __forceinline__ float2 relu2(float2 v) { return make_float2(relu(v.x), relu(v.y)); }
__device__ __forceinline__ float2 ld2(const float *p) { return *reinterpret_cast<const float2 *>(p); }

// relu(acc + b) of a strip as three BF16 terms P[nt][h] (row g + 8 h); acc + b goes to out (row g of the
// strip, channel 4w; `step` floats between the strip's rows). bs: the layer's biases from channel 4w on
__device__ __forceinline__ void store_split(const float (&acc)[4][4], const float *bs, float *out, int step,
                                            unsigned (&P)[4][2][3])
{
    float2 b[4];
    load8(bs, b);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        float2 z[4];
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            z[nt] = make_float2(acc[nt][2 * e] + b[nt].x, acc[nt][2 * e + 1] + b[nt].y);
            split<3>(relu2(z[nt]), P[nt][e]);
        }
        float4 *o = reinterpret_cast<float4 *>(out + 8 * e * step);
        o[0] = make_float4(z[0].x, z[0].y, z[1].x, z[1].y);
        o[4] = make_float4(z[2].x, z[2].y, z[3].x, z[3].y);
    }
}

// the strip one row down, as shift_rows of the inference kernel, for each term
__device__ __forceinline__ void shift_terms(const unsigned (&P)[4][2][3], unsigned (&carry)[4][3], unsigned (&S)[4][2][3])
{
    const int lane = lane_id();
    const bool first = lane < 4;
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const unsigned lo = __shfl_sync(kFull, P[nt][0][i], lane + 28), hi = __shfl_sync(kFull, P[nt][1][i], lane + 28);
            S[nt][0][i] = first ? carry[nt][i] : lo;
            S[nt][1][i] = first ? lo : hi;
            carry[nt][i] = hi;
        }
}

// acc += strip P (tap `tap`) of a K = 96 layer
__device__ __forceinline__ void tap_mma3(float (&acc)[4][4], const unsigned (&P)[4][2][3], const bf16 *sW, int tap)
{
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
        unsigned bw[4][2];
        load_wfrag(sW, 2 * tap + hh, bw);
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int nt = 0; nt < 4; ++nt)
                mma_bf16(acc[nt], P[2 * hh][0][i], P[2 * hh][1][i], P[2 * hh + 1][0][i], P[2 * hh + 1][1][i], bw[nt][0],
                         bw[nt][1]);
    }
}

// The three convolutions of a batch, one warp per beam: the inference kernel's strips of equal residues (conv1 at
// 4u + r, conv2 at 2u and 2u + 1, conv3 at u; see k_conv_infer) with three terms per activation, every layer's
// pre-activations written once and read by nobody here; h receives relu(z3) as three BF16 terms,
// hstride elements apart (fc1's operand). A batch of 4096 writes 142 MB in 46 us (21 us at the copy
// rate); 12 warps per SM at 168 registers leave the MMA chains' latency in sight. Layer by layer, each reading
// the one before: 85 us; as index-function GEMMs 198 us.
constexpr int kFwdWarps = 4;
__global__ void __launch_bounds__(kFwdWarps * 32, 3)
    k_convs_fwd(int N, const unsigned *__restrict__ x, const bf16 *__restrict__ w, const float *__restrict__ params,
                float *__restrict__ z1, float *__restrict__ z2, float *__restrict__ z3, bf16 *__restrict__ h, size_t hstride)
{
    launch_dependents();
    __shared__ __align__(16) bf16 sW1[kCh * 8];
    __shared__ __align__(16) bf16 sW2[kCh * kS2];
    __shared__ __align__(16) bf16 sW3[kCh * kS2];
    __shared__ __align__(16) float sb[3 * kCh];
    for (int e = threadIdx.x; e < 3 * kCh; e += kFwdWarps * 32)
        sb[e] = params[(e < kCh ? oB1 : e < 2 * kCh ? oB2 : oB3) + e % kCh];
    for (int e = threadIdx.x; e < kCh * 8; e += kFwdWarps * 32)
        sW1[e] = e % 8 < kK * kCin ? w[oW1 + chan(e / 8) * kK * kCin + e % 8] : __float2bfloat16_rn(0.0f);
    for (int e = threadIdx.x; e < kCh * kS2; e += kFwdWarps * 32) {
        const int kk = e % kS2, at = chan(e / kS2) * kK * kCh + (kk & ~31) + chan(kk & 31);
        sW2[e] = kk < kK * kCh ? w[oW2 + at] : __float2bfloat16_rn(0.0f);
        sW3[e] = kk < kK * kCh ? w[oW3 + at] : __float2bfloat16_rn(0.0f);
    }
    __syncthreads();
    const int lane = lane_id(), g = lane >> 2, wq = lane & 3;
    const float *b1 = sb + 4 * wq, *b2 = b1 + kCh, *b3 = b2 + kCh;
    unsigned bw1[4];
    ldsm_x4(smem_u32(sW1 + lane * 8), bw1[0], bw1[1], bw1[2], bw1[3]);
    for (int n = blockIdx.x * kFwdWarps + (threadIdx.x >> 5); n < N; n += gridDim.x * kFwdWarps) {
        const unsigned *xr = x + (size_t)n * kL;
        unsigned carry1[4][3] = {}, carry2[4][3] = {};
#pragma unroll 1
        for (int s = 0; s < 2; ++s) {  // u = 16 s + row
            const int u = 16 * s + g;
            auto conv1 = [&](int r, unsigned(&P)[4][2][3]) {  // positions 4u + r
                const int i = 8 * u + 2 * r - 1 + wq;
                const unsigned a0 = wq < 3 && i >= 0 ? __ldg(xr + i) : 0u, a1 = wq < 3 ? __ldg(xr + i + 64) : 0u;
                float acc[4][4] = {};
#pragma unroll
                for (int nt = 0; nt < 4; ++nt) mma_bf16_k8(acc[nt], a0, a1, bw1[nt]);
                store_split(acc, b1, z1 + ((size_t)n * 128 + 4 * u + r) * kCh + 4 * wq, 4 * kCh, P);
            };
            float ev[4][4] = {}, od[4][4] = {}, acc[4][4] = {};
            unsigned P1[4][2][3], P3[4][2][3], Q[4][2][3];
            conv1(3, P3);
            shift_terms(P3, carry1, Q);
            conv1(1, P1);
            tap_mma3(ev, Q, sW2, 0);
            tap_mma3(od, P1, sW2, 0);
            conv1(0, Q);
            tap_mma3(ev, Q, sW2, 1);
            conv1(2, Q);
            tap_mma3(od, Q, sW2, 1);
            tap_mma3(ev, P1, sW2, 2);
            tap_mma3(od, P3, sW2, 2);
            store_split(ev, b2, z2 + ((size_t)n * 64 + 2 * u) * kCh + 4 * wq, 2 * kCh, P1);
            store_split(od, b2, z2 + ((size_t)n * 64 + 2 * u + 1) * kCh + 4 * wq, 2 * kCh, P3);
            shift_terms(P3, carry2, Q);
            tap_mma3(acc, Q, sW3, 0);
            tap_mma3(acc, P1, sW3, 1);
            tap_mma3(acc, P3, sW3, 2);
            const size_t o = ((size_t)n * 32 + u) * kCh + 4 * wq;
            store_split(acc, b3, z3 + o, kCh, Q);
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    uint2 *d = reinterpret_cast<uint2 *>(h + i * hstride + o + 8 * e * kCh);
                    d[0] = make_uint2(Q[0][e][i], Q[1][e][i]);
                    d[4] = make_uint2(Q[2][e][i], Q[3][e][i]);
                }
        }
    }
}

// ---- fc1's three products ---------------------------------------------------------------------------
//
// C[m][n] = sum over the term products of sum_k A_i(m, k) B_j(k, n), with the operands' BF16 terms in
// memory (written by their producers), `ta` / `tb` elements apart: TA terms of A, TB of B, the products
// (i, 0) and, with TB = 2, (0, 1). AT / BT: the operand is stored with k along the rows (A [k][m],
// B [k][n]), else along the columns (A [m][k], B [n][k]). Blocks of 128 x 64 outputs, 8 warps of
// 32 x 32; K in stages of 32 through a 3-stage cp.async ring, 16-byte chunks XOR-swizzled so that
// ldmatrix (.trans for k-row storage) meets every bank once. Block z takes k in [z kper, (z + 1) kper).
// Rows past M and k past K read as zero; lda, ldb and the starts are multiples of 8 elements, N of 64.
//
// A batch of 4096: 26 us forward (three products, 6.4 GFLOP of MMAs each here and in the weight gradient, the
// tensor pipe 55 % busy), 24 us weight gradient, 28 us data gradient; 79, 83 and 75 us when the blocks
// gathered and split FP32 operands element by element.
constexpr int kGmM = 128, kGmN = 64, kGmK = 32, kGmStages = 3;
template <int TA, int TB>
constexpr int kGmSmem = kGmStages * (TA * kGmM + TB * kGmN) * kGmK * 2;

__device__ __forceinline__ void cp_async16(unsigned dst, const void *src, bool ok)
{
    const int bytes = ok ? 16 : 0;  // 0: the 16 bytes are zero-filled and src is not read
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

__device__ __forceinline__ void ldsm_x4t(unsigned addr, unsigned &r0, unsigned &r1, unsigned &r2, unsigned &r3)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}

// one operand's tile of a stage: R rows (of m or n) x 32 k into shared memory at s
template <int R, bool T>
__device__ __forceinline__ void stage_tile(unsigned s, const bf16 *src, int ld, int r0, int rmax, int k0, int kend)
{
#pragma unroll
    for (int c = threadIdx.x; c < R * 4; c += 256) {
        if (T) {  // [k][row]: R / 8 chunks per k
            const int k = c / (R / 8), q = c % (R / 8);
            const bool ok = k0 + k < kend && r0 + 8 * q < rmax;
            cp_async16(s + k * R * 2 + ((q ^ (k & 7)) << 4), ok ? src + (size_t)(k0 + k) * ld + r0 + 8 * q : src, ok);
        } else {  // [row][k]: 4 chunks per row
            const int r = c >> 2, q = c & 3;
            const bool ok = r0 + r < rmax && k0 + 8 * q < kend;
            cp_async16(s + r * 64 + ((q ^ ((r >> 1) & 3)) << 4), ok ? src + (size_t)(r0 + r) * ld + k0 + 8 * q : src, ok);
        }
    }
}

// address of the 16-byte chunk holding rows r .. r + 7 (T) or row r (else) at k (T) or k .. k + 7
template <int R, bool T>
__device__ __forceinline__ unsigned tile_at(unsigned s, int r, int k)
{
    return T ? s + k * R * 2 + (((r >> 3) ^ (k & 7)) << 4) : s + r * 64 + (((k >> 3) ^ ((r >> 1) & 3)) << 4);
}

template <int TA, int TB, bool AT, bool BT, class FE>
__global__ void __launch_bounds__(256, 2)
    k_gemm_terms(int M, int N, int K, int kper, const bf16 *__restrict__ A, size_t ta, int lda, const bf16 *__restrict__ B,
                 size_t tb, int ldb, FE fe, bool beside)
{
    const EndAfterPrevious end{beside && blockIdx.x + blockIdx.y + blockIdx.z == 0};
    if (!beside) wait_previous();
    launch_dependents();
    extern __shared__ __align__(128) unsigned char gsm[];
    constexpr int kA = kGmM * kGmK * 2, kB = kGmN * kGmK * 2, kStage = TA * kA + TB * kB;
    const unsigned s0 = smem_u32(gsm);
    const int lane = lane_id(), w = threadIdx.x >> 5, wm = (w >> 1) * 32, wn = (w & 1) * 32;
    const int m0 = blockIdx.y * kGmM, n0 = blockIdx.x * kGmN;
    const int kbeg = blockIdx.z * kper, kend = min(K, kbeg + kper);
    const int steps = kend > kbeg ? (kend - kbeg + kGmK - 1) / kGmK : 0;
    auto fill = [&](int step) {
        if (step < steps) {
            const unsigned s = s0 + (step % kGmStages) * kStage;
            const int k0 = kbeg + step * kGmK;
#pragma unroll
            for (int i = 0; i < TA; ++i) stage_tile<kGmM, AT>(s + i * kA, A + i * ta, lda, m0, M, k0, kend);
#pragma unroll
            for (int i = 0; i < TB; ++i) stage_tile<kGmN, BT>(s + TA * kA + i * kB, B + i * tb, ldb, n0, N, k0, kend);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float acc[2][4][4] = {};
#pragma unroll
    for (int i = 0; i < kGmStages - 1; ++i) fill(i);
    for (int step = 0; step < steps; ++step) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kGmStages - 2) : "memory");
        __syncthreads();  // the stage has landed for all, and the one filled next is no longer read
        fill(step + kGmStages - 1);
        const unsigned s = s0 + (step % kGmStages) * kStage, sb = s + TA * kA;
#pragma unroll
        for (int ks = 0; ks < kGmK; ks += 16) {
            unsigned a[TA][2][4], b[TB][4][2];
#pragma unroll
            for (int i = 0; i < TA; ++i)
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) {
                    const int m = wm + 16 * mt;
                    if (AT)
                        ldsm_x4t(tile_at<kGmM, true>(s + i * kA, m + 8 * ((lane >> 3) & 1), ks + (lane & 7) + 8 * (lane >> 4)),
                                 a[i][mt][0], a[i][mt][1], a[i][mt][2], a[i][mt][3]);
                    else
                        ldsm_x4(tile_at<kGmM, false>(s + i * kA, m + (lane & 15), ks + 8 * (lane >> 4)), a[i][mt][0],
                                a[i][mt][1], a[i][mt][2], a[i][mt][3]);
                }
#pragma unroll
            for (int i = 0; i < TB; ++i)
#pragma unroll
                for (int np = 0; np < 2; ++np) {
                    const int n = wn + 16 * np;
                    if (BT)
                        ldsm_x4t(tile_at<kGmN, true>(sb + i * kB, n + 8 * (lane >> 4), ks + (lane & 7) + 8 * ((lane >> 3) & 1)),
                                 b[i][2 * np][0], b[i][2 * np][1], b[i][2 * np + 1][0], b[i][2 * np + 1][1]);
                    else
                        ldsm_x4(tile_at<kGmN, false>(sb + i * kB, n + (lane & 7) + 8 * (lane >> 4), ks + 8 * ((lane >> 3) & 1)),
                                b[i][2 * np][0], b[i][2 * np][1], b[i][2 * np + 1][0], b[i][2 * np + 1][1]);
                }
#pragma unroll
            for (int i = 0; i < TA + TB - 1; ++i)  // the products (i, 0), then (0, 1)
#pragma unroll
                for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                    for (int nt = 0; nt < 4; ++nt) {
                        const unsigned(&x)[4] = a[i < TA ? i : 0][mt];
                        const unsigned(&y)[2] = b[i < TA ? 0 : TB - 1][nt];
                        mma_bf16(acc[mt][nt], x[0], x[1], x[2], x[3], y[0], y[1]);
                    }
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int m = m0 + wm + 16 * mt + (lane >> 2) + 8 * e, n = n0 + wn + 8 * nt + 2 * (lane & 3);
                if (m < M) fe(m, n, make_float2(acc[mt][nt][2 * e], acc[mt][nt][2 * e + 1]));
            }
}

struct StorePart {  // part[z][m][n] = acc
    float *part;
    int rows, ld;
    __device__ void operator()(int m, int n, float2 v) const
    {
        *reinterpret_cast<float2 *>(part + ((size_t)blockIdx.z * rows + m) * ld + n) = v;
    }
};
struct StoreMask {  // out[m][n] = acc [mask[m][n] > 0]
    float *out;
    const float *mask;
    int ld;
    __device__ void operator()(int m, int n, float2 v) const
    {
        const size_t i = (size_t)m * ld + n;
        const float2 k = ld2(mask + i);
        *reinterpret_cast<float2 *>(out + i) = make_float2(k.x > 0.0f ? v.x : 0.0f, k.y > 0.0f ? v.y : 0.0f);
    }
};

// Splits of K in fc1's forward product, for two 64-row by 64-column tiles per SM at least and 256 of K per split: 2
// for a batch of 4096, whose 256 blocks of 128 x 64 run in one wave. Each sum's value depends on the split (the
// tensor cores' accumulators round toward zero), so this rule is part of the results: a sum next to
// zero decides whether a hidden unit's gradient counts.
constexpr int kFc1Splits = 4;  // at most
int fc1_forward_splits(int N)
{
    const long long tiles = (long long)(N + 63) / 64 * (kHid / 64);
    int splits = 1;
    while (splits < kFc1Splits && tiles * splits < 2LL * sm_count()) splits *= 2;
    return splits;
}

// splits of the batch in fc1's weight gradient (32 output blocks): a function of N alone, so that a step's
// sums are in the same order on every run
int fc1_splits(int N) { return std::max(1, std::min(8, (N + 255) / 256)); }

template <int TA, int TB, bool AT, bool BT, class FE>
cudaError_t gemm_terms(int M, int N, int K, int splits, const bf16 *A, size_t ta, int lda, const bf16 *B, size_t tb, int ldb,
                       FE fe, bool beside, cudaStream_t s)
{
    auto kern = k_gemm_terms<TA, TB, AT, BT, FE>;
    const int smem = kGmSmem<TA, TB>;
    int occ = 0;
    cudaError_t e = resident_blocks((const void *)kern, 256, smem, occ);
    if (e != cudaSuccess) return e;
    const int kper = ((K + splits - 1) / splits + kGmK - 1) / kGmK * kGmK;
    return launch_kernel(true, kern, dim3(N / kGmN, (M + kGmM - 1) / kGmM, splits), 256, smem, s, M, N, K, kper, A, ta, lda,
                         B, tb, ldb, fe, beside);
}

// out[e] = sum over z of part[z][e], in order
__global__ void k_split_reduce(int E, int splits, const float *__restrict__ part, float *__restrict__ out)
{
    const EndAfterPrevious end{blockIdx.x == 0};
    launch_dependents();
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < E; e += gridDim.x * blockDim.x) {
        float v = 0.0f;
        for (int z = 0; z < splits; ++z) v += part[(size_t)z * E + e];
        out[e] = v;
    }
}

// ---- head -------------------------------------------------------------------------------------------
//
// z4[n][j] = b4[j] + the sums of fc1's product over the splits of K (part1 [splits][N][256]),
// pred[n] = b5 + sum_j W5[j] relu(z4[n][j]) and, with targets, d = pred - y, dpred = 2 d / N,
// dz4[n][j] = dpred W5[j] [z4 > 0] as two BF16 terms (dz, N * 256 elements apart) and the block's sums over its
// rows of dpred relu(z4) (gW5), dz4 (gb4), dpred (gb5) and d^2 (loss) into part[block][514]. A
// warp takes 4 consecutive rows, a lane the columns 4 lane + k and 128 + 4 lane + k.
constexpr int kHeadRows = 32, kHeadOut = 2 * kHid + 2;
__global__ void __launch_bounds__(256)
    k_head(const float *__restrict__ part1, const bf16 *__restrict__ w, const float *__restrict__ params,
           const float *__restrict__ y, int N, float *__restrict__ z4, float *__restrict__ pred, bf16 *__restrict__ dz,
           float *__restrict__ part, int splits)
{
    wait_previous();
    launch_dependents();
    __shared__ float sum[8][kHeadOut];
    const int lane = lane_id(), wp = threadIdx.x >> 5;
    float w5[8], b4[8], g5[8] = {}, g4[8] = {}, gb = 0.0f, loss = 0.0f;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        w5[k] = bf(w, oW5 + 128 * (k >> 2) + 4 * lane + (k & 3));
        b4[k] = params[oB4 + 128 * (k >> 2) + 4 * lane + (k & 3)];
    }
    const float b5 = params[oB5];
    for (int r = 0; r < kHeadRows / 8; ++r) {
        const int n = blockIdx.x * kHeadRows + wp * (kHeadRows / 8) + r;
        if (n >= N) break;
        float z[8];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const size_t o = (size_t)n * kHid + 128 * q + 4 * lane;
            float4 v[kFc1Splits];
#pragma unroll
            for (int k = 0; k < kFc1Splits; ++k)
                if (k < splits) v[k] = *reinterpret_cast<const float4 *>(part1 + (size_t)k * N * kHid + o);
#pragma unroll
            for (int k = 1; k < kFc1Splits; ++k)
                if (k < splits) v[0] = make_float4(v[0].x + v[k].x, v[0].y + v[k].y, v[0].z + v[k].z, v[0].w + v[k].w);
            z[4 * q] = v[0].x + b4[4 * q];
            z[4 * q + 1] = v[0].y + b4[4 * q + 1];
            z[4 * q + 2] = v[0].z + b4[4 * q + 2];
            z[4 * q + 3] = v[0].w + b4[4 * q + 3];
            *reinterpret_cast<float4 *>(z4 + o) = make_float4(z[4 * q], z[4 * q + 1], z[4 * q + 2], z[4 * q + 3]);
        }
        float a = 0.0f;
#pragma unroll
        for (int k = 0; k < 8; ++k) a = fmaf(w5[k], relu(z[k]), a);
        a = warp_sum(a) + b5;
        if (lane == 0) pred[n] = a;
        if (y) {
            const float d = a - y[n], dp = 2.0f * d / (float)N;
            loss = fmaf(d, d, loss);
            gb += dp;
            float v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                v[k] = z[k] > 0.0f ? dp * w5[k] : 0.0f;
                g4[k] += v[k];
                g5[k] = fmaf(dp, relu(z[k]), g5[k]);
            }
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                unsigned t0[2], t1[2];
                split<2>(make_float2(v[4 * q], v[4 * q + 1]), t0);
                split<2>(make_float2(v[4 * q + 2], v[4 * q + 3]), t1);
                const size_t o = (size_t)n * kHid + 128 * q + 4 * lane;
                *reinterpret_cast<uint2 *>(dz + o) = make_uint2(t0[0], t1[0]);
                *reinterpret_cast<uint2 *>(dz + (size_t)N * kHid + o) = make_uint2(t0[1], t1[1]);
            }
        }
    }
    if (!y) return;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int j = 128 * (k >> 2) + 4 * lane + (k & 3);
        sum[wp][j] = g5[k];
        sum[wp][kHid + j] = g4[k];
    }
    if (lane == 0) {
        sum[wp][2 * kHid] = gb;
        sum[wp][2 * kHid + 1] = loss;
    }
    __syncthreads();
    for (int j = threadIdx.x; j < kHeadOut; j += 256) {
        float t = 0.0f;
#pragma unroll
        for (int k = 0; k < 8; ++k) t += sum[k][j];
        part[(size_t)blockIdx.x * kHeadOut + j] = t;
    }
}

// ---- the convolutions' backward pass ----------------------------------------------------------------
//
// One pass per 32 -> 32 conv layer over its dz [N][Lout][32] (Lout = Lin / 2), two warps per strip of 16
// positions t, each for 16 of the channels of the layer below:
//   data gradient: an even input position 2t takes tap 1 at t, an odd one 2t + 1 taps 0 at t + 1 and 2
//     at t, so the strip and the strip one row on, as A operands, give the strips of positions 2t and
//     2t + 1 (K = 32 and 64, no zero taps), masked by the layer below's ReLU;
//   weight gradient: gW[c][k][ci] = sum over t of dz[t][c] relu(z)[2t + k - 1][ci], an MMA with the
//     strip's 16 positions as K. Both operands are the fragments at hand transposed (movmatrix), and
//     the 32 x 96 sums stay in registers over all of a warp's strips;
//   bias gradient: the column sums of dz.
// LAST (conv2): conv1's gradients follow at once from the strips of dz1, which is never stored.
// The grid, the strips of each warp and the order of the sums depend only on N: the blocks' sums go to
// part[block][...] and are added in block order (k_grads), so a step gives the same floats on every run.
// The sums take 52 registers per lane, and two blocks of 8 warps per SM do not hide the strips' loads; the
// next strip's rows are prefetched toward L1. A batch of 4096: 38 us (conv3) and 85 us (conv2 and conv1); with the
// weight gradients from two terms per operand 33 and 66 us, but up to 2.5 times as far from 64 bits. Blocks
// of 6 warps with 168 registers instead of 128 (56 bytes spilled instead of 224): the same time. In the two-term form one
// warp per strip with all 32 channels took 38 and 77 us against 34 and 68; the separate data, weight and bias
// gradient kernels 320 us.
constexpr int kBwdWarps = 8, kBwdBlocks = 304;
constexpr int kTrPitch = kCh + 8;  // row pitch of the staged weights: 80 B, eight rows in eight bank groups
template <bool LAST>
constexpr int kBwdOut = kCh * kK * kCh + kCh + (LAST ? kCh * kK * kCin + kCh : 0);

__device__ __forceinline__ unsigned transpose8(unsigned v)
{
    unsigned r;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(v));
    return r;
}

// acc += (T_0 + T_1 + T_2)^T (U_0 + U_1 + U_2) without the products below 2^-26: T (32 columns) and U (tile nt's 8)
// strips of 16 positions as three BF16 terms, transposed (A fragments of the 32 rows c, B fragments of an n8
// tile). The strip's sum is formed by itself, from its smallest products on, and added in FP32: the tensor cores'
// accumulators round toward zero, and a sum kept in them over all strips would shrink.
__device__ __forceinline__ void strip_outer(float (&acc)[2][2][4], int nt, const unsigned (&T)[4][2][3], const unsigned (&U)[2][3])
{
    constexpr int kI[6] = {0, 2, 1, 0, 1, 0}, kJ[6] = {2, 0, 1, 1, 0, 0};
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) {
        float s[4] = {};
#pragma unroll
        for (int p = 0; p < 6; ++p) {
            const int i = kI[p], j = kJ[p];
            mma_bf16(s, T[2 * mt][0][i], T[2 * mt + 1][0][i], T[2 * mt][1][i], T[2 * mt + 1][1][i], U[0][j], U[1][j]);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[mt][nt][q] += s[q];
    }
}

template <bool LAST>
__global__ void __launch_bounds__(kBwdWarps * 32, 2)
    k_conv_bwd(int N, int Lin, const float *__restrict__ dz, const bf16 *__restrict__ w, const float *__restrict__ zprev,
               const bf16 *__restrict__ x, float *__restrict__ out, float *__restrict__ part)
{
    wait_previous();
    launch_dependents();
    constexpr int kO = kBwdOut<LAST>, kW = kCh * kK * kCh;
    __shared__ __align__(16) bf16 sW[kK * kCh * kTrPitch];  // [k][ci][c]
    __shared__ float sum[kO];
    for (int e = threadIdx.x; e < kK * kCh * kCh; e += kBwdWarps * 32) {
        const int k = e / (kCh * kCh), ci = (e / kCh) % kCh, c = e % kCh;
        sW[(k * kCh + ci) * kTrPitch + c] = w[(chan(c) * kK + k) * kCh + chan(ci)];
    }
    for (int e = threadIdx.x; e < kO; e += kBwdWarps * 32) sum[e] = 0.0f;
    __syncthreads();
    const int lane = lane_id(), g = lane >> 2, wq = lane & 3, wp = threadIdx.x >> 5;
    const int half = wp & 1, ch = 16 * half;  // this warp's columns of the layer below (channels 16 half + 4w .. + 3)
    const int Lout = Lin >> 1, tpb = Lout / 16;
    const long long units = (long long)N * tpb, np = (long long)gridDim.x * (kBwdWarps / 2),
                    me = (long long)blockIdx.x * (kBwdWarps / 2) + (wp >> 1);
    const int u0 = (int)(units * me / np), u1 = (int)(units * (me + 1) / np);  // (a strip's rows take 6 KB and more)
    float acc[3][2][2][4] = {}, acc1[4] = {};
    float2 gb[2] = {}, gb1[2] = {};
    for (int u = u0; u < u1; ++u) {
        const int n = u / tpb, t0 = u % tpb * 16;
        if (u + 1 < u1) {  // the next strip's rows, which follow this one's, toward L1
            const float *nd = dz + (size_t)(u + 1) * 16 * kCh, *nz = zprev + (size_t)(u + 1) * 32 * kCh;
            asm volatile("prefetch.global.L1 [%0];" ::"l"(lane < 16 ? nd + lane * kCh : nz + (lane - 16 + 16 * half) * kCh));
        }
        // weight gradient: three terms of dz's strip, transposed
        unsigned a[4][2][3];
        const float *dr = dz + ((size_t)n * Lout + t0 + g) * kCh + 4 * wq;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            float2 v[4];
            load8(dr + 8 * e * kCh, v);
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) split<3>(v[nt], a[nt][e]);
#pragma unroll
            for (int nt = 0; nt < 2; ++nt) {
                gb[nt].x += half ? v[nt + 2].x : v[nt].x;
                gb[nt].y += half ? v[nt + 2].y : v[nt].y;
            }
        }
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int i = 0; i < 3; ++i) a[nt][e][i] = transpose8(a[nt][e][i]);
        // the layer below at 2t + tap - 1, rows g and g + 8 of the strip: the other factor of the weight
        // gradient and (taps 1, 2) the mask of the data gradient at 2t and 2t + 1. Tap 0 is tap 2's strip one
        // row down, its first row from memory.
        unsigned p[2][2][3], mask = 0u;
        const size_t zo = ((size_t)n * Lin + 2 * (t0 + g)) * kCh + 16 * half + 4 * wq;
#pragma unroll
        for (int tap = 1; tap < 3; ++tap) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float4 z = *reinterpret_cast<const float4 *>(zprev + zo + (tap - 1 + 16 * e) * kCh);
                split<3>(relu2(make_float2(z.x, z.y)), p[0][e]);
                split<3>(relu2(make_float2(z.z, z.w)), p[1][e]);
                mask |= ((z.x > 0.0f) | (z.y > 0.0f) << 1 | (z.z > 0.0f) << 2 | (z.w > 0.0f) << 3) << (8 * (tap - 1) + 4 * e);
            }
#pragma unroll
            for (int nt = 0; nt < 2; ++nt) {
                unsigned q[2][3];
#pragma unroll
                for (int e = 0; e < 2; ++e)
#pragma unroll
                    for (int i = 0; i < 3; ++i) q[e][i] = transpose8(p[nt][e][i]);
                strip_outer(acc[tap], nt, a, q);
            }
        }
        {
            float4 z = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (g == 0 && t0 > 0) z = *reinterpret_cast<const float4 *>(zprev + zo - kCh);
#pragma unroll
            for (int nt = 0; nt < 2; ++nt) {
                unsigned first[3], q[2][3];
                split<3>(relu2(nt ? make_float2(z.z, z.w) : make_float2(z.x, z.y)), first);
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    const unsigned lo = __shfl_sync(kFull, p[nt][0][i], lane + 28), hi = __shfl_sync(kFull, p[nt][1][i], lane + 28);
                    q[0][i] = transpose8(g == 0 ? first[i] : lo);
                    q[1][i] = transpose8(g == 0 ? lo : hi);
                }
                strip_outer(acc[0], nt, a, q);
            }
        }
        // data gradient: two terms of dz at t (the first two, transposed back) and at t + 1, 16 channels at a time
        float ev[2][4] = {}, od[2][4] = {};
#pragma unroll
        for (int ks = 0; ks < 2; ++ks) {
            unsigned r[2][2][2], r1[2][2][2];
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int e = 0; e < 2; ++e)
#pragma unroll
                    for (int i = 0; i < 2; ++i) r[h][e][i] = transpose8(a[2 * ks + h][e][i]);
            {  // one row on: lane + 4's row, the last from memory (zero past the beam)
                float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (g == 7 && t0 + 16 < Lout) v = *reinterpret_cast<const float4 *>(dr + 9 * kCh + 16 * ks);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    unsigned t[2];
                    split<2>(h ? make_float2(v.z, v.w) : make_float2(v.x, v.y), t);
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const unsigned lo = __shfl_sync(kFull, r[h][0][i], lane + 4), hi = __shfl_sync(kFull, r[h][1][i], lane + 4);
                        r1[h][0][i] = g == 7 ? hi : lo;
                        r1[h][1][i] = g == 7 ? t[i] : hi;
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                unsigned bw[2][2];
                ldsm_x4(smem_u32(sW + (k * kCh + ch + (lane & 7) + 8 * (lane >> 4)) * kTrPitch + ks * 16 + 8 * ((lane >> 3) & 1)),
                        bw[0][0], bw[0][1], bw[1][0], bw[1][1]);
                float(&d)[2][4] = k == 1 ? ev : od;
                const unsigned(&s)[2][2][2] = k == 0 ? r1 : r;
#pragma unroll
                for (int q = 0; q < 2; ++q)
#pragma unroll
                    for (int i = 0; i < 2; ++i) mma_bf16(d[q], s[0][0][i], s[0][1][i], s[1][0][i], s[1][1][i], bw[q][0], bw[q][1]);
            }
        }
#pragma unroll
        for (int odd = 0; odd < 2; ++odd)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float(&d)[2][4] = odd ? od : ev;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    float &v = d[k >> 1][2 * e + (k & 1)];
                    v = mask >> (8 * odd + 4 * e + k) & 1u ? v : 0.0f;
                }
                if (!LAST)
                    *reinterpret_cast<float4 *>(out + zo + (odd + 16 * e) * kCh) =
                        make_float4(d[0][2 * e], d[0][2 * e + 1], d[1][2 * e], d[1][2 * e + 1]);
            }
        if (LAST) {
            // conv1: gW1[c][k][ci] = sum over positions p of dz1[p][c] x[2p + k - 1][ci], column 2k + ci of the
            // n8 tile (6 of 8 used; x is exact in BF16)
            const unsigned short *xr = reinterpret_cast<const unsigned short *>(x) + (size_t)n * kL * kCin;
            float sum1[4] = {};
#pragma unroll
            for (int odd = 0; odd < 2; ++odd) {  // p = 2t + odd
                float(&d)[2][4] = odd ? od : ev;
                unsigned t[2][2][3], bx[2];
#pragma unroll
                for (int nt = 0; nt < 2; ++nt) {
                    gb1[nt].x += d[nt][0] + d[nt][2];
                    gb1[nt].y += d[nt][1] + d[nt][3];
#pragma unroll
                    for (int e = 0; e < 2; ++e) split<3>(make_float2(d[nt][2 * e], d[nt][2 * e + 1]), t[nt][e]);
                }
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int i0 = 4 * (t0 + 2 * wq + 8 * e) + 2 * odd - 1 + (g >> 1);  // sample of row 2w; row 2w + 1: + 4
                    const unsigned lo = g < 6 && i0 >= 0 ? __ldg(xr + 2 * i0 + (g & 1)) : 0u;
                    const unsigned hi = g < 6 ? __ldg(xr + 2 * (i0 + 4) + (g & 1)) : 0u;
                    bx[e] = lo | hi << 16;
                }
#pragma unroll
                for (int i = 2; i >= 0; --i)
                    mma_bf16(sum1, transpose8(t[0][0][i]), transpose8(t[1][0][i]), transpose8(t[0][1][i]),
                             transpose8(t[1][1][i]), bx[0], bx[1]);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) acc1[q] += sum1[q];
        }
    }
    // the columns' sums over the eight row groups, then the block's sums, pair by pair of warps (the two of a
    // pair hold different outputs)
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
            gb[nt].x += __shfl_xor_sync(kFull, gb[nt].x, o);
            gb[nt].y += __shfl_xor_sync(kFull, gb[nt].y, o);
            if (LAST) {
                gb1[nt].x += __shfl_xor_sync(kFull, gb1[nt].x, o);
                gb1[nt].y += __shfl_xor_sync(kFull, gb1[nt].y, o);
            }
        }
    for (int k = 0; k < kBwdWarps / 2; ++k) {
        if ((wp >> 1) == k) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int row = g + 8 * (q >> 1), col = 2 * wq + (q & 1);
#pragma unroll
                for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                    for (int tap = 0; tap < 3; ++tap)
#pragma unroll
                        for (int nt = 0; nt < 2; ++nt)
                            sum[chan(16 * mt + row) * kK * kCh + tap * kCh + chan(ch + 8 * nt + col)] += acc[tap][mt][nt][q];
                if (LAST && col < kK * kCin) sum[kW + kCh + chan(ch + row) * kK * kCin + col] += acc1[q];
            }
            if (g == 0) {
#pragma unroll
                for (int nt = 0; nt < 2; ++nt) {
                    const int c = ch + 4 * wq + 2 * nt;
                    sum[kW + c] += gb[nt].x;
                    sum[kW + c + 1] += gb[nt].y;
                    if (LAST) {
                        sum[kO - kCh + c] += gb1[nt].x;
                        sum[kO - kCh + c + 1] += gb1[nt].y;
                    }
                }
            }
        }
        __syncthreads();
    }
    for (int e = threadIdx.x; e < kO; e += kBwdWarps * 32) part[(size_t)blockIdx.x * kO + e] = sum[e];
}

// The gradients from the blocks' sums: output o of the list [head | conv3 | conv2 and conv1] adds its column
// over the blocks, in a fixed order: a block takes 32 outputs (one per lane), its 8 warps the 8 contiguous
// eighths of the blocks, and the eighths' sums are added in order.
__global__ void __launch_bounds__(256)
    k_grads(int N, int head_blocks, const float *__restrict__ head, const float *__restrict__ c3, const float *__restrict__ c2,
            int conv_blocks, float *__restrict__ grad, float *__restrict__ loss)
{
    wait_previous();
    constexpr int O3 = kBwdOut<false>, O2 = kBwdOut<true>, kW = kCh * kK * kCh;
    __shared__ float sh[8][32];
    const int lane = lane_id(), w = threadIdx.x >> 5;
    const int o = blockIdx.x * 32 + lane;
    const float *src = nullptr;
    int stride = 0, nb = 0;
    float *dst = nullptr;
    if (o < kHeadOut) {
        src = head + o;
        stride = kHeadOut;
        nb = head_blocks;
        dst = o < kHid ? grad + oW5 + o : o < 2 * kHid ? grad + oB4 + o - kHid : o == 2 * kHid ? grad + oB5 : loss;
    } else if (o < kHeadOut + O3) {
        const int e = o - kHeadOut;
        src = c3 + e;
        stride = O3;
        nb = conv_blocks;
        dst = grad + (e < kW ? oW3 + e : oB3 + e - kW);
    } else if (o < kHeadOut + O3 + O2) {
        const int e = o - kHeadOut - O3;
        src = c2 + e;
        stride = O2;
        nb = conv_blocks;
        dst = grad + (e < kW ? oW2 + e : e < kW + kCh ? oB2 + e - kW : e < O2 - kCh ? oW1 + e - kW - kCh : oB1 + e - (O2 - kCh));
    }
    const int b0 = (int)((long long)nb * w / 8), b1 = (int)((long long)nb * (w + 1) / 8);
    float t = 0.0f;
#pragma unroll 8
    for (int b = b0; b < b1; ++b) t += src[(size_t)b * stride];
    sh[w][lane] = t;
    __syncthreads();
    if (w == 0 && dst) {
        float v = 0.0f;
        for (int k = 0; k < 8; ++k) v += sh[k][lane];
        *dst = dst == loss ? v / (float)N : v;
    }
}

// ---- the conv stack in registers ------------------------------------------------------------------
//
// One warp per beam. An accumulator tile of mma.m16n8k16 holds (row g, columns 2w, 2w + 1) and
// (row g + 8, the same), g = lane / 4, w = lane % 4; packed to BF16 pairs that is the A operand
// of the next layer's MMA for the same rows. A stride-2 conv's row t reads its input at positions
// 2t - 1, 2t, 2t + 1, so the layers are computed for strips of 16 positions t with equal residues:
// for conv3's positions u = u0 .. u0 + 15, conv2 at 2u and 2u + 1, conv1 at 4u .. 4u + 3. Each strip is
// then the next layer's operand for one tap as it stands; the remaining tap, position 4u - 1 (2u - 1), is
// the strip of 4u + 3 (2u + 1) one row down, two shuffles per pair of registers. No activation
// goes through shared memory: a beam writes its profile there (1 KB) and reads it as conv1's operand.
//
// What bounds it: the kernel with the activations in shared memory moved about 700 wavefronts of
// shared memory per beam (its pipe 78 % busy, the tensor pipe 39 %) and 1,835 warp instructions; this one
// moves 185 and issues 1,000, and the tensor pipe (62 % busy) is the bound. 4096 x 360 beams: 2.65 ms
// against 4.27 ms. Three blocks of four warps per SM leave 168 registers, which hold conv2's weight
// fragments. Measured on the same batch, conv and fc together: 3.29 ms so; 3.32 ms with four blocks and
// conv2's weights read per strip, 3.38 - 3.61 ms with the next beam's samples fetched ahead (registers),
// 3.78 ms with both strips of a beam unrolled.
constexpr int kConvWarps = 4;
constexpr int kXWords = 4 + kL;  // a beam's profile, with zeros before it
// block: W1 [32][8], W2 / W3 [32][104] bf16, kL zero words, then each warp's profile
constexpr int kConvSmem = kCh * 8 * 2 + 2 * kCh * kS2 * 2 + kL * 4 + kConvWarps * kXWords * 4;

// relu(acc + b) as bf16 pairs: P[nt][h] = columns 8 nt + 2w, + 1 of row g + 8 h
__device__ __forceinline__ void relu_pack(const float (&acc)[4][4], const float2 (&b)[4], unsigned (&P)[4][2])
{
    const __nv_bfloat162 zero = __floats2bfloat162_rn(0.0f, 0.0f);
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const __nv_bfloat162 v = __hmax2(__floats2bfloat162_rn(acc[nt][2 * h] + b[nt].x, acc[nt][2 * h + 1] + b[nt].y), zero);
            P[nt][h] = *reinterpret_cast<const unsigned *>(&v);
        }
}

// The strip one row down: row g takes row g - 1, row 0 the last row of the strip before (carry, which
// then holds this strip's last row).
__device__ __forceinline__ void shift_rows(const unsigned (&P)[4][2], unsigned (&carry)[4], unsigned (&S)[4][2])
{
    const int lane = lane_id();
    const bool first = lane < 4;
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
        const unsigned lo = __shfl_sync(kFull, P[nt][0], lane + 28), hi = __shfl_sync(kFull, P[nt][1], lane + 28);
        S[nt][0] = first ? carry[nt] : lo;
        S[nt][1] = first ? lo : hi;
        carry[nt] = hi;
    }
}

// acc += (channels 16 hh .. of one tap's strip P) W
__device__ __forceinline__ void tap_mma(float (&acc)[4][4], const unsigned (&P)[4][2], int hh, const unsigned (&bw)[4][2])
{
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
        mma_bf16(acc[nt], P[2 * hh][0], P[2 * hh][1], P[2 * hh + 1][0], P[2 * hh + 1][1], bw[nt][0], bw[nt][1]);
}

// Conv stack for N beams: profiles from the map (map != nullptr; beam n = pose n / B, direction
// n % B) or given (x [N][256] bf16 pairs). h0 [N][1024] bf16 (index t * 32 + c).
__global__ void __launch_bounds__(kConvWarps * 32, 3)
    k_conv_infer(const float *__restrict__ map, int W, int H, const int32_t *__restrict__ poses,
                 const int32_t *__restrict__ dirs, int B, int keep, const __nv_bfloat162 *__restrict__ xg, long long N,
                 const bf16 *__restrict__ w, const float *__restrict__ params, bf16 *__restrict__ h0,
                 unsigned long long *queue, int chunk)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    bf16 *sW1 = (bf16 *)smem_raw;  // [32][8]
    bf16 *sW2 = sW1 + kCh * 8;     // [32][104]
    bf16 *sW3 = sW2 + kCh * kS2;   // [32][104], row 8 nt + n = output channel 8 (n / 2) + 2 nt + n % 2
    unsigned *zero = (unsigned *)(sW3 + kCh * kS2);
    unsigned *xs = zero + kL + (threadIdx.x >> 5) * kXWords + 4;
    for (int e = threadIdx.x; e < kCh * 8; e += blockDim.x) {
        const int c = e / 8, kk = e % 8;
        sW1[e] = kk < kK * kCin ? w[oW1 + c * kK * kCin + kk] : __float2bfloat16_rn(0.0f);
    }
    for (int e = threadIdx.x; e < kCh * kS2; e += blockDim.x) {
        const int r = e / kS2, kk = e % kS2, c3 = 8 * ((r & 7) >> 1) + 2 * (r >> 3) + (r & 1);
        sW2[e] = kk < kK * kCh ? w[oW2 + r * kK * kCh + kk] : __float2bfloat16_rn(0.0f);
        sW3[e] = kk < kK * kCh ? w[oW3 + c3 * kK * kCh + kk] : __float2bfloat16_rn(0.0f);
    }
    for (int e = threadIdx.x; e < kL; e += blockDim.x) zero[e] = 0u;
    const int lane = lane_id(), g = lane >> 2, wq = lane & 3;
    if (lane < 4) xs[lane - 4] = 0u;  // position -1
    __syncthreads();
    // biases of this lane's columns (conv3: channels 8 w + 2 nt, + 1), W1's fragments
    float2 b1[4], b2[4], b3[4];
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
        const int c = 8 * nt + 2 * wq, c3 = 8 * wq + 2 * nt;
        b1[nt] = make_float2(params[oB1 + c], params[oB1 + c + 1]);
        b2[nt] = make_float2(params[oB2 + c], params[oB2 + c + 1]);
        b3[nt] = make_float2(params[oB3 + c3], params[oB3 + c3 + 1]);
    }
    unsigned bw1[4], bw2[6][4][2];
    ldsm_x4(smem_u32(sW1 + lane * 8), bw1[0], bw1[1], bw1[2], bw1[3]);
#pragma unroll
    for (int ks = 0; ks < 6; ++ks) load_wfrag(sW2, ks, bw2[ks]);
    // conv1's operand for position p: taps 0 .. 2 are the words x[2p - 1 + w], the fourth is zero
    const unsigned *xa = wq < 3 ? xs + 8 * g + wq - 1 : zero;
    // a warp takes `chunk` (<= 32) consecutive beams per queue grab, lane j the j-th's origin and direction
    for (;;) {
        unsigned long long b0 = 0;
        if (lane == 0) b0 = atomicAdd(queue, (unsigned long long)chunk);
        b0 = __shfl_sync(kFull, b0, 0);
        if ((long long)b0 >= N) break;
        const int nb = (int)min((long long)chunk, N - (long long)b0);
        int ox = 0, oy = 0, dx = 0, dy = 0;
        if (map && lane < nb) {
            const long long n = (long long)b0 + lane;
            int pi, bi;
            if (n <= 0x7fffffffLL) {  // 32-bit division, the common case
                pi = (int)((unsigned)n / (unsigned)B);
                bi = (int)((unsigned)n - (unsigned)pi * (unsigned)B);
            } else {
                pi = (int)(n / B);
                bi = (int)(n % B);
            }
            const int32_t *pose = poses + 4 * (size_t)pi;
            ox = pose[0];
            oy = pose[1];
            beam_dir_2d(pose, dirs + 2 * (size_t)bi, dx, dy);
        }
        for (int j = 0; j < nb; ++j) {
            const long long n = (long long)b0 + j;
            if (map) {
                // sample i lies in the cell floor of the Q31 position (o << 15) + (2 i + 1) d; the low 32
                // bits of the shifted position are the cell inside the map and at least its extent outside
                const int sx = __shfl_sync(kFull, ox, j), sy = __shfl_sync(kFull, oy, j);
                const int ex = __shfl_sync(kFull, dx, j), ey = __shfl_sync(kFull, dy, j);
                long long px = ((long long)sx << 15) + (2LL * lane + 1) * ex;
                long long py = ((long long)sy << 15) + (2LL * lane + 1) * ey;
                float o[kL / 32];
                bool in[kL / 32];
#pragma unroll
                for (int k = 0; k < kL / 32; ++k) {
                    const unsigned cx = (unsigned)(px >> 31), cy = (unsigned)(py >> 31);
                    in[k] = lane + 32 * k < keep && cx < (unsigned)W && cy < (unsigned)H;
                    o[k] = in[k] ? __ldg(map + ((size_t)cy * W + cx)) : 0.0f;
                    px += 64LL * ex;
                    py += 64LL * ey;
                }
#pragma unroll
                for (int k = 0; k < kL / 32; ++k) xs[lane + 32 * k] = pack_bf16x2(o[k], in[k] ? 1.0f : 0.0f);
            } else {
                const unsigned *xr = reinterpret_cast<const unsigned *>(xg) + n * kL;
#pragma unroll
                for (int k = 0; k < kL / 32; ++k) xs[lane + 32 * k] = xr[lane + 32 * k];
            }
            __syncwarp();
            unsigned carry1[4] = {0u, 0u, 0u, 0u}, carry2[4] = {0u, 0u, 0u, 0u};
#pragma unroll 1
            for (int s = 0; s < 2; ++s) {  // u = 16 s + row
                unsigned P[4][4][2], S[4][2];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const unsigned *x = xa + 128 * s + 2 * r;
                    const unsigned a0 = x[0], a1 = x[wq < 3 ? 64 : 0];
                    float acc[4][4];
#pragma unroll
                    for (int nt = 0; nt < 4; ++nt) {
                        acc[nt][0] = acc[nt][1] = acc[nt][2] = acc[nt][3] = 0.0f;
                        mma_bf16_k8(acc[nt], a0, a1, bw1[nt]);
                    }
                    relu_pack(acc, b1, P[r]);
                }
                shift_rows(P[3], carry1, S);
                float ev[4][4] = {}, od[4][4] = {};
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    tap_mma(ev, S, hh, bw2[hh]);
                    tap_mma(od, P[1], hh, bw2[hh]);
                }
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    tap_mma(ev, P[0], hh, bw2[2 + hh]);
                    tap_mma(od, P[2], hh, bw2[2 + hh]);
                }
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    tap_mma(ev, P[1], hh, bw2[4 + hh]);
                    tap_mma(od, P[3], hh, bw2[4 + hh]);
                }
                unsigned E[4][2], O[4][2];
                relu_pack(ev, b2, E);
                relu_pack(od, b2, O);
                shift_rows(O, carry2, S);
                float acc[4][4] = {};
#pragma unroll
                for (int ks = 0; ks < 6; ++ks) {
                    unsigned bw[4][2];
                    load_wfrag(sW3, ks, bw);
                    tap_mma(acc, ks < 2 ? S : ks < 4 ? E : O, ks & 1, bw);
                }
                unsigned Q[4][2];
                relu_pack(acc, b3, Q);  // lane w: channels 8 w .. 8 w + 7 of rows g and g + 8
                uint4 *dst = reinterpret_cast<uint4 *>(h0 + n * kFlat + (16 * s + g) * kCh + 8 * wq);
                dst[0] = make_uint4(Q[0][0], Q[1][0], Q[2][0], Q[3][0]);
                dst[kCh] = make_uint4(Q[0][1], Q[1][1], Q[2][1], Q[3][1]);  // 8 rows of 32 bf16 further
            }
            __syncwarp();
        }
    }
}

// ---- fc1 + ReLU + fc2 on the 5th-generation tensor cores (tcgen05, accumulators in TMEM) ------------
//
// Persistent CTAs of 6 warps, one per SM, each taking 128-row tiles: D[128][256] = h0_tile[128][1024]
// W4^T accumulates in 256 TMEM columns (FP32, row i in TMEM lane i), in one of two accumulators so
// that a tile's epilogue overlaps the next tile's MMAs. K runs in chunks of 64 through a 4-stage
// TMA pipeline; each stage holds A (128 x 64) and B (256 x 64) in the K-major layout with the
// 128-byte swizzle (16-byte chunk c of row r at c ^ (r & 7), 8-row groups 1024 B apart, 1024-byte
// aligned), written so by the tensor-map copies. Roles: warp 4 issues the copies (stage ring with
// "full" / "empty" mbarriers), warp 5 issues 4 MMAs (M = 128, N = 256, K = 16) per chunk, commits
// them to the stage's "empty" barrier and, after a tile's last chunk, to the accumulator's "tfull"
// barrier; warps 0-3 read their 32 TMEM lanes each (one row per thread), release the accumulator
// ("tempty") and form b5 + sum_j W5[j] relu(D + b4). Every wait is bounded: on timeout the kernel
// sets FSMI_STATUS_TIMEOUT, writes NaN for the rows it could not finish and returns after its
// copies and MMAs in flight have landed (again with bounded waits).

constexpr int kTcRows = 128, kTcK = 64, kTcStages = 4, kTcThreads = 192;
constexpr int kTcStageBytes = (kTcRows + kHid) * kTcK * 2;  // 48 KB
constexpr int kTcChunks = kFlat / kTcK;                      // 16
constexpr unsigned kTcAcc = 256;                             // TMEM columns per accumulator (FP32)
constexpr unsigned kTcCols = 2 * kTcAcc;
constexpr int kTcBars = 2 * kTcStages + 5;                   // full, empty, tfull[2], tempty[2], drain
constexpr size_t kTcSmem = 1024 + (size_t)kTcStages * kTcStageBytes + 8 * kTcBars + kHid * 8 + 16;
// instruction descriptor, kind::f16: D F32 (bits 4-5 = 1), A BF16 (bits 7-9 = 1), B BF16
// (bits 10-12 = 1), both K-major, N / 8 at bits 17-22, M / 16 at bits 24-28
constexpr unsigned kTcIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(kHid >> 3) << 17) |
                              ((unsigned)(kTcRows >> 4) << 24);
constexpr long long kWaitPolls = 1LL << 22;
// poll limit of the epilogue's wait for its accumulator, per host thread (fsmi_set_wait_limit)
thread_local long long g_epi_polls = kWaitPolls;

// shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups 1024 B apart
__device__ __forceinline__ unsigned long long sdesc_sw128(unsigned saddr)
{
    unsigned long long d = (unsigned long long)((saddr & 0x3FFFFu) >> 4);
    d |= 1ull << 16;                      // leading byte offset: not used by swizzled K-major operands
    d |= (unsigned long long)(1024 >> 4) << 32;  // stride byte offset
    d |= 1ull << 46;                      // descriptor version of the sm_100 family
    d |= 2ull << 61;                      // 128-byte swizzle
    return d;
}

__device__ __forceinline__ void mbar_init(unsigned addr, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(addr), "r"(count) : "memory");
}

__device__ __forceinline__ bool mbar_test(unsigned addr, unsigned parity)
{
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(addr), "r"(parity)
        : "memory");
    return ok != 0;
}

// bounded wait for the phase with the given parity to complete (at most `polls` tests)
__device__ __forceinline__ bool mbar_wait(unsigned addr, unsigned parity, long long polls = kWaitPolls)
{
    for (long long i = 0; i < polls; ++i)
        if (mbar_test(addr, parity)) return true;
    return false;
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tc_mma(unsigned dtmem, unsigned long long adesc, unsigned long long bdesc,
                                       unsigned idesc, unsigned accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(dtmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void tc_commit(unsigned mbar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar) : "memory");
}

// 32 consecutive FP32 columns of this thread's TMEM lane
__device__ __forceinline__ void tc_ld32(unsigned taddr, float (&v)[32])
{
    unsigned r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,"
        "%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void mbar_expect_tx(unsigned addr, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(addr), "r"(bytes) : "memory");
}

// TMA: a box of the 2D tensor map at (x = element along K, y = row) into shared memory, completing
// `bytes` of the mbarrier's transaction count
__device__ __forceinline__ void tma_load_2d(unsigned dst, const CUtensorMap *map, int x, int y, unsigned mbar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(mbar)
        : "memory");
}

__device__ __forceinline__ void mbar_arrive(unsigned addr)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(addr) : "memory");
}

__device__ __forceinline__ int flag_of(const int *flag) { return *(const volatile int *)flag; }

__global__ void __launch_bounds__(kTcThreads, 1)
    k_fc_tc(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, long long N,
            const bf16 *__restrict__ w, const float *__restrict__ params, float *__restrict__ pred, int *status,
            long long epi_polls)
{
    extern __shared__ unsigned char smem_raw[];
    unsigned char *base = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned long long *full = (unsigned long long *)(base + (size_t)kTcStages * kTcStageBytes);
    unsigned long long *empty = full + kTcStages;
    unsigned long long *tfull = empty + kTcStages;
    unsigned long long *tempty = tfull + 2;
    unsigned long long *drain = tempty + 2;
    float2 *bw = (float2 *)(drain + 1);  // (b4[j], W5[j])
    unsigned *tmem_slot = (unsigned *)(bw + kHid);
    __shared__ int flag;  // 0 while every wait succeeded
    const int tid = threadIdx.x, warp = tid >> 5, lane = lane_id();
    if (warp == 5) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(kTcCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int i = 0; i < kTcStages; ++i) {
            mbar_init(smem_u32(full + i), 1);
            mbar_init(smem_u32(empty + i), 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(tfull + i), 1);
            mbar_init(smem_u32(tempty + i), 4);  // lane 0 of each epilogue warp
        }
        mbar_init(smem_u32(drain), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        flag = 0;
    }
    if (tid == 4 * 32) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<unsigned long long>(&tmA)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<unsigned long long>(&tmB)) : "memory");
    }
    for (int j = tid; j < kHid; j += kTcThreads) bw[j] = make_float2(params[oB4 + j], bf(w, oW5 + j));
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = *tmem_slot;
    const long long tiles = (N + kTcRows - 1) / kTcRows;
    if (warp == 4) {
        if (lane == 0) {  // TMA producer
            long long it = 0;  // chunks issued by this CTA; stage it % S, its use number it / S
            bool ok = true;
            for (long long t = blockIdx.x; t < tiles && ok; t += gridDim.x)
                for (int kc = 0; kc < kTcChunks; ++kc) {
                    const int st = (int)(it % kTcStages);
                    const long long u = it / kTcStages;
                    if (u > 0 && !mbar_wait(smem_u32(empty + st), (unsigned)((u - 1) & 1))) ok = false;
                    if (!ok || flag_of(&flag)) {
                        ok = false;
                        break;
                    }
                    const unsigned a0 = smem_u32(base + (size_t)st * kTcStageBytes);
                    mbar_expect_tx(smem_u32(full + st), (unsigned)kTcStageBytes);
                    tma_load_2d(a0, &tmA, kc * kTcK, (int)(t * kTcRows), smem_u32(full + st));
                    tma_load_2d(a0 + kTcRows * kTcK * 2, &tmB, kc * kTcK, 0, smem_u32(full + st));
                    ++it;
                }
            // copies in flight: the last fill of every stage has landed
            for (long long j = it - 1; j >= 0 && j >= it - kTcStages; --j)
                if (!mbar_wait(smem_u32(full + (int)(j % kTcStages)), (unsigned)((j / kTcStages) & 1))) ok = false;
            if (!ok) atomicOr(&flag, 1);
        }
    } else if (warp == 5) {
        if (lane == 0) {  // MMA issuer
            long long it = 0;
            int tl = 0;
            bool ok = true;
            for (long long t = blockIdx.x; t < tiles && ok; t += gridDim.x, ++tl) {
                const int b = tl & 1, v = tl >> 1;
                if (v > 0 && !mbar_wait(smem_u32(tempty + b), (unsigned)((v - 1) & 1))) ok = false;
                if (!ok || flag_of(&flag)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const unsigned d = tmem + (unsigned)b * kTcAcc;
                for (int kc = 0; kc < kTcChunks; ++kc, ++it) {
                    const int st = (int)(it % kTcStages);
                    if (!mbar_wait(smem_u32(full + st), (unsigned)((it / kTcStages) & 1))) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const unsigned a0 = smem_u32(base + (size_t)st * kTcStageBytes), b0 = a0 + kTcRows * kTcK * 2;
#pragma unroll
                    for (int k = 0; k < kTcK / 16; ++k)  // K = 16 per MMA: 32 bytes along the swizzled row
                        tc_mma(d, sdesc_sw128(a0 + 32 * k), sdesc_sw128(b0 + 32 * k), kTcIdesc, (kc | k) != 0);
                    tc_commit(smem_u32(empty + st));
                }
                if (ok) tc_commit(smem_u32(tfull + b));
            }
            if (!ok) atomicOr(&flag, 1);
            tc_commit(smem_u32(drain));  // every MMA issued has completed once this arrives
            if (!mbar_wait(smem_u32(drain), 0u)) atomicOr(&flag, 1);
        }
    } else {  // epilogue: warp w holds TMEM lanes 32w .. 32w + 31, one row per thread
        int tl = 0;
        bool ok = true;
        for (long long t = blockIdx.x; t < tiles; t += gridDim.x, ++tl) {
            const int b = tl & 1, v = tl >> 1;
            const long long row = t * kTcRows + warp * 32 + lane;
            float acc = 0.0f;
            // the one wait whose limit the caller sets (fsmi_set_wait_limit): the producer's and the
            // MMA issuer's waits keep the full limit, so that every copy and MMA in flight has landed
            // before TMEM is freed, whatever happens here
            if (ok) ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(tfull + b), (unsigned)(v & 1), epi_polls));
            if (ok) {
                tc_fence_after();
                const unsigned ta = tmem + ((unsigned)(warp * 32) << 16) + (unsigned)b * kTcAcc;
                for (int c0 = 0; c0 < kHid; c0 += 32) {
                    float x[32];
                    tc_ld32(ta + (unsigned)c0, x);
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const float2 q = bw[c0 + j];
                        acc = fmaf(relu(x[j] + q.x), q.y, acc);
                    }
                }
                tc_fence_before();
            } else if (lane == 0) {
                atomicOr(&flag, 1);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(tempty + b));
            if (row < N) pred[row] = ok ? params[oB5] + acc : __int_as_float(0x7fc00000);
        }
    }
    __syncthreads();
    if (tid == 0 && flag != 0) set_status(status, FSMI_STATUS_TIMEOUT);
    if (warp == 5) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcCols) : "memory");
    }
}

// ---- selection -------------------------------------------------------------------------------------

// Indices of the k largest of v[0..n) in descending order (ties: lower index first), by a bitonic
// sort of (value, index) keys in shared memory. One block; n <= 16384.
__global__ void __launch_bounds__(1024) k_topk(const float *__restrict__ v, int n, int k, int32_t *__restrict__ idx)
{
    extern __shared__ unsigned long long keys[];
    int m = 1;
    while (m < n) m <<= 1;
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        unsigned long long key = 0ull;  // padding sorts last
        if (i < n) {
            float f = v[i];
            if (f != f) f = -FLT_MAX;  // NaN ranks with the smallest
            unsigned u = __float_as_uint(f);
            u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);  // order-preserving map to unsigned
            key = ((unsigned long long)u << 32) | (unsigned)(0xFFFFFFFFu - (unsigned)i);
            if (key == 0ull) key = 1ull;
        }
        keys[i] = key;
    }
    __syncthreads();
    // descending bitonic sort
    for (int size = 2; size <= m; size <<= 1)
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int i = threadIdx.x; i < m; i += blockDim.x) {
                const int j = i ^ stride;
                if (j > i) {
                    const bool desc = (i & size) == 0;
                    const unsigned long long a = keys[i], b = keys[j];
                    if (desc ? (a < b) : (a > b)) {
                        keys[i] = b;
                        keys[j] = a;
                    }
                }
            }
            __syncthreads();
        }
    for (int i = threadIdx.x; i < k; i += blockDim.x) idx[i] = (int32_t)(0xFFFFFFFFu - (unsigned)(keys[i] & 0xFFFFFFFFull));
}

// dst[r][.] = src[idx[r]][.] for rows of `width` int32; an index outside [0, nrows) gives zeros
__global__ void k_gather_rows(const int32_t *__restrict__ src, long long nrows, int width,
                              const int32_t *__restrict__ idx, int k, int32_t *__restrict__ dst, int *status)
{
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < k * width; e += gridDim.x * blockDim.x) {
        const long long r = idx[e / width];
        const bool ok = r >= 0 && r < nrows;
        if (!ok && e % width == 0) set_status(status, FSMI_STATUS_BAD_BEAM);
        dst[e] = ok ? src[r * width + e % width] : 0;
    }
}

}  // namespace

// ---- launchers -----------------------------------------------------------------------------------

size_t surrogate_train_floats(int N)
{
    const size_t n = (size_t)N;
    const size_t z = n * (128 + 64 + 32) * kCh + n * kHid;  // z1..z4
    const size_t g = n * 128 * kCh;                          // relu(z3) and dz4 in terms, dz3, dz2: 4864 n of 2 g = 8192 n
    const size_t part = (size_t)64 * kHid * kFlat;           // the sums over blocks (fc1's, the head's, the convolutions')
    return z + 3 * ((n + 3) & ~(size_t)3) + 2 * g + part + 64;  // pred, dpred, lossp each padded to 4 floats
}

cudaError_t launch_profiles(const float *map, int W, int H, const int32_t *poses, int P, const int32_t *dirs, int B,
                            int keep, const int32_t *beam_ids, long long N, void *out, int *status, cudaStream_t s)
{
    if (N <= 0) return cudaSuccess;
    k_profiles<<<grid_cap((N + 7) / 8), 256, 0, s>>>(map, W, H, poses, dirs, B, keep, (long long)P * B, beam_ids, N,
                                                     (__nv_bfloat162 *)out, status);
    return cudaGetLastError();
}

cudaError_t launch_surrogate_loss_grad(const float *params, const void *wbf16, const void *x, const float *y, int N,
                                       float *grad, float *loss, float *pred_out, float *ws, cudaStream_t s)
{
    const bf16 *w = (const bf16 *)wbf16;
    const size_t n = (size_t)N, pad = (n + 3) & ~(size_t)3;
    float *q = ws;
    auto take = [&](size_t floats) {  // every buffer 16-byte aligned
        float *r = q;
        q += (floats + 3) & ~(size_t)3;
        return r;
    };
    float *z1 = take(n * 128 * kCh), *z2 = take(n * 64 * kCh), *z3 = take(n * 32 * kCh), *z4 = take(n * kHid);
    float *pred_ws = take(pad);
    bf16 *h = (bf16 *)take(n * kFlat * 3 / 2);  // relu(z3), three terms
    bf16 *dz4 = (bf16 *)take(n * kHid);         // two terms
    float *dz3 = take(n * kFlat), *dz2 = take(n * 64 * kCh);
    const int splits = fc1_splits(N), head_blocks = (N + kHeadRows - 1) / kHeadRows;
    float *part4 = take((size_t)splits * kHid * kFlat), *part_h = take((size_t)head_blocks * kHeadOut);
    float *part3 = take((size_t)kBwdBlocks * kBwdOut<false>), *part2 = take((size_t)kBwdBlocks * kBwdOut<true>);
    bf16 *w4 = (bf16 *)w + oW4;
    cudaError_t e;
#define FSMI_TRY(...)            \
    do {                         \
        e = (__VA_ARGS__);       \
        if (e != cudaSuccess) return e; \
    } while (0)
    if ((uintptr_t)w4 & 15) {  // weights off a 16-byte boundary: the copies of the products need an aligned W4
        w4 = (bf16 *)take((size_t)kHid * kFlat / 2);
        FSMI_TRY(cudaMemcpyAsync(w4, w + oW4, (size_t)kHid * kFlat * sizeof(bf16), cudaMemcpyDeviceToDevice, s));
    }
    // Each launch below may be early, so that its blocks are in place when the one before ends; a kernel waits for
    // that end before it reads anything but weights (`beside`: it needs nothing of the launch before, only of
    // the one before that, and ends after both). In order: the first, and the one that reads dz3, whose
    // memory the head read as part1 (no line of it may be left in an L1). A batch of 4096 with the weight gradients
    // from two terms: 265 us with every launch in order, 243 us like this (268 us with three terms).
    // forward
    k_convs_fwd<<<grid_cap(((long long)N + kFwdWarps - 1) / kFwdWarps), kFwdWarps * 32, 0, s>>>(N, (const unsigned *)x, w, params, z1,
                                                                                              z2, z3, h, n * kFlat);
    FSMI_TRY(cudaGetLastError());
    float *part1 = dz3;  // fc1's sums by splits of K, added by the head
    const int fsplits = fc1_forward_splits(N);
    FSMI_TRY(gemm_terms<3, 1, false, false>(N, kHid, kFlat, fsplits, h, n * kFlat, kFlat, w4, 0, kFlat,
                                            StorePart{part1, N, kHid}, false, s));
    FSMI_TRY(launch_kernel(true, k_head, head_blocks, 256, 0, s, part1, w, params, y, N, z4, pred_out ? pred_out : pred_ws, dz4,
                           part_h, fsplits));
    if (!y) return cudaSuccess;
    // backward: fc1's weights gW4[j][i] = sum_n dz4[n][j] relu(z3)[n][i] and data dz3 = (dz4 W4) [z3 > 0], the
    // second beside the first
    FSMI_TRY(gemm_terms<2, 2, true, true>(kHid, kFlat, N, splits, dz4, n * kHid, kHid, h, n * kFlat, kFlat,
                                          StorePart{part4, kHid, kFlat}, false, s));
    FSMI_TRY(gemm_terms<2, 1, false, true>(N, kFlat, kHid, 1, dz4, n * kHid, kHid, w4, 0, kFlat, StoreMask{dz3, z3, kFlat}, true,
                                           s));
    // conv3, then conv2 and conv1; fc1's sum over the splits beside the last
    FSMI_TRY(launch_kernel(false, k_conv_bwd<false>, kBwdBlocks, kBwdWarps * 32, 0, s, N, 64, dz3, w + oW3, z2, (const bf16 *)nullptr, dz2,
                           part3));
    FSMI_TRY(launch_kernel(true, k_conv_bwd<true>, kBwdBlocks, kBwdWarps * 32, 0, s, N, 128, dz2, w + oW2, z1, (const bf16 *)x,
                           (float *)nullptr, part2));
    FSMI_TRY(launch_kernel(true, k_split_reduce, grid_cap(kHid * kFlat / 256), 256, 0, s, kHid * kFlat, splits, part4, grad + oW4));
    const int outs = kHeadOut + kBwdOut<false> + kBwdOut<true>;
    return launch_kernel(true, k_grads, (outs + 31) / 32, 256, 0, s, N, head_blocks, part_h, part3, part2, kBwdBlocks, grad, loss);
#undef FSMI_TRY
}

cudaError_t launch_surrogate_adam(float *p, float *m, float *v, const float *g, float lr, float b1, float b2, float eps,
                                  int t, void *wbf16, cudaStream_t s)
{
    const float c1 = (float)(1.0 - pow((double)b1, (double)t)), c2 = (float)(1.0 - pow((double)b2, (double)t));
    k_adam<<<grid_cap((kNParams + 255) / 256), 256, 0, s>>>(p, m, v, g, kNParams, lr, b1, b2, eps, c1, c2,
                                                           (bf16 *)wbf16);
    return cudaGetLastError();
}

cudaError_t launch_surrogate_cast(const float *p, void *wbf16, cudaStream_t s)
{
    k_cast<<<grid_cap((kNParams + 255) / 256), 256, 0, s>>>(p, kNParams, (bf16 *)wbf16);
    return cudaGetLastError();
}

}  // namespace fsmi

namespace fsmi {

size_t surrogate_infer_bytes(long long N) { return kQueueBytes + (size_t)N * kFlat * sizeof(bf16); }

namespace {

// cuTensorMapEncodeTiled through the runtime's driver entry point (looked up once)
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder()
{
    static std::once_flag once;
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    });
    return fn;
}

// Row-major BF16 matrix [rows][cols] (16-byte aligned, rows of cols * 2 bytes) as a 2D tensor map
// with boxes of box_cols x box_rows and the 128-byte swizzle; out-of-range rows read as zero.
cudaError_t encode_bf16_2d(CUtensorMap *map, const void *ptr, unsigned long long cols, unsigned long long rows,
                           unsigned box_cols, unsigned box_rows)
{
    PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
    if (!enc) return cudaErrorNotSupported;
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {cols * 2};
    const cuuint32_t box[2] = {box_cols, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(ptr), dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_surrogate_infer(const float *map, int W, int H, const int32_t *poses, const int32_t *dirs, int B,
                                   int keep, const void *x, long long N, const void *wbf16, const float *params,
                                   float *pred, void *ws, int *status, cudaStream_t s)
{
    if (N <= 0) return cudaSuccess;
    const bf16 *w = (const bf16 *)wbf16;
    unsigned long long *queue = (unsigned long long *)ws;
    bf16 *h0 = (bf16 *)((char *)ws + kQueueBytes);
    const size_t smem_conv = kConvSmem;
    int occ = 0;
    cudaError_t e = resident_blocks((const void *)k_conv_infer, kConvWarps * 32, smem_conv, occ);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(queue, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    long long grid = (long long)sm_count() * occ;
    if (grid > (N + kConvWarps - 1) / kConvWarps) grid = (N + kConvWarps - 1) / kConvWarps;
    const long long chunk = N / (grid * kConvWarps * 8);  // eight grabs per warp at least, up to 8 beams each
    k_conv_infer<<<(unsigned)grid, kConvWarps * 32, smem_conv, s>>>(map, W, H, poses, dirs, B, keep,
                                                                     (const __nv_bfloat162 *)x, N, w, params, h0, queue,
                                                                     (int)std::max(1LL, std::min(8LL, chunk)));
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const long long tiles = (N + kTcRows - 1) / kTcRows;
    CUtensorMap tmA, tmB;
    e = encode_bf16_2d(&tmA, h0, kFlat, (unsigned long long)N, kTcK, kTcRows);
    if (e == cudaSuccess) e = encode_bf16_2d(&tmB, w + oW4, kFlat, kHid, kTcK, kHid);
    if (e != cudaSuccess) return e;
    e = resident_blocks((const void *)k_fc_tc, kTcThreads, kTcSmem, occ);
    if (e != cudaSuccess) return e;
    k_fc_tc<<<(unsigned)(tiles < (long long)sm_count() ? tiles : sm_count()), kTcThreads, kTcSmem, s>>>(
        tmA, tmB, N, w, params, pred, status, g_epi_polls);
    return cudaGetLastError();
}

void set_epilogue_polls(long long polls) { g_epi_polls = polls < 0 ? kWaitPolls : polls; }

cudaError_t launch_topk(const float *v, int n, int k, int32_t *idx, cudaStream_t s)
{
    int m = 1;
    while (m < n) m <<= 1;
    const size_t smem = (size_t)m * sizeof(unsigned long long);
    cudaError_t e = cudaFuncSetAttribute(k_topk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_topk<<<1, 1024, smem, s>>>(v, n, k, idx);
    return cudaGetLastError();
}

cudaError_t launch_gather_rows(const int32_t *src, long long nrows, int width, const int32_t *idx, int k,
                               int32_t *dst, int *status, cudaStream_t s)
{
    if (k <= 0) return cudaSuccess;
    k_gather_rows<<<grid_cap((k * width + 255) / 256), 256, 0, s>>>(src, nrows, width, idx, k, dst, status);
    return cudaGetLastError();
}

cudaError_t prepare_surrogate()
{
    cudaFuncAttributes a;
    cudaError_t e = cudaFuncGetAttributes(&a, k_conv_infer);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_fc_tc);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_topk);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_gather_rows);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_profiles);
    return e;
}

}  // namespace fsmi
