// Device helpers shared by the 2D and RLE kernels: warp scans, the per-cell gain, the Gaussian
// tail, integer powers.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "fsmi_internal.h"

namespace fsmi {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }

__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// inclusive scans across the 32 lanes
__device__ __forceinline__ float warp_incl_add(float v)
{
    const int lane = lane_id();
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        float t = __shfl_up_sync(kFull, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

__device__ __forceinline__ float warp_incl_mul(float v)
{
    const int lane = lane_id();
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        float t = __shfl_up_sync(kFull, v, o);
        if (lane >= o) v *= t;
    }
    return v;
}

__device__ __forceinline__ int warp_incl_add_int(int v)
{
    const int lane = lane_id();
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(kFull, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// Information gain of one cell whose odds are multiplied by delta (Section 2.2). Written as the
// Bernoulli KL divergence between posterior o' = o delta / (1 + a), a = o (delta - 1), and prior
// o, which equals the printed f(delta, r) and stays accurate as o -> 0 or 1:
//   f = o' log1p((delta - 1)(1 - o) / (1 + a)) - (1 - o) / (1 + a) log1p(a).
// Every operation is rounded explicitly (no contraction left to the compiler), so that the kernels
// that inline it all compute the same floats.
__device__ __forceinline__ float cell_gain(float delta, float o)
{
    const float dm1 = __fsub_rn(delta, 1.0f);
    const float a = __fmul_rn(o, dm1);
    const float ria = __fdiv_rn(1.0f, __fadd_rn(1.0f, a));
    const float omo = __fsub_rn(1.0f, o);
    const float post = __fmul_rn(__fmul_rn(o, delta), ria);
    const float l1 = log1pf(__fmul_rn(__fmul_rn(dm1, omo), ria));
    return __fsub_rn(__fmul_rn(post, l1), __fmul_rn(__fmul_rn(omo, ria), log1pf(a)));
}

// Upper Gaussian tail in the erfc variable: 0.5 * erfc(z) = 1 - Phi(z sqrt(2)), z >= 0.
__device__ __forceinline__ float half_erfc(float z) { return 0.5f * erfcf(z); }

// x^k for integer k >= 0 by binary powering (x^0 = 1, also for x = 0).
__device__ __forceinline__ float ipowf(float x, int k)
{
    float r = 1.0f;
    while (k > 0) {
        if (k & 1) r *= x;
        x *= x;
        k >>= 1;
    }
    return r;
}

// Warp scan over the n cells held in shared memory (16-byte aligned arrays with room for n + 4). On entry
// sp = o, sc = f_occ, sx = f_emp. On exit sp = P(e_j), sc = C_j (sc[n] = 0), and for the uniform variant
// sx = D_j; the entries after the last cell are left undefined (sc[n] apart). Returns P(e_0).
//
// A lane takes 4 V consecutive cells as V 16-byte loads per array (V = ceil(n / 128)): a quarter of the
// shared-memory instructions of one-float accesses for the same wavefronts (with V = 2 the lanes' loads
// meet two to a bank; 8-byte accesses in odd blocks avoid that and were slower: Uniform-FSMI on the
// 2048x2048 office batch 688 against 665 us). The products go cell by cell: in groups of four, a span of equal
// cells rounds alike in every group and the product drifts (700 cells and more: 1.0e-6 rms against 6e-7).
__device__ __forceinline__ float cell_prefixes(float *sp, float *sc, float *sx, int n, bool want_d)
{
    const int lane = lane_id();
    if (lane < 4) {  // the tail of the last group: o = 0, f_emp = 0 change no prefix
        sp[n + lane] = 0.0f;
        sx[n + lane] = 0.0f;
    }
    __syncwarp();
    const int V = (n + 127) >> 7, lo = 4 * V * lane, hi = min(n, lo + 4 * V);
    float prod = 1.0f, sum = 0.0f;
    for (int i = lo; i < hi; i += 4) {
        const float4 o = *reinterpret_cast<const float4 *>(sp + i), f = *reinterpret_cast<const float4 *>(sx + i);
        prod = (((prod * (1.0f - o.x)) * (1.0f - o.y)) * (1.0f - o.z)) * (1.0f - o.w);
        sum += (f.x + f.y) + (f.z + f.w);
    }
    const float iprod = warp_incl_mul(prod);
    const float isum = warp_incl_add(sum);
    float E = __shfl_up_sync(kFull, iprod, 1);
    float q = __shfl_up_sync(kFull, isum, 1);
    if (lane == 0) {
        E = 1.0f;
        q = 0.0f;
    }
    const float pe0 = __shfl_sync(kFull, iprod, 31);
    float csum = 0.0f;
    for (int i = lo; i < hi; i += 4) {
        const float4 o = *reinterpret_cast<const float4 *>(sp + i), g = *reinterpret_cast<const float4 *>(sc + i),
                     f = *reinterpret_cast<const float4 *>(sx + i);
        float4 P, C;
        P.x = E * o.x;  // Algorithm 2
        E *= 1.0f - o.x;
        P.y = E * o.y;
        E *= 1.0f - o.y;
        P.z = E * o.z;
        E *= 1.0f - o.z;
        P.w = E * o.w;
        E *= 1.0f - o.w;
        C.x = q + g.x;  // Algorithm 3
        q += f.x;
        C.y = q + g.y;
        q += f.y;
        C.z = q + g.z;
        q += f.z;
        C.w = q + g.w;
        q += f.w;
        *reinterpret_cast<float4 *>(sp + i) = P;
        *reinterpret_cast<float4 *>(sc + i) = C;
        csum += (C.x + C.y) + (C.z + C.w);
    }
    if (want_d) {  // Algorithm 4: D_k = sum_{i<=k} C_i (the last lane's sum past n is not used)
        const float ic = warp_incl_add(csum);
        float Dacc = __shfl_up_sync(kFull, ic, 1);
        if (lane == 0) Dacc = 0.0f;
        for (int i = lo; i < hi; i += 4) {
            const float4 C = *reinterpret_cast<const float4 *>(sc + i);
            float4 D;
            D.x = Dacc + C.x;
            D.y = D.x + C.y;
            D.z = D.y + C.z;
            D.w = D.z + C.w;
            Dacc = D.w;
            *reinterpret_cast<float4 *>(sx + i) = D;
        }
    }
    __syncwarp();
    if (lane == 0) sc[n] = 0.0f;
    __syncwarp();
    return pe0;
}

// Warp-level work loop of the persistent evaluation kernels: calls f(item) for items 0 .. n-1,
// one warp per item. Without a queue the items are dealt out grid-stride; with one, each warp
// takes `chunk` consecutive items per atomic grab on the 64-bit counter, which must be zero at
// launch (the counter then ends at n + chunk * (number of warps)).
template <typename F>
__device__ __forceinline__ void for_each_item(long long n, unsigned long long *queue, int chunk, F &&f)
{
    const int lane = lane_id(), warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    if (queue) {
        for (;;) {
            unsigned long long b0 = 0;
            if (lane == 0) b0 = atomicAdd(queue, (unsigned long long)chunk);
            b0 = __shfl_sync(kFull, b0, 0);
            if ((long long)b0 >= n) break;
            const long long b1 = min((long long)b0 + chunk, n);
            for (long long i = (long long)b0; i < b1; ++i) f(i);
        }
    } else {
        for (long long i = (long long)blockIdx.x * wpb + warp; i < n; i += (long long)gridDim.x * wpb) f(i);
    }
}

// Lets an early launch behind this one start once every block has got here.
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Waits for the end of the launch before this one and for its writes (returns at once on a launch that was not
// early). The last statement of a kernel's block 0 makes the kernel end no earlier than the one before it.
__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

struct EndAfterPrevious {
    bool on;
    __device__ __forceinline__ ~EndAfterPrevious()
    {
        if (on) wait_previous();
    }
};

__device__ __forceinline__ void set_status(int *status, int bits)
{
    if (status) atomicOr(status, bits);
}

}  // namespace fsmi
