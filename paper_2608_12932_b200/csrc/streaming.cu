// Two pieces of streaming prefill that sit beside the quantised linears (Sec. 3.1, "Streaming design").
//
// rope_shifted_keys_kernel: keys are cached BEFORE the rotary embedding, because a cached token's position changes
// when the window slides (what was at p is now at p - delta); the rotation is applied when the keys are used, at
// the shifted positions.  Rotate-half form: with i < D/2, theta_i = base^(-2i/D), phi = (pos[t] - delta) theta_i,
//   out[i] = k[i] cos(phi) - k[i + D/2] sin(phi),   out[i + D/2] = k[i + D/2] cos(phi) + k[i] sin(phi).
// One warp per token and all its heads (the angles do not depend on the head).  The angle is formed in fp64, as a number
// of half turns, and reduced to [-1, 1] there (a position of several thousand times theta_0 = 1 has no bits to spare in
// fp32); sine and cosine of pi times it are taken in fp32, products and sums in fp32, one rounding to bf16.  Both forms
// below do this with the same numbers in the same order, so that a key's rotation does not depend on which of them a
// window's size selects.
// Memory-bound: 2 B in and 2 B out per element.  The wide form takes 16 bytes per lane and half row; a lane's eight
// neighbouring elements are not the ones whose angles it computed, so a token's sines and cosines go through a small
// table in shared memory, and theta comes from the host (64 fp64 exponentials in front of a CTA's first load cost a
// microsecond of latency).  The 4-byte form (any D, any alignment, and few tokens) keeps everything in the lane; its theta
// come from the host too where the wide form could be taken for another window (D <= 2 ROPE_MAX_HALF).
//
// streaming_mask_kernel: the new frame's tokens are inserted at the last-frame place of each camera view (the
// sequence is view-major), only they are queries, and attention stays causal in that order:
//   mask[q][j] = (j <= position of query q),  position of query (v, i) = ((v F + F - 1) n + i).
#include <cuda_bf16.h>
#include <cmath>
#include <type_traits>
#include "ptx_sm100.cuh"
#include "w4a8_internal.cuh"

namespace w4a8 {
namespace {

constexpr int ROPE_WARPS = 8;
constexpr int ROPE_MAX_HALF = 128;
struct RopeTheta { double t[ROPE_MAX_HALF]; };               // theta_i / pi

// The 4-byte form's angle and rotation: the operations of the wide form, each multiply-add as the compiler contracts it there
// (the wide form spells them out in place; through these functions it is 0.5 to 1 % slower: 32768 x 8 x 128 25.2 and 25.5 us).
// (cos, sin) of q theta_i
__device__ __forceinline__ float2 rope_cos_sin(double q, double theta_over_pi) {
    const double a = __dmul_rn(q, theta_over_pi);
    float2 cs;
    sincospif((float)__fma_rn(-2.0, rint(0.5 * a), a), &cs.y, &cs.x);
    return cs;
}
// x, y: two neighbouring elements of the first and of the second half of a row; returns their rotation in place
__device__ __forceinline__ void rope_rotate2(uint32_t& x, uint32_t& y, float c0, float s0, float c1, float s1) {
    const float x0 = __uint_as_float(x << 16), x1 = __uint_as_float(x & 0xFFFF0000u);
    const float y0 = __uint_as_float(y << 16), y1 = __uint_as_float(y & 0xFFFF0000u);
    x = ptx::pack_bf16x2(fmaf(x0, c0, -__fmul_rn(y0, s0)), fmaf(x1, c1, -__fmul_rn(y1, s1)));
    y = ptx::pack_bf16x2(fmaf(x0, s0, __fmul_rn(y0, c0)), fmaf(x1, s1, __fmul_rn(y1, c1)));
}

// TABLE: theta from the host; otherwise (longer half rows) from base ^ (-2 i / D) here.  Eight heads at a time, the rest by
// code of their own lengths, and four CTAs per SM: with a bounds check per head the compiler keeps 128 to 200 registers of
// addresses and loads, at half the warps per SM and up to twice the time.  Measured on B200, the angle in radians with checks
// against this form: 4000 x 8 x 128 5.7 and 4.8 us, 8192 x 4 x 64 6.7 and 5.3, 30000 x 2 x 272 36.2 and 27.0.
template <bool TABLE>
__global__ void __launch_bounds__(ROPE_WARPS * 32, 4)
rope_shifted_keys_kernel(const uint32_t* __restrict__ k_pre, const int32_t* __restrict__ pos, int delta, int T, int H, int D,
                         double log2_base, const __grid_constant__ RopeTheta theta, uint32_t* __restrict__ k_rot) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int half = D >> 1, pairs = half >> 1;              // 32-bit words (two bf16) per half row
    __shared__ double th[TABLE ? ROPE_MAX_HALF : 1];         // once per CTA: lanes reading a parameter each at its own index take turns
    if (TABLE) {
        for (int i = threadIdx.x; i < half; i += ROPE_WARPS * 32) th[i] = theta.t[i];
        __syncthreads();
    }
    for (int w0 = lane; w0 < pairs; w0 += 32) {
        // this lane's elements i = 2 w0 and 2 w0 + 1 of the first half and their partners in the second
        constexpr double INV_PI = 0.31830988618379067154;
        const double th0 = TABLE ? th[2 * w0] : exp2(-(double)(4 * w0) / (double)D * log2_base) * INV_PI;
        const double th1 = TABLE ? th[2 * w0 + 1] : exp2(-(double)(4 * w0 + 2) / (double)D * log2_base) * INV_PI;
        // a warp per token: the angles do not depend on the head, so sine and cosine are taken once for all H rows
        for (int t = blockIdx.x * ROPE_WARPS + warp; t < T; t += gridDim.x * ROPE_WARPS) {
            const double p = (double)(__ldg(pos + t) - delta);
            const float2 r0 = rope_cos_sin(p, th0), r1 = rope_cos_sin(p, th1);
            const uint32_t* src = k_pre + (size_t)t * H * half + w0;
            uint32_t* dst = k_rot + (size_t)t * H * half + w0;
            auto heads = [&](auto count) {
                constexpr int C = decltype(count)::value;
                uint32_t lo[C], hi[C];
#pragma unroll
                for (int j = 0; j < C; ++j) { lo[j] = __ldg(src + j * half); hi[j] = __ldg(src + j * half + pairs); }
#pragma unroll
                for (int j = 0; j < C; ++j) {
                    rope_rotate2(lo[j], hi[j], r0.x, r0.y, r1.x, r1.y);
                    dst[j * half] = lo[j];
                    dst[j * half + pairs] = hi[j];
                }
                src += C * half;
                dst += C * half;
            };
            int h = 0;
            for (; h + 8 <= H; h += 8) heads(std::integral_constant<int, 8>());
            if (H & 4) heads(std::integral_constant<int, 4>());
            if (H & 2) heads(std::integral_constant<int, 2>());
            if (H & 1) heads(std::integral_constant<int, 1>());
        }
    }
}

// The form for many tokens, half rows of 8 n <= ROPE_MAX_HALF elements and 16-byte-aligned keys: a warp per token, U pairs
// of 16-byte pieces per lane (first and second half of a row) at a time.  Swept on B200: U = 2 and four warps per CTA, a CTA
// for every four tokens (persistent warps with the next token's keys requested ahead lose more to their uneven last round).
constexpr int ROPE_WIDE_WARPS = 4;
constexpr long long ROPE_WIDE_MIN_ELEMENTS = 4 << 20;
__global__ void __launch_bounds__(ROPE_WIDE_WARPS * 32)
rope_shifted_keys_wide_kernel(const uint4* __restrict__ k_pre, const int32_t* __restrict__ pos, int delta, int T, int H, int D,
                              const __grid_constant__ RopeTheta theta, uint4* __restrict__ k_rot) {
    constexpr int U = 2, WARPS = ROPE_WIDE_WARPS;
    __shared__ __align__(16) float2 rot[WARPS][ROPE_MAX_HALF];      // (cos, sin) of the warp's token, read two at a time
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int half = D >> 1, pieces = half >> 3;             // 16-byte pieces per half row
    const int total = H * pieces;                            // ... per token and half
    ptx::pdl_launch_dependents();
    const int t = blockIdx.x * WARPS + warp;
    __shared__ double th[ROPE_MAX_HALF];
    for (int i = threadIdx.x; i < half; i += WARPS * 32) th[i] = theta.t[i];
    __syncthreads();
    ptx::pdl_wait();
    if (t >= T) return;
    const int p = __ldcg(pos + t);
    const size_t row0 = (size_t)t * total * 2;
    for (int base = 0; base < total; base += 32 * U) {
        uint4 lo[U], hi[U];
        size_t at[U];
        int w[U];
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int idx = base + lane + 32 * k, head = idx / pieces;
            w[k] = idx - head * pieces;
            at[k] = row0 + head * (2 * pieces) + w[k];
            if (idx < total) {
                lo[k] = __ldcg(k_pre + at[k]);
                hi[k] = __ldcg(k_pre + at[k] + pieces);
            }
        }
        if (base == 0) {
            const double q = (double)(p - delta);
            for (int i = lane; i < half; i += 32) {
                double a = q * th[i];
                a -= 2.0 * rint(0.5 * a);
                float2 cs;
                sincospif((float)a, &cs.y, &cs.x);
                rot[warp][i] = cs;
            }
            __syncwarp();
        }
#pragma unroll
        for (int k = 0; k < U; ++k) {
            if (base + lane + 32 * k < total) {
                const float4* cs = reinterpret_cast<const float4*>(&rot[warp][8 * w[k]]);
                uint32_t ox[4], oy[4];
                const uint32_t xs[4] = {lo[k].x, lo[k].y, lo[k].z, lo[k].w}, ys[4] = {hi[k].x, hi[k].y, hi[k].z, hi[k].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float4 c = cs[e];                  // cos, sin of element 2 e, then of 2 e + 1
                    const float x0 = __uint_as_float(xs[e] << 16), x1 = __uint_as_float(xs[e] & 0xFFFF0000u);
                    const float y0 = __uint_as_float(ys[e] << 16), y1 = __uint_as_float(ys[e] & 0xFFFF0000u);
                    const __nv_bfloat162 olo = __floats2bfloat162_rn(x0 * c.x - y0 * c.y, x1 * c.z - y1 * c.w);
                    const __nv_bfloat162 ohi = __floats2bfloat162_rn(y0 * c.x + x0 * c.y, y1 * c.z + x1 * c.w);
                    ox[e] = *reinterpret_cast<const uint32_t*>(&olo);
                    oy[e] = *reinterpret_cast<const uint32_t*>(&ohi);
                }
                k_rot[at[k]] = make_uint4(ox[0], ox[1], ox[2], ox[3]);
                k_rot[at[k] + pieces] = make_uint4(oy[0], oy[1], oy[2], oy[3]);
            }
        }
    }
}

__global__ void __launch_bounds__(256)
streaming_mask_kernel(int V, int F, int n, uint8_t* __restrict__ mask) {
    const long long kv = (long long)V * F * n, total = (long long)V * n * kv;
    for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += (long long)gridDim.x * blockDim.x) {
        const long long q = idx / kv, j = idx - q * kv;
        const long long v = q / n, i = q - v * n;
        const long long p = (v * F + F - 1) * n + i;
        mask[idx] = j <= p ? 1 : 0;
    }
}

}  // namespace

cudaError_t launch_rope_shifted_keys(const void* k_pre, const int32_t* pos, int delta, int T, int H, int D, double base,
                                     void* k_rot, cudaStream_t stream) {
    int grid = (T + ROPE_WARPS - 1) / ROPE_WARPS;
    const bool table = D <= 2 * ROPE_MAX_HALF;
    const double log2_base = log2(base);
    RopeTheta theta;
    for (int i = 0; table && i < D / 2; ++i) theta.t[i] = exp2(-(double)(2 * i) / (double)D * log2_base) * 0.31830988618379067154;
    // Measured on B200 (cold keys, 4-byte and wide form, us, back to back in a graph): 16384 x 8 x 64 10.6 and 7.9, 16384 x 16 x 64 15.6
    // and 11.3, 32768 x 16 x 32 27.7 and 13.0, 8192 x 4 x 128 6.2 and 5.3, 2048 x 8 x 128 3.4 and 4.4.  From 8 Mi elements of D = 128 on,
    // where a half row fills a warp of 4-byte accesses, the 4-byte kernel itself is the quicker one (16384 x 8 x 128 11.3 and 13.3), but
    // not in a stream of eager calls, where it does not start under its predecessor (14.6 and 14.2).
    if ((long long)T * H * D >= ROPE_WIDE_MIN_ELEMENTS && D % 16 == 0 && table && ((reinterpret_cast<uintptr_t>(k_pre) | reinterpret_cast<uintptr_t>(k_rot)) & 15) == 0) {
        cudaLaunchConfig_t cfg = {};
        cfg.stream = stream;
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        cfg.gridDim = dim3((unsigned)((T + ROPE_WIDE_WARPS - 1) / ROPE_WIDE_WARPS), 1, 1);
        cfg.blockDim = dim3(ROPE_WIDE_WARPS * 32, 1, 1);
        return cudaLaunchKernelEx(&cfg, rope_shifted_keys_wide_kernel, static_cast<const uint4*>(k_pre), pos, delta, T, H, D, theta,
                                  static_cast<uint4*>(k_rot));
    }
    const int cap = device_sm_count() * 8;
    if (grid > cap) grid = cap;
    if (table)
        rope_shifted_keys_kernel<true><<<grid, ROPE_WARPS * 32, 0, stream>>>(static_cast<const uint32_t*>(k_pre), pos, delta, T, H, D,
                                                                             log2_base, theta, static_cast<uint32_t*>(k_rot));
    else
        rope_shifted_keys_kernel<false><<<grid, ROPE_WARPS * 32, 0, stream>>>(static_cast<const uint32_t*>(k_pre), pos, delta, T, H, D,
                                                                              log2_base, theta, static_cast<uint32_t*>(k_rot));
    return cudaGetLastError();
}

cudaError_t launch_streaming_mask(int V, int F, int n, uint8_t* mask, cudaStream_t stream) {
    const long long total = (long long)V * n * V * F * n;
    long long grid = (total + 255) / 256;
    const long long cap = (long long)device_sm_count() * 8;
    if (grid > cap) grid = cap;
    streaming_mask_kernel<<<(unsigned)grid, 256, 0, stream>>>(V, F, n, mask);
    return cudaGetLastError();
}

}  // namespace w4a8
