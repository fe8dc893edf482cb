// Two pieces of streaming prefill that sit beside the quantised linears (Sec. 3.1, "Streaming design").
//
// rope_shifted_keys_kernel: keys are cached BEFORE the rotary embedding, because a cached token's position changes
// when the window slides (what was at p is now at p - delta); the rotation is applied when the keys are used, at
// the shifted positions.  Rotate-half form: with i < D/2, theta_i = base^(-2i/D), phi = (pos[t] - delta) theta_i,
//   out[i] = k[i] cos(phi) - k[i + D/2] sin(phi),   out[i + D/2] = k[i + D/2] cos(phi) + k[i] sin(phi).
// One warp per token and all its heads (the angles do not depend on the head).  The angle is formed in fp64, as a number
// of half turns, and reduced to [-1, 1] there (a position of several thousand times theta_0 = 1 has no bits to spare in
// fp32); sine and cosine of pi times it are taken in fp32, products and sums in fp32, one rounding to bf16.
// Memory-bound: 2 B in and 2 B out per element.  The wide form takes 16 bytes per lane and half row; a lane's eight
// neighbouring elements are not the ones whose angles it computed, so a token's sines and cosines go through a small
// table in shared memory, and theta comes from the host (64 fp64 exponentials in front of a CTA's first load cost a
// microsecond of latency).  The 4-byte form (any D, any alignment, and few tokens) keeps everything in the lane.
//
// streaming_mask_kernel: the new frame's tokens are inserted at the last-frame place of each camera view (the
// sequence is view-major), only they are queries, and attention stays causal in that order:
//   mask[q][j] = (j <= position of query q),  position of query (v, i) = ((v F + F - 1) n + i).
#include <cuda_bf16.h>
#include <cmath>
#include "ptx_sm100.cuh"
#include "w4a8_internal.cuh"

namespace w4a8 {
namespace {

constexpr int ROPE_WARPS = 8;

__global__ void __launch_bounds__(ROPE_WARPS * 32)
rope_shifted_keys_kernel(const uint32_t* __restrict__ k_pre, const int32_t* __restrict__ pos, int delta, int T, int H, int D,
                         double log2_base, uint32_t* __restrict__ k_rot) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int half = D >> 1, pairs = half >> 1;              // 32-bit words (two bf16) per half row
    const double two_pi = 6.283185307179586476925286766559, inv_two_pi = 0.15915494309189533576888376337251;
    for (int w0 = lane; w0 < pairs; w0 += 32) {
        // this lane's elements i = 2 w0 and 2 w0 + 1 of the first half and their partners in the second
        const double th0 = exp2(-(double)(4 * w0) / (double)D * log2_base), th1 = exp2(-(double)(4 * w0 + 2) / (double)D * log2_base);
        // a warp per token: the angles do not depend on the head, so sine and cosine are taken once for all H rows
        for (int t = blockIdx.x * ROPE_WARPS + warp; t < T; t += gridDim.x * ROPE_WARPS) {
            const double p = (double)(__ldg(pos + t) - delta);
            double a0 = p * th0, a1 = p * th1;
            a0 -= two_pi * rint(a0 * inv_two_pi);
            a1 -= two_pi * rint(a1 * inv_two_pi);
            float s0, c0, s1, c1;
            sincosf((float)a0, &s0, &c0);
            sincosf((float)a1, &s1, &c1);
            for (int h0 = 0; h0 < H; h0 += 8) {
                uint32_t lo[8], hi[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const size_t base_w = ((size_t)t * H + h0 + j) * (D >> 1);
                    if (h0 + j < H) { lo[j] = __ldg(k_pre + base_w + w0); hi[j] = __ldg(k_pre + base_w + pairs + w0); }
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    if (h0 + j >= H) break;
                    const size_t base_w = ((size_t)t * H + h0 + j) * (D >> 1);
                    const float x0 = __uint_as_float(lo[j] << 16), x1 = __uint_as_float(lo[j] & 0xFFFF0000u);
                    const float y0 = __uint_as_float(hi[j] << 16), y1 = __uint_as_float(hi[j] & 0xFFFF0000u);
                    const __nv_bfloat162 olo = __floats2bfloat162_rn(x0 * c0 - y0 * s0, x1 * c1 - y1 * s1);
                    const __nv_bfloat162 ohi = __floats2bfloat162_rn(y0 * c0 + x0 * s0, y1 * c1 + x1 * s1);
                    k_rot[base_w + w0] = *reinterpret_cast<const uint32_t*>(&olo);
                    k_rot[base_w + pairs + w0] = *reinterpret_cast<const uint32_t*>(&ohi);
                }
            }
        }
    }
}

// The form for many tokens, half rows of 8 n <= ROPE_MAX_HALF elements and 16-byte-aligned keys: a warp per token, U pairs
// of 16-byte pieces per lane (first and second half of a row) at a time.  Swept on B200: U = 2 and four warps per CTA, a CTA
// for every four tokens (persistent warps with the next token's keys requested ahead lose more to their uneven last round).
constexpr int ROPE_MAX_HALF = 128, ROPE_WIDE_WARPS = 4;
constexpr long long ROPE_WIDE_MIN_ELEMENTS = 4 << 20;
struct RopeTheta { double t[ROPE_MAX_HALF]; };               // theta_i / pi
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
                const uint32_t xs[4] = {lo[k].x, lo[k].y, lo[k].z, lo[k].w}, ys[4] = {hi[k].x, hi[k].y, hi[k].z, hi[k].w};
                uint32_t ox[4], oy[4];
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
    // measured on B200 (cold keys, 4-byte -> wide form): 30000 x 16 x 64 35.8 -> 21.6 us, 16384 x 8 x 128 15.4 -> 13.7, 65536 x 8 x 128
    // 48.5 -> 47.8; 2000 x 8 x 128 3.6 -> 4.4 (one wave of CTAs: the shorter latency chain of the 4-byte form wins)
    if ((long long)T * H * D >= ROPE_WIDE_MIN_ELEMENTS && D % 16 == 0 && D <= 2 * ROPE_MAX_HALF && ((reinterpret_cast<uintptr_t>(k_pre) | reinterpret_cast<uintptr_t>(k_rot)) & 15) == 0) {
        cudaLaunchConfig_t cfg = {};
        cfg.stream = stream;
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        RopeTheta theta;
        for (int i = 0; i < D / 2; ++i) theta.t[i] = exp2(-(double)(2 * i) / (double)D * log2(base)) * 0.31830988618379067154;
        cfg.gridDim = dim3((unsigned)((T + ROPE_WIDE_WARPS - 1) / ROPE_WIDE_WARPS), 1, 1);
        cfg.blockDim = dim3(ROPE_WIDE_WARPS * 32, 1, 1);
        return cudaLaunchKernelEx(&cfg, rope_shifted_keys_wide_kernel, static_cast<const uint4*>(k_pre), pos, delta, T, H, D, theta,
                                  static_cast<uint4*>(k_rot));
    }
    const int cap = device_sm_count() * 8;
    if (grid > cap) grid = cap;
    rope_shifted_keys_kernel<<<grid, ROPE_WARPS * 32, 0, stream>>>(static_cast<const uint32_t*>(k_pre), pos, delta, T, H, D,
                                                                   log2(base), static_cast<uint32_t*>(k_rot));
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
