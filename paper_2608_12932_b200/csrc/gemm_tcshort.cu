// W4A8 GEMM on the tensor cores for token tiles of 64 rows (17 to a few hundred tokens, layers of more than four groups;
// up to 32 tokens any layer): the scheme of
// gemm_tcgen05.cu - weights as bytes in tensor memory, tokens on the MMA's N side, one drain per quantisation group.
// (Sec. 3.4: INT8 tensor cores; Sec. 4: between decode and prefill a call is bound by neither alone.)
//
// What bounds a short tile is not HBM (a blob every 383 cycles is an SM's share) nor the tensor pipe (a group's MMAs
// take 328 cycles, each reading 4 KB of weights out of tensor memory, however few tokens it multiplies) but
// instructions on the CUDA cores and the barrier round trips between them: every accumulator element is converted and
// scaled once per group, every weight is unpacked once per token tile, and all of it shares four schedulers and a
// half-rate integer pipe.  Hence
//  * THE FIFTH K SLICE.  A group is four MMAs of K = 32 over the codes 0..15 as they are, and one more MMA of K = 32
//    whose operands carry the zero points and an accumulator bias:
//        weights      [ -8z x 16 | -z | -128 x 15 ]          activations  [ A >> 7 x 16 | A & 127 | -128 x 15 ]
//    with A = sum q_a of the (token, group): the slice adds -z A + 15 * 2^14, so the accumulator is D + 245760 exactly
//    and always positive (|D| <= 243840).  The unpack is left with a mask (and a shift for the high nibbles):
//    48 integer instructions per row and group instead of 112.  The drain is left with no conversion: the bits of a
//    small positive integer n ARE the float n * 2^-149, so one packed add of -245760 * 2^-149 (exact) and one packed
//    FMA with the group scale times 2^100 replace two conversions and two FMAs; the sums run at 2^-49 of their value,
//    every rounding as without it, and the token scale takes the factor out.
//  * a pipeline step is TWO groups (one bulk copy of two neighbouring blobs, one 3-D TMA box with both groups'
//    activations, one weight stage) and two teams of four unpack warps take the steps in turn: a barrier round trip
//    costs a role 100-150 cycles, which a short tile cannot hide any other way;
//  * the unpack threads hand the group scales on through a small shared-memory ring: the drain reads nothing from
//    global memory inside the loop;
//  * the MMA's N is the tile's own token count rounded up to 16, a drain warp whose columns lie past the last token
//    only passes the barriers on, and up to 32 tokens the tile is cut to 32 columns;
//  * a K split exchanges its partials 16 bytes at a time (four tokens of a channel) and stores its sums 128 bytes a row,
//    with the residual requested ahead of the exchange's second barrier (2 bytes a lane and the residual after it:
//    12288 -> 4096 with residual at 64 tokens in four slices 13.4 us, now 12.7; 4096 -> 4096 in two 9.6, now 8.6).
// Measured on B200 (one 128-channel tile per SM, slope over K): 349 -> 253 ns a group at 64 tokens, 349 -> 226 at 32
// tokens (4.4 TB/s of weights); 64 tokens, 4096 -> 6144 behind the quantiser 14.7 -> 12.0 us, 12288 -> 4096 18.9 -> 16.1.
// Of the parts, two groups a step alone made it slower (448 ns): it is the instruction count that has to fall.
// A 128-row form was slower than the one-group pipeline (513 against 448 ns a group) and a 208-row form far slower
// (820 against 528): the packed sums need aligned register pairs, and that many of them beside as many loaded columns
// leave the compiler copying registers.
//
// Warp roles (640 threads):
//   warp 0   activation tiles (3-D TMA loads)       warp 1   MMA issuer (elected lane), TMEM allocation
//   warp 2   packed blobs (bulk copies)             warp 3   the activations' part of the fifth K slice, from asum
//   warps 4-11   unpack: two teams, a thread per weight row (= TMEM lane)
//   warps 12-19  drain: lanes = channels, two column halves
//
// Work distribution (whole tiles, K split over a cluster, balanced walk) and its reductions are those of
// gemm_tcgen05.cu.  Every wait is bounded; on expiry the CTA records W4A8_ERR_TIMEOUT, frees TMEM and exits.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include "ptx_sm100.cuh"
#include "w4a8_internal.cuh"

namespace w4a8 {
namespace {

constexpr int TS_THREADS = 640;
constexpr int WARP_ACT = 0, WARP_MMA = 1, WARP_BLOB = 2, WARP_SLICE = 3, WARP_UNPACK0 = 4, WARP_DRAIN0 = 12;
constexpr int NUM_DRAIN_WARPS = 8, TEAM_WARPS = 4;
constexpr int DONE_RING = 8;                          // "done" barriers; no role is further than this from another
constexpr int SCALE_RING = 8;                         // steps whose group scales are kept for the drain
constexpr int TMEM_COLS = 512;
constexpr int SLICE_K = 32;                           // bytes per row of the fifth K slice
constexpr uint32_t ACC_BIAS = 15u << 14;              // what the slice's constant part adds: 15 x (-128) x (-128)
constexpr float SCALE_UP = 1.2676506002282294e30f;    // 2^100, on the group scales (the accumulators are worth 2^-149 of their bits)
constexpr float SCALE_OUT = 562949953421312.0f;       // 2^49, on the token scales
template <int TILE_M>
struct Cfg {
    static constexpr int GPS = 2;                                             // groups per pipeline step
    static constexpr int NBU = 2;                                             // accumulator buffers (of a step's two groups)
    static constexpr int A_G = (GROUP + SLICE_K) / 4;                         // TMEM columns of a group's weight rows
    static constexpr int A_COLS = GPS * A_G;
    static constexpr int A_COL0 = NBU * GPS * TILE_M;
    static constexpr int SA = TILE_M == 64 ? (TMEM_COLS - A_COL0) / A_COLS : 4;   // weight stages
    static constexpr int SB = 4;                                              // activation stages
    static constexpr int SR = TILE_M == 64 ? 7 : 9;                           // blob-pair stages: over 100 KB in flight
    static constexpr int RAW_BYTES = GPS * BLOB_BYTES;                        // 17 024 = 133 x 128
    static constexpr int B_BYTES = GPS * TILE_M * GROUP;                      // activations of a step
    static constexpr int X_BYTES = GPS * TILE_M * SLICE_K;                    // their part of the fifth slice
    static constexpr int X_OFF = SB * B_BYTES;
    static constexpr int RAW_OFF = X_OFF + SB * X_BYTES;
    static constexpr int BAR_OFF = RAW_OFF + SR * RAW_BYTES;
    static constexpr int NUM_BARS = 2 * SR + SB + SA + NBU + DONE_RING + 1;
    static constexpr int MISC_OFF = (BAR_OFF + NUM_BARS * 8 + 15) & ~15;
    static constexpr int W = TILE_M / 2;                                      // tokens per drain warp
    static constexpr int SCALE_OFF = MISC_OFF + 16;                           // [step % SCALE_RING][group][channel] fp16
    static constexpr int SA_OFF = SCALE_OFF + SCALE_RING * GPS * TILE_N * 2;  // per drain warp: token scales as fp32
    static constexpr int OUT_OFF = (SA_OFF + NUM_DRAIN_WARPS * W * 4 + 127) & ~127;   // per drain warp: 32 tokens x 32 channels bf16
    static constexpr int SMEM_BYTES = OUT_OFF + NUM_DRAIN_WARPS * 2048;
    static constexpr int SMEM_ALLOC = SMEM_BYTES + 1024;                      // slack to align the base to 1024 B
    static_assert(TILE_M == 64 || TILE_M == 32, "token tile");
    static_assert(SA >= 2 && A_COL0 + SA * A_COLS <= TMEM_COLS, "tensor memory");
    static_assert(SB < DONE_RING && SA < DONE_RING && NBU < DONE_RING, "a stage is freed by the step that used it, at most DONE_RING steps ago");
    static_assert(SA + NBU <= SCALE_RING, "a scale slot is rewritten only after the drain has passed the step that used it");
    static_assert(BAR_OFF >= 4 * ((TILE_M / 4 + 3) / 4 + 1) * TILE_N * 16 && BAR_OFF >= TILE_M * TILE_N * 4, "the split-K exchange buffer lives in the rings");
    static_assert((TILE_M * GROUP) % 1024 == 0 && X_OFF % 128 == 0 && RAW_OFF % 128 == 0 && RAW_BYTES % 128 == 0, "alignment");
    static_assert(SCALE_OFF % 16 == 0 && SA_OFF % 16 == 0, "alignment");
    static_assert(SMEM_ALLOC <= 227 * 1024, "shared memory");
};

// RES: the epilogue adds a residual (its own instantiations: the plain kernels keep their registers).
template <int TILE_M, bool DEBUG, bool SPLIT, bool BAL, bool RES>
__global__ void __launch_bounds__(TS_THREADS, 1)
gemm_tcshort_kernel(const __grid_constant__ CUtensorMap tmap_qa, const __grid_constant__ CUtensorMap tmap_y,
                    const uint8_t* __restrict__ packed, const uint16_t* __restrict__ sa, const int32_t* __restrict__ asum,
                    __nv_bfloat16* y, const __nv_bfloat16* residual, int32_t* __restrict__ debug_partials,
                    uint32_t* __restrict__ status, int M, int N, int K, int m_tiles, int total_tiles, int S,
                    float* __restrict__ handover, uint32_t* __restrict__ handover_flags) {
    // Programmatic dependent launch: set-up and the weight stream may run under the previous kernel; the roles that
    // touch activations, their scales and sums, the workspace or the output wait below.
    ptx::pdl_launch_dependents();
    using C = Cfg<TILE_M>;
    static_assert(!(SPLIT && BAL), "one work distribution");
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem = smem_raw + (smem_base - ptx::smem_u32(smem_raw));
    const int GK = K / GROUP;                                   // groups of the whole K range (blob and output indexing)
    // The warp index comes out of a shuffle: the compiler then knows it to be warp-uniform and keeps ring indices, barrier and
    // tensor-memory addresses on the uniform datapath (B200, before and after: 4096 -> 24576 at 40 and 64 tokens 19.7 and 19.9 us, 18.9
    // and 19.2; 4096 -> 6144 at 40 9.7, 9.4).
    const int tid = threadIdx.x, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0), lane = tid & 31;
    const int slice = SPLIT ? (int)ptx::cluster_ctarank() : 0;
    const int unit = SPLIT ? (int)blockIdx.x / S : (int)blockIdx.x;
    const int num_units = SPLIT ? (int)gridDim.x / S : (int)gridDim.x;
    const int g_lo = SPLIT ? (int)(((long long)slice * GK) / S) : 0;
    const int G = SPLIT ? (int)(((long long)(slice + 1) * GK) / S) - g_lo : GK;

    auto bar = [&](int i) { return smem_base + C::BAR_OFF + 8 * i; };
    // DONE[st % DONE_RING]: the MMAs of pipeline step st have finished - its weight and activation stages are free, its
    // accumulators complete
    const int RAW_FULL = 0, RAW_EMPTY = C::SR, B_FULL = 2 * C::SR, A_FULL = B_FULL + C::SB, ACC_EMPTY = A_FULL + C::SA,
              DONE = ACC_EMPTY + C::NBU, FINAL = DONE + DONE_RING;
    auto step_bar = [&](uint32_t st) { return bar(DONE + (int)(st % DONE_RING)); };
    auto ring_parity = [](uint32_t i) { return (i / DONE_RING) & 1u; };
    volatile uint32_t* tmem_holder = reinterpret_cast<volatile uint32_t*>(smem + C::MISC_OFF);
    volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem + C::MISC_OFF + 4);

    if (warp == WARP_MMA) {
        if (lane == 0) {
            *abort_flag = 0;
            for (int i = 0; i < C::SR; ++i) {
                ptx::mbar_init(bar(RAW_FULL + i), 1);
                ptx::mbar_init(bar(RAW_EMPTY + i), TEAM_WARPS);
            }
            for (int i = 0; i < C::SB; ++i) ptx::mbar_init(bar(B_FULL + i), 2);       // the TMA box and the fifth slice
            for (int i = 0; i < C::SA; ++i) ptx::mbar_init(bar(A_FULL + i), TEAM_WARPS);
            for (int i = 0; i < C::NBU; ++i) ptx::mbar_init(bar(ACC_EMPTY + i), NUM_DRAIN_WARPS);
            for (int i = 0; i < DONE_RING + 1; ++i) ptx::mbar_init(bar(DONE + i), 1);
            ptx::fence_mbar_init();
        }
        __syncwarp();
        ptx::tmem_alloc(smem_base + C::MISC_OFF, TMEM_COLS);
        ptx::tmem_relinquish();
    }
    if (warp == WARP_ACT && lane == 0) ptx::prefetch_tmap(&tmap_qa);
    if (warp == WARP_DRAIN0 && lane == 0) ptx::prefetch_tmap(&tmap_y);
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_holder;
    auto tile_of = [&](int t, int& ntile, int& mtile) {
        ntile = t / m_tiles;
        mtile = t % m_tiles;
    };

    // The work of a CTA as a list of segments (tile, groups [gb, ge) of it).  Plain persistent walk: whole
    // tiles unit, unit + num_units, ...  Balanced walk (more tiles than CTAs): the tiles x groups units are
    // dealt out in equal contiguous ranges, so a CTA's first and last segment may be part of a tile; the CTA
    // that holds the later groups of such a tile reaches them first (they open its range) and hands its
    // fp32 sums over through global memory to the CTA that holds the earlier groups (they close its range).
    const long bal_lo = BAL ? ((long)blockIdx.x * total_tiles * G) / gridDim.x : 0;
    const int bal_n = BAL ? (int)(((long)(blockIdx.x + 1) * total_tiles * G) / gridDim.x - bal_lo) : 0;
    const int bal_tile = BAL ? (int)(bal_lo / G) : 0, bal_g = BAL ? (int)(bal_lo % G) : 0;
    auto segment = [&](int idx, int& tile, int& gb, int& ge) -> bool {
        if (BAL) {
            tile = bal_tile + idx;
            gb = idx == 0 ? bal_g : 0;
            const int left = bal_g + bal_n - idx * G;
            ge = left < G ? left : G;
            return gb < ge;
        }
        tile = unit + idx * num_units;
        gb = 0;
        ge = G;
        return tile < total_tiles;
    };

    bool exchanged = false;                     // SPLIT: this thread has passed the two cluster barriers
    constexpr int RUNS = TILE_M / 4;            // SPLIT: runs of four tokens; CTA o of the cluster reduces runs run_lo(o) .. run_lo(o + 1) - 1
    const int runs_max = SPLIT ? (RUNS + S - 1) / S : 0;
    auto run_lo = [&](int o) { return o * RUNS / S; };
    if (warp < WARP_UNPACK0) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
        if (warp == WARP_ACT && lane == 0) {
            // ------------------------------------------------ producer: activation tiles ----
            ptx::pdl_wait();                                    // the activations are the previous kernel's output
            uint32_t st = 0;
            bool ok = true;
            for (int si = 0; ok; ++si) {
                int tile, gb, ge, ntile, mtile;
                if (!segment(si, tile, gb, ge)) break;
                tile_of(tile, ntile, mtile);
                for (int g = gb; g < ge; g += C::GPS, ++st) {
                    const uint32_t sb = st % C::SB;
                    if (st >= (uint32_t)C::SB && !(ok = ptx::mbar_wait(step_bar(st - C::SB), ring_parity(st - C::SB), abort_flag))) break;
                    // the box always delivers GPS groups (zeros past the last one); a lone last group leaves the second unused
                    ptx::mbar_arrive_expect_tx(bar(B_FULL + sb), C::B_BYTES);
                    ptx::tma_load_3d(smem_base + sb * C::B_BYTES, &tmap_qa, 0, mtile * TILE_M, g_lo + g, bar(B_FULL + sb));
                }
            }
            if (!ok) {   // let copies already in flight land before shared memory is released
                const uint64_t t0 = ptx::globaltimer_ns();
                while (ptx::globaltimer_ns() - t0 < 200000ull) {}
            }
        } else if (warp == WARP_BLOB && lane == 0) {
            // --------------------------------------------------- producer: packed blobs ----
            uint32_t st = 0;
            bool ok = true;
            for (int si = 0; ok; ++si) {
                int tile, gb, ge, ntile, mtile;
                if (!segment(si, tile, gb, ge)) break;
                tile_of(tile, ntile, mtile);
                const uint8_t* src = packed + ((size_t)ntile * GK + g_lo) * BLOB_BYTES;
                for (int g = gb; g < ge; g += C::GPS, ++st) {
                    const uint32_t sr = st % C::SR, pr = (st / C::SR) & 1;
                    if (!(ok = ptx::mbar_wait(bar(RAW_EMPTY + sr), pr ^ 1, abort_flag))) break;
                    const uint32_t bytes = ge - g >= C::GPS ? C::RAW_BYTES : BLOB_BYTES;
                    ptx::mbar_arrive_expect_tx(bar(RAW_FULL + sr), bytes);
                    ptx::bulk_g2s(smem_base + C::RAW_OFF + sr * C::RAW_BYTES, src + (size_t)g * BLOB_BYTES, bytes, bar(RAW_FULL + sr));
                }
            }
            if (!ok) {
                const uint64_t t0 = ptx::globaltimer_ns();
                while (ptx::globaltimer_ns() - t0 < 200000ull) {}
            }
        } else if (warp == WARP_SLICE) {
            // ------------------------------- the activations' part of the fifth K slice ----
            // Row of token t: sixteen bytes A >> 7, then A & 127 and fifteen bytes -128; stored as two planes of 16 bytes
            // per token (core matrices of 8 rows x 16 bytes, no swizzle).  The sums of the step after the next are
            // requested before this step's are written: an L2 round trip is longer than a step.
            ptx::pdl_wait();                                    // the group sums are the previous kernel's output
            constexpr int NT = TILE_M / 32;
            int lsi = 0, lg, lge;                                // the segment and group that the next load belongs to
            bool lvalid;
            uint32_t lbase, lmask;                               // lane's first token: index into asum; which of its tokens exist
            auto enter = [&]() {
                int tile, gb;
                lvalid = segment(lsi, tile, gb, lge);
                lg = gb;
                const int m0 = (tile % m_tiles) * TILE_M + lane;
                lbase = (uint32_t)m0 * (uint32_t)GK + (uint32_t)(g_lo + gb);
                lmask = 0;
#pragma unroll
                for (int i = 0; i < NT; ++i) lmask |= (m0 + 32 * i < M ? 1u : 0u) << i;
            };
            enter();
            auto load = [&](int (&v)[C::GPS][NT]) -> bool {
                if (!lvalid) return false;
#pragma unroll
                for (int gg = 0; gg < C::GPS; ++gg) {
#pragma unroll
                    for (int i = 0; i < NT; ++i)
                        v[gg][i] = (lmask >> i & 1u) && lg + gg < lge ? __ldcg(asum + (lbase + (uint32_t)(i * 32 * GK + gg))) : 0;
                }
                lg += C::GPS;
                lbase += C::GPS;
                if (lg >= lge) { ++lsi; enter(); }
                return true;
            };
            uint32_t st = 0;
            auto one = [&](int (&v)[C::GPS][NT]) -> bool {
                const uint32_t sb = st % C::SB;
                if (st >= (uint32_t)C::SB && !ptx::mbar_wait(step_bar(st - C::SB), ring_parity(st - C::SB), abort_flag)) return false;
                const uint32_t dst = smem_base + C::X_OFF + sb * C::X_BYTES + lane * 16;
#pragma unroll
                for (int gg = 0; gg < C::GPS; ++gg) {
#pragma unroll
                    for (int i = 0; i < NT; ++i) {
                        {
                            const uint32_t hi = __byte_perm((uint32_t)(v[gg][i] >> 7), 0, 0x0000), lo = ((uint32_t)v[gg][i] & 127u) | 0x80808000u;
                            const uint32_t at = dst + gg * (TILE_M * SLICE_K) + i * 512;
                            ptx::sts128u(at, hi, hi, hi, hi);
                            ptx::sts128u(at + TILE_M * 16, lo, 0x80808080u, 0x80808080u, 0x80808080u);
                        }
                    }
                }
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(bar(B_FULL + sb));
                ++st;
                return true;
            };
            int v0[C::GPS][NT], v1[C::GPS][NT];
            bool have0 = load(v0), have1 = load(v1);
            while (have0) {
                if (!one(v0)) break;
                have0 = load(v0);
                if (!have1 || !one(v1)) break;
                have1 = load(v1);
            }
        } else if (warp == WARP_MMA) {
            // ----------------------------------------------------------------- MMA issuer ----
            // The whole warp walks the loop and one elected lane issues: with warp-uniform control flow the MMA operands
            // are computed once per warp in uniform registers, which is where the tensor instructions take them from.
            const uint32_t tmem_u = __shfl_sync(0xFFFFFFFFu, tmem_base, 0);
            const uint64_t b_desc0 = ptx::smem_desc_k_sw128(smem_base);
            const uint64_t x_desc0 = ptx::smem_desc_k_none(smem_base + C::X_OFF, TILE_M * 16, 128);
            uint32_t st = 0;
            bool ok = true;
            for (int si = 0; ok; ++si) {
                int tile, gb, ge, ntile, mtile;
                if (!segment(si, tile, gb, ge)) break;
                tile_of(tile, ntile, mtile);
                // N of the MMA: the tile's tokens, rounded up to 16
                const int rows = M - mtile * TILE_M;
                const uint32_t mma_n = __shfl_sync(0xFFFFFFFFu, rows >= TILE_M ? TILE_M : ((rows + 15) & ~15), 0);
                const uint32_t idesc = ptx::idesc_i8(TILE_N, 0, true, true) | ((mma_n >> 3) << 17);
                for (int g = gb; g < ge; g += C::GPS, ++st) {
                    const uint32_t sb = st % C::SB, sa_ = st % C::SA, ub = st % C::NBU;
                    const int ng = ge - g >= C::GPS ? C::GPS : 1;
                    if (!(ok = ptx::mbar_wait(bar(B_FULL + sb), (st / C::SB) & 1, abort_flag))) break;
                    if (!(ok = ptx::mbar_wait(bar(A_FULL + sa_), (st / C::SA) & 1, abort_flag))) break;
                    if (!(ok = ptx::mbar_wait(bar(ACC_EMPTY + ub), (st / C::NBU) & 1, abort_flag))) break;
                    ptx::tc_fence_after_sync();
                    const uint64_t bd0 = b_desc0 + (uint64_t)(sb * (C::B_BYTES / 16)), xd0 = x_desc0 + (uint64_t)(sb * (C::X_BYTES / 16));
                    const uint32_t a0 = tmem_u + C::A_COL0 + sa_ * C::A_COLS, d0 = tmem_u + ub * (C::GPS * TILE_M);
                    const uint32_t done = step_bar(st);
                    if (ptx::elect_one()) {
#pragma unroll
                        for (int gg = 0; gg < C::GPS; ++gg) {
                            const uint64_t bd = bd0 + (uint64_t)(gg * (TILE_M * GROUP / 16)), xd = xd0 + (uint64_t)(gg * (TILE_M * SLICE_K / 16));
                            const uint32_t a_tmem = a0 + gg * C::A_G, d_tmem = d0 + gg * TILE_M;
                            // the fifth slice first: it overwrites the buffer (a second group that is not there: D = 0)
                            ptx::mma_i8_ts(d_tmem, a_tmem + GROUP / 4, xd, idesc, 0u);
                            if (gg < ng) {
#pragma unroll
                                for (int kk = 0; kk < GROUP / 32; ++kk) ptx::mma_i8_ts(d_tmem, a_tmem + 8 * kk, bd + 2 * kk, idesc, 1u);
                            }
                        }
                        ptx::tc_commit(done);
                    }
                    __syncwarp();
                }
            }
            if (ptx::elect_one()) ptx::tc_commit(bar(FINAL));
            __syncwarp();
            ptx::mbar_wait(bar(FINAL), 0, abort_flag);          // nothing may still be executing when TMEM is freed
        }
    } else if (warp < WARP_DRAIN0) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
        // -------------------------------------------------------------------- unpack ----
        // One weight row (= one TMEM lane) per thread: 64 packed bytes -> 128 codes as bytes -> 32 TMEM columns, k
        // ascending, and the row's 32 bytes of the fifth slice.  Team t takes the steps st = t (mod TEAMS).
        const uint32_t team = (warp - WARP_UNPACK0) / TEAM_WARPS;
        const int u = ((warp - WARP_UNPACK0) % TEAM_WARPS) * 32 + lane;
        const uint32_t sw0 = blob_chunk_pos(u, 0) * 16;
        const uint32_t a_lane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + C::A_COL0;
        uint32_t st = 0;
        bool ok = true;
        for (int si = 0; ok; ++si) {
            int tile, gb, ge;
            if (!segment(si, tile, gb, ge)) break;
            for (int g = gb; g < ge; g += C::GPS, ++st) {
                if ((st & 1u) != team) continue;
                const uint32_t sr = st % C::SR, sa_ = st % C::SA;
                if (!(ok = ptx::mbar_wait(bar(RAW_FULL + sr), (st / C::SR) & 1, abort_flag))) break;
                const uint32_t raw = smem_base + C::RAW_OFF + sr * C::RAW_BYTES;
                uint4 w[C::GPS][4];
                uint32_t z[C::GPS], sc[C::GPS];
#pragma unroll
                for (int gg = 0; gg < C::GPS; ++gg) {        // a lone last group: the second half is stale bytes that no MMA uses
                    z[gg] = (ptx::lds_u8(raw + gg * BLOB_BYTES + BLOB_ZERO_OFF + (u >> 1)) >> ((u & 1) * 4)) & 0xFu;
                    sc[gg] = ptx::lds_u16(raw + gg * BLOB_BYTES + BLOB_SCALE_OFF + 2 * u);
                    // chunk p of row u sits at position p ^ ((u >> 1) & 3): eight consecutive rows hit eight bank groups
#pragma unroll
                    for (int p = 0; p < 4; ++p) w[gg][p] = ptx::lds128(raw + gg * BLOB_BYTES + u * 64 + (sw0 ^ (16 * p)));
                }
                // the MMAs that read this stage's previous contents have completed
                if (st >= (uint32_t)C::SA && !(ok = ptx::mbar_wait(step_bar(st - C::SA), ring_parity(st - C::SA), abort_flag))) break;
                ptx::tc_fence_after_sync();
                if (ge - g < C::GPS) z[C::GPS - 1] = sc[C::GPS - 1] = 0;     // a group that is not there: D = 0, scale 0
#pragma unroll
                for (int gg = 0; gg < C::GPS; ++gg) {
                    const uint32_t a_addr = a_lane + sa_ * C::A_COLS + gg * C::A_G;
                    ptx::sts_u16(smem_base + C::SCALE_OFF + ((st % SCALE_RING) * C::GPS + gg) * (TILE_N * 2) + 2 * u, sc[gg]);
                    // words 0..3 of a chunk hold the runs of four k (a0, a2), (a1, a3), (a4, a6), (a5, a7) in their
                    // (low, high) nibbles: columns in k order are lo(x), lo(y), hi(x), hi(y), lo(z), lo(w), hi(z), hi(w)
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        const uint4 v = w[gg][p];
                        constexpr uint32_t LO = 0x0F0F0F0Fu;
                        ptx::tmem_st_32x8(a_addr + 8 * p, v.x & LO, v.y & LO, (v.x >> 4) & LO, (v.y >> 4) & LO,
                                          v.z & LO, v.w & LO, (v.z >> 4) & LO, (v.w >> 4) & LO);
                    }
                    const uint32_t m8 = ((0u - 8u * z[gg]) & 0xFFu) * 0x01010101u, m1 = ((0u - z[gg]) & 0xFFu) | 0x80808000u;
                    ptx::tmem_st_32x8(a_addr + GROUP / 4, m8, m8, m8, m8, m1, 0x80808080u, 0x80808080u, 0x80808080u);
                }
                ptx::tmem_st_wait();
                ptx::tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) {
                    ptx::mbar_arrive(bar(A_FULL + sa_));
                    ptx::mbar_arrive(bar(RAW_EMPTY + sr));
                }
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 136;");
        // --------------------------------------------------------------------- drain ----
        // Warp (q, h): TMEM lanes 32q..32q+31 (output channels), accumulator columns h*W.. (tokens).
        ptx::pdl_wait();                                        // token scales, hand-over flags, residual and output
        const int q = warp & 3, h = (warp - WARP_DRAIN0) >> 2;
        const int n_local = q * 32 + lane;
        const uint32_t lane_taddr = tmem_base + ((uint32_t)(q * 32) << 16) + h * C::W;
        const uint32_t scale_src = smem_base + C::SCALE_OFF + n_local * 2;
        const uint64_t nb2 = ptx::pack2(0x80000000u | ACC_BIAS, 0x80000000u | ACC_BIAS);     // -bias * 2^-149
        if (lane == 0) {                                          // the accumulator buffers start out free
            for (int i = 0; i < C::NBU; ++i) ptx::mbar_arrive(bar(ACC_EMPTY + i));
        }
        uint32_t st = 0;
        bool ok = true;
        // token scales (raw fp16 bits) of the next segment, requested before the epilogue of the current one
        uint16_t next_sa_bits = 0;
        auto request = [&](int idx) {
            int t2, gb2, ge2, nt2, mt2;
            if (!segment(idx, t2, gb2, ge2)) return;
            tile_of(t2, nt2, mt2);
            const int m = mt2 * TILE_M + h * C::W + lane;
            next_sa_bits = lane < C::W && m < M ? __ldg(sa + m) : (uint16_t)0;
        };
        request(0);
        for (int si = 0; ok; ++si) {
            int tile, gb, ge, ntile, mtile;
            if (!segment(si, tile, gb, ge)) break;
            tile_of(tile, ntile, mtile);
            const int n = ntile * TILE_N + n_local;
            const int m_base = mtile * TILE_M + h * C::W;
            uint64_t facc[C::W / 2];                              // pairs of neighbouring tokens
#pragma unroll
            for (int i = 0; i < C::W / 2; ++i) facc[i] = 0ull;
            auto sum = [&](int i) { const float2 t = ptx::unpack2(facc[i / 2]); return i & 1 ? t.y : t.x; };
            if (RES) {
                // the residual of this warp's part of the tile (W tokens x 64 bytes) is asked into L2 now; the epilogue's
                // loads then find it there
                const int m = m_base + lane;
                if (lane < C::W && m < M)
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(residual + (size_t)m * N + (size_t)ntile * TILE_N + q * 32));
            }
            // this warp's token scales, widened once per tile (rows past M get 0 and are never stored)
            float* sa_w = reinterpret_cast<float*>(smem + C::SA_OFF) + (warp - WARP_DRAIN0) * C::W;
            __syncwarp();
            if (lane < C::W) sa_w[lane] = __half2float(__ushort_as_half(next_sa_bits)) * SCALE_OUT;
            __syncwarp();
            if (m_base >= M) {                                    // none of this warp's columns is a token
                for (int g = gb; g < ge; g += C::GPS, ++st) {
                    if (!(ok = ptx::mbar_wait(step_bar(st), ring_parity(st), abort_flag))) break;
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(bar(ACC_EMPTY + st % C::NBU));
                }
            } else {
                for (int g = gb; g < ge; g += C::GPS, ++st) {
                    const uint32_t ub = st % C::NBU;
                    if (!(ok = ptx::mbar_wait(step_bar(st), ring_parity(st), abort_flag))) break;
                    ptx::tc_fence_after_sync();
                    // All of this warp's columns go to registers with back-to-back loads, the buffer is handed back, then
                    // the arithmetic.  One straight line for every case (columns past the last token and a missing second
                    // group are summed like the rest): paths that join cost a register copy per running sum.
                    const uint32_t taddr = lane_taddr + ub * (C::GPS * TILE_M);
                    uint32_t v[C::GPS][C::W];
#pragma unroll
                    for (int c = 0; c < C::GPS; ++c) {
                        if constexpr (C::W == 32) ptx::tmem_ld_32x32(taddr + c * TILE_M, v[c]);
                        else ptx::tmem_ld_32x16(taddr + c * TILE_M, v[c]);
                    }
                    uint64_t s2[C::GPS];
#pragma unroll
                    for (int c = 0; c < C::GPS; ++c) {
                        const float f = __half2float(__ushort_as_half((unsigned short)ptx::lds_u16(
                                            scale_src + ((st % SCALE_RING) * C::GPS + c) * (TILE_N * 2)))) * SCALE_UP;
                        s2[c] = ptx::pack2(__float_as_uint(f), __float_as_uint(f));
                    }
                    ptx::tmem_ld_wait();
                    ptx::tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(bar(ACC_EMPTY + ub));
#pragma unroll
                    for (int c = 0; c < C::GPS; ++c) {
#pragma unroll
                        for (int i = 0; i < C::W; i += 2) {
                            ptx::add_fma2(facc[i / 2], v[c][i], v[c][i + 1], nb2, s2[c]);
                            if (DEBUG) {
                                if (g + c < ge && m_base + i < M)
                                    debug_partials[((size_t)(m_base + i) * GK + g_lo + g + c) * N + n] = (int32_t)v[c][i] - (int32_t)ACC_BIAS;
                                if (g + c < ge && m_base + i + 1 < M)
                                    debug_partials[((size_t)(m_base + i + 1) * GK + g_lo + g + c) * N + n] = (int32_t)v[c][i + 1] - (int32_t)ACC_BIAS;
                            }
                        }
                    }
                }
            }
            if (!ok) break;
            request(si + 1);
            if (BAL && gb > 0) {
                // Balanced walk: the tile's earlier groups belong to the CTA before this one, which reaches
                // them at the end of its range.  Hand this CTA's sums over: element (token t, channel n) at
                // t * 128 + n of this CTA's slot, then this warp's bit of the slot's flag word (release).  Warp by warp, because
                // a barrier of the drain warps has no limit: after a time-out elsewhere the warps that gave up never reach it.
                float* slot = handover + (size_t)blockIdx.x * (TILE_M * TILE_N);
#pragma unroll
                for (int i = 0; i < C::W; ++i) __stcg(slot + (size_t)(h * C::W + i) * TILE_N + n_local, sum(i));
                __syncwarp();
                if (lane == 0) ptx::red_or_release_gpu_u32(handover_flags + blockIdx.x, 1u << (warp - WARP_DRAIN0));
                continue;                       // the other CTA stores the tile
            }
            if (BAL && ge < G) {
                // ... and this CTA holds the earlier groups of a tile whose later groups the next CTA summed
                // long ago (they opened its range): wait for this warp's bit (bounded), add its sums, clear the bit
                ok = ptx::warp_wait_bit_acquire_gpu(handover_flags + blockIdx.x + 1, 1u << (warp - WARP_DRAIN0), abort_flag);
                if (!ok) break;
                const float* slot = handover + (size_t)(blockIdx.x + 1) * (TILE_M * TILE_N);
#pragma unroll
                for (int i = 0; i < C::W; i += 2) {
                    const float* p = slot + (size_t)(h * C::W + i) * TILE_N + n_local;
                    facc[i / 2] = ptx::add2(facc[i / 2], ptx::pack2(__float_as_uint(__ldcg(p)), __float_as_uint(__ldcg(p + TILE_N))));
                }
                __syncwarp();
                if (lane == 0) atomicAnd(handover_flags + blockIdx.x + 1, ~(1u << (warp - WARP_DRAIN0)));     // zero again for the next call
            }
            if (SPLIT) {
                // every CTA of the cluster is past its last MMA: the rings are free and become
                // the exchange buffers; push this thread's partials to the CTAs that own them
                ptx::cluster_sync();
                exchanged = true;
                // The tile's runs of four tokens are dealt out to the S CTAs; a thread pushes 16 bytes (its channel, four
                // tokens) at a time: slot [pusher][run of the owner][channel], even channels first, so that the lane that sums
                // channels 2 p and 2 p + 1 reads beside its neighbours.
                const int slot_n = (n_local & 1) * 64 + (n_local >> 1);
                const int lo1 = run_lo(1), lo2 = S > 2 ? run_lo(2) : RUNS, lo3 = S > 3 ? run_lo(3) : RUNS;
#pragma unroll
                for (int i = 0; i < C::W; i += 4) {
                    if (m_base + i < M) {
                        const int run = (h * C::W + i) / 4;
                        const int owner = (run >= lo1) + (run >= lo2) + (run >= lo3);
                        const int first = run >= lo3 ? lo3 : (run >= lo2 ? lo2 : (run >= lo1 ? lo1 : 0));
                        const uint32_t at = smem_base + (uint32_t)((slice * runs_max + run - first) * TILE_N + slot_n) * 16u;
                        const float2 p0 = ptx::unpack2(facc[i / 2]), p1 = ptx::unpack2(facc[i / 2 + 1]);
                        ptx::st_dsmem_f32x4(ptx::map_to_cta(at, (uint32_t)owner), make_float4(p0.x, p0.y, p1.x, p1.y));
                    }
                }
                // This CTA's share, by the drain warps: half a run at a time (four tokens x 64 channels, two to a lane, stores of
                // 128 bytes a row).  The residual is asked for before the second barrier: its round trip runs under the exchange.
                constexpr int ITEMS = (RUNS + NUM_DRAIN_WARPS - 1) / NUM_DRAIN_WARPS;          // S >= 2: at most RUNS / 2 runs
                const int w8 = warp - WARP_DRAIN0, lo = run_lo(slice), cnt = 2 * (run_lo(slice + 1) - lo);
                const int pair = (w8 & 1) * 32 + lane, m_first = mtile * TILE_M + 4 * (lo + (w8 >> 1));      // items are four runs apart
                const size_t at0 = (size_t)m_first * N + (size_t)ntile * TILE_N + 2 * pair;
                uint32_t rr[RES ? ITEMS : 1][4];
                if (RES) {
#pragma unroll
                    for (int j = 0; j < ITEMS; ++j)
#pragma unroll
                        for (int t = 0; t < 4; ++t)
                            rr[j][t] = w8 + 8 * j < cnt && m_first + 16 * j + t < M
                                           ? __ldcg(reinterpret_cast<const uint32_t*>(residual + at0 + (size_t)(16 * j + t) * N)) : 0u;
                }
                ptx::cluster_sync();                       // release after the pushes, acquire before the sums
                if (*abort_flag) break;
#pragma unroll
                for (int j = 0; j < ITEMS; ++j) {
                    if (w8 + 8 * j < cnt && m_first + 16 * j < M) {
                        float4 a0 = make_float4(0.0f, 0.0f, 0.0f, 0.0f), a1 = a0;
                        for (int s2 = 0; s2 < S; ++s2) {                                // rank order: deterministic
                            const uint32_t src = smem_base + (uint32_t)((s2 * runs_max + (w8 >> 1) + 4 * j) * TILE_N + pair) * 16u;
                            const float4 v0 = ptx::lds128f(src), v1 = ptx::lds128f(src + 1024);
                            a0.x += v0.x; a0.y += v0.y; a0.z += v0.z; a0.w += v0.w;
                            a1.x += v1.x; a1.y += v1.y; a1.z += v1.z; a1.w += v1.w;
                        }
                        const float f0[4] = {a0.x, a0.y, a0.z, a0.w}, f1[4] = {a1.x, a1.y, a1.z, a1.w};
#pragma unroll
                        for (int t = 0; t < 4; ++t) {
                            const int m = m_first + 16 * j + t;
                            if (m < M) {
                                const float ts = __half2float(__ushort_as_half(__ldg(sa + m))) * SCALE_OUT;
                                const uint32_t o = RES ? ptx::pack_bf16x2(fmaf(f0[t], ts, __uint_as_float(rr[j][t] << 16)),
                                                                          fmaf(f1[t], ts, __uint_as_float(rr[j][t] & 0xFFFF0000u)))
                                                       : ptx::pack_bf16x2(f0[t] * ts, f1[t] * ts);
                                *reinterpret_cast<uint32_t*>(y + at0 + (size_t)(16 * j + t) * N) = o;
                            }
                        }
                    }
                }
                break;                          // one tile per cluster
            }
            // Epilogue: token scale, bf16, and a transpose through shared memory so that global stores run along the
            // channel dimension (a thread owns a channel, the output is token-major): a block of W tokens x this warp's
            // 32 channels, one TMA tile store (32 tokens) or 16-byte stores per lane.
            if (m_base >= M) continue;
            uint8_t* ob = smem + C::OUT_OFF + (warp - WARP_DRAIN0) * 2048;
            const uint32_t ob_addr = smem_base + C::OUT_OFF + (warp - WARP_DRAIN0) * 2048;
            uint4 rv[C::W / 8];
            if (RES) {
                // The projection's output joins the residual stream, added in fp32 before the one rounding.  The residual is
                // fetched in the layout of the stores (16 bytes per lane, rows of 64 bytes) and written into the output block,
                // from which each lane reads its own channel's column back, adds, rounds and overwrites.  y may be the
                // residual buffer: this warp reads its block before it stores it.
#pragma unroll
                for (int k = 0; k < C::W / 8; ++k) {
                    const int m = m_base + 8 * k + (lane >> 2);
                    rv[k] = make_uint4(0u, 0u, 0u, 0u);
                    if (m < M)
                        rv[k] = __ldcg(reinterpret_cast<const uint4*>(residual + (size_t)m * N + (size_t)ntile * TILE_N + q * 32 + 8 * (lane & 3)));
                }
            }
            if (lane == 0) ptx::bulk_wait_group_read0();          // the previous tile's store has read `ob`
            __syncwarp();
            if (RES) {
#pragma unroll
                for (int k = 0; k < C::W / 8; ++k)
                    *reinterpret_cast<uint4*>(ob + (8 * k + (lane >> 2)) * 64 + 16 * (lane & 3)) = rv[k];
                __syncwarp();
            }
            constexpr int EB = RES ? 8 : 16;
#pragma unroll
            for (int part = 0; part < C::W / EB; ++part) {
                // EB token scales (and residuals) to registers ahead of the stores below: both are shared-memory
                // accesses that the compiler keeps in order
                float sc[EB], rs[EB];
#pragma unroll
                for (int k = 0; k < EB / 4; ++k) {
                    const float4 t = *reinterpret_cast<const float4*>(sa_w + EB * part + 4 * k);
                    sc[4 * k] = t.x; sc[4 * k + 1] = t.y; sc[4 * k + 2] = t.z; sc[4 * k + 3] = t.w;
                }
                if (RES) {
#pragma unroll
                    for (int i = 0; i < EB; ++i)
                        rs[i] = __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(ob + (EB * part + i) * 64)[lane]);
                }
#pragma unroll
                for (int i = 0; i < EB; ++i) {
                    const int e = EB * part + i;
                    const float o = RES ? fmaf(sum(e), sc[i], rs[i]) : sum(e) * sc[i];
                    reinterpret_cast<__nv_bfloat16*>(ob + e * 64)[lane] = __float2bfloat16_rn(o);
                }
            }
            if (C::W == 32) {
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {                                  // rows past M are clipped by the map
                    ptx::tma_store_2d(&tmap_y, ntile * TILE_N + q * 32, m_base, ob_addr);
                    ptx::bulk_commit_group();
                }
            } else {
                __syncwarp();
#pragma unroll
                for (int k = 0; k < C::W / 8; ++k) {
                    const int row = 8 * k + (lane >> 2), m = m_base + row;
                    if (m < M)
                        *reinterpret_cast<uint4*>(y + (size_t)m * N + (size_t)ntile * TILE_N + q * 32 + 8 * (lane & 3)) =
                            *reinterpret_cast<const uint4*>(ob + row * 64 + 16 * (lane & 3));
                }
                __syncwarp();
            }
        }
        if (lane == 0) ptx::bulk_wait_group_read0();              // every tile store of this warp has read its block
        __syncwarp();
    }

    ptx::pdl_wait();                            // every thread, before the split-K tail's stores and the status word
    if (SPLIT && !exchanged) {                  // both barriers for every thread that has not passed them in the drain role
        ptx::cluster_sync();
        ptx::cluster_sync();
    }
    if (*abort_flag && lane == 0) atomicExch(status, (uint32_t)W4A8_ERR_TIMEOUT);
    ptx::tc_fence_before_sync();
    __syncthreads();
    if (warp == WARP_MMA) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc(tmem_base, TMEM_COLS);
    }
}

template <int TILE_M, bool DEBUG, bool SPLIT, bool BAL, bool RES>
cudaError_t launch_short(const int8_t* qa, const uint16_t* sa, const int32_t* asum, const void* packed, void* y, const void* residual,
                        int M, int N, int K, int S, void* workspace, int32_t* debug_partials, cudaStream_t stream) {
    using C = Cfg<TILE_M>;
    CUtensorMap tmap, tmap_y;
    cudaError_t e = make_qa_group_map(&tmap, qa, M, K, TILE_M, C::GPS);
    if (e != cudaSuccess) return e;
    e = make_y_tensor_map(&tmap_y, y, M, N);
    if (e != cudaSuccess) return e;
    int dev = 0;
    e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    static bool attr_done[64] = {false};
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!attr_done[dev]) {
        e = cudaFuncSetAttribute(gemm_tcshort_kernel<TILE_M, DEBUG, SPLIT, BAL, RES>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 C::SMEM_ALLOC);
        if (e != cudaSuccess) return e;
        attr_done[dev] = true;
    }
    const int sms = device_sm_count();
    const int m_tiles = (M + TILE_M - 1) / TILE_M;
    const int total = m_tiles * (N / TILE_N);
    // persistent: at most one CTA per SM; split-K: one cluster of S CTAs per tile
    const int grid = SPLIT ? total * S : (total < sms ? total : sms);
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    // BAL: the tiles x groups units are dealt out evenly (a tile may then be shared by two neighbouring
    // CTAs, which meet through the hand-over area of the workspace); the caller has checked that it applies
    if (BAL && !(total > grid && grid <= HANDOVER_SLOTS && handover_bytes(M, N, K) > 0)) return cudaErrorInvalidConfiguration;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid, 1, 1);
    cfg.blockDim = dim3(TS_THREADS, 1, 1);
    cfg.dynamicSmemBytes = C::SMEM_ALLOC;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = SPLIT ? (unsigned)S : 1u;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, gemm_tcshort_kernel<TILE_M, DEBUG, SPLIT, BAL, RES>, tmap, tmap_y, static_cast<const uint8_t*>(packed), sa,
                              asum, static_cast<__nv_bfloat16*>(y), static_cast<const __nv_bfloat16*>(residual), debug_partials,
                              reinterpret_cast<uint32_t*>(ws + WS_STATUS_OFF),
                              M, N, K, m_tiles, total, S, reinterpret_cast<float*>(ws + WS_SHARED_OFF),
                              reinterpret_cast<uint32_t*>(ws + WS_COUNTER_OFF));
}

template <int TILE_M>
int query_clusters(int S) {
    using C = Cfg<TILE_M>;
    int n = 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(S * 64), 1, 1);
    cfg.blockDim = dim3(TS_THREADS, 1, 1);
    cfg.dynamicSmemBytes = C::SMEM_ALLOC;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)S;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    if (cudaFuncSetAttribute(gemm_tcshort_kernel<TILE_M, false, true, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             C::SMEM_ALLOC) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, gemm_tcshort_kernel<TILE_M, false, true, false, false>, &cfg) != cudaSuccess)
        return 0;
    return n;
}

template <int TILE_M, bool DEBUG, bool RES>
cudaError_t launch_walk(int S, bool balanced, const int8_t* qa, const uint16_t* sa, const int32_t* asum, const void* packed, void* y,
                        const void* residual, int M, int N, int K, void* workspace, int32_t* dp, cudaStream_t st) {
    if (S > 1) return launch_short<TILE_M, DEBUG, true, false, RES>(qa, sa, asum, packed, y, residual, M, N, K, S, workspace, dp, st);
    if (balanced) return launch_short<TILE_M, DEBUG, false, true, RES>(qa, sa, asum, packed, y, residual, M, N, K, 1, workspace, dp, st);
    return launch_short<TILE_M, DEBUG, false, false, RES>(qa, sa, asum, packed, y, residual, M, N, K, 1, workspace, dp, st);
}

template <bool DEBUG, bool RES>
cudaError_t launch_height(int S, bool balanced, const int8_t* qa, const uint16_t* sa, const int32_t* asum, const void* packed,
                          void* y, const void* residual, int M, int N, int K, void* workspace, int32_t* dp, cudaStream_t st) {
    // up to 32 tokens the tile is cut to 32 columns: half the drain's loads and arithmetic
    if (M <= 32) return launch_walk<32, DEBUG, RES>(S, balanced, qa, sa, asum, packed, y, residual, M, N, K, workspace, dp, st);
    return launch_walk<64, DEBUG, RES>(S, balanced, qa, sa, asum, packed, y, residual, M, N, K, workspace, dp, st);
}

}  // namespace

int tcshort_max_clusters(int S) {
    const int a = query_clusters<64>(S), b = query_clusters<32>(S);
    return a < b ? a : b;
}

cudaError_t launch_gemm_tcshort(int S, bool balanced, const int8_t* qa, const uint16_t* sa, const int32_t* asum,
                                const void* packed, void* y, const void* residual, int M, int N, int K, void* workspace,
                                int32_t* debug_partials, cudaStream_t stream) {
    if (residual)                                   // (no partials dump in this form)
        return launch_height<false, true>(S, balanced, qa, sa, asum, packed, y, residual, M, N, K, workspace, nullptr, stream);
    if (debug_partials)
        return launch_height<true, false>(S, balanced, qa, sa, asum, packed, y, nullptr, M, N, K, workspace, debug_partials, stream);
    return launch_height<false, false>(S, balanced, qa, sa, asum, packed, y, nullptr, M, N, K, workspace, nullptr, stream);
}

}  // namespace w4a8
