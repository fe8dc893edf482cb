// Large-M W4A8 GEMM for sm_100a (token tiles of 208 and 128 rows; 64-row tiles, for fewer tokens, run in
// gemm_tcshort.cu - the per-channel form below has them here, and layers of up to four groups at more than 32 tokens): bulk copies -> shared memory -> int4->int8 unpack into TENSOR
// MEMORY -> tcgen05.mma kind::i8 (weights from TMEM, activations from shared memory) with int32
// accumulators in TMEM -> per-group fp32 scaling -> bf16.
// (Sec. 3.4: quantising the activations to 8 bits is what lets the compute-bound prefill run on
// INT8 tensor cores; Sec. 4: prefill is one long matrix multiplication.)
//
// Orientation ("swap-AB"): the 128 output channels of a tile are the MMA's M side (TMEM lanes),
// the tokens are its N side (TMEM columns).  A drain thread therefore owns ONE output channel:
// its group scale is a per-thread scalar and the per-group work on the CUDA cores is one
// int->float convert and half a packed FMA per accumulator element.
//
// One pipeline step = one quantisation group = 128 k = four K=32 MMAs; the accumulator must be
// drained after every group because the scale changes, so TMEM holds two accumulator buffers:
// the tensor core fills one while the drain warps empty the other.  The first MMA of a group
// overwrites its buffer, so a buffer needs no preparation: the drain hands it back as soon as
// its columns are in registers.
//
// The tensor pipe is not what bounds this kernel (it is busy under a third of the time): the CUDA
// cores must take every accumulator element out of TMEM after every group and spend one and
// a half instructions on it, the unpack shares the integer pipe with that conversion, and shared memory
// (about 128 B/clk per SM) is shared by the tensor core's operand reads, the bulk-copy fills and
// ordinary loads.  Design choices made on measurements:
//  * the unpacked weights never touch shared memory: an unpack thread owns one weight row
//    (= one TMEM lane), converts its 64 packed bytes in registers and writes the 128 signed
//    bytes to 32 TMEM columns with tcgen05.st; the MMA takes its A operand from TMEM.  That
//    removes a 16 KB store and a 16 KB operand read per group from shared memory;
//  * the token tile is 208 rows, not 256: two accumulator buffers of 208 columns plus three
//    32-column weight stages fill the 512 TMEM columns exactly, and M = 1024 or 4096 splits
//    into 208-row tiles with 1.5 % padding;
//  * there is no accumulator bias / re-arm (which would turn the int->float conversion into an
//    FMA-pipe add): tcgen05.st traffic to TMEM costs as much port time as tcgen05.ld traffic, more
//    than the conversion;
//  * two warps issue the MMAs, one for the even and one for the odd steps (a step costs its issuer
//    three barrier waits, four MMAs and a commit); the whole warp walks the loop and an elected lane
//    issues, which keeps the MMA operands in uniform registers (from inside a one-lane branch every
//    MMA cost its thread about a hundred cycles of register-to-uniform moves);
//  * what paces a step of a 208-row tile is the chain of a drain warp - the look at its barrier, the loads, the hand-back and the
//    sums, 100 to 200 cycles for each of the first three however long ago the MMAs finished (measured with stamps; the
//    barrier has completed at the first look five times out of six).  So the warp index is made warp-uniform (ring indices,
//    barrier and tensor-memory addresses on the uniform datapath) and two sums take one packed FMA; in 208-row tiles without a
//    residual arrivals are predicated instructions instead of one-lane branches, and without a residual, at every height, the
//    next step's barrier is looked at under the loads (where these two cost instead, they are not taken: see BRANCH below).
//    Together, 4096 -> 24576 at 1024 and 4096 tokens 132.2 and 521 us before, 127.2 and 471 after, 4096 -> 6144 43.8 and 138.3, 41.7
//    and 131.9, 5120 -> 27648 at 1391 241.5 and 237.0; with a residual 12288 -> 4096 at 1024 and 4096 70.5 and 273.9, 69.6 and 269.9,
//    4096 -> 4096 equal (B200, weights cold, both builds in turn).  Tried on top, none quicker: the conversion moved to the FMA pipe by a constant bias in the
//    accumulators (131), for half of the columns (134), the two halves of the columns filled and handed back on their own (144),
//    columns loaded in pieces ahead of the sums (129.6), a tile's outputs staged whole (127.4 before the look ahead, equal);
//  * one tcgen05.commit per step, on a ring of "step done" barriers, frees the step's weight and
//    activation stages and publishes its accumulator.
//
// Zero points are subtracted while unpacking (weights become signed, -15..15), so the int32
// accumulator is directly D = sum (q_w - z) q_a; identical to P - z*sum(q_a), and it moves the
// correction from the per-(token, channel, group) drain to the per-weight unpack.
//
// Warp roles (512 threads, four warpgroups so that setmaxnreg can move registers to the drain:
// 40 / 40 / 216 / 216 per thread for 208-row tiles, 48 / 96 / 160 / 160 for shorter ones):
//   warp 0       producer of the activation tiles (2-D TMA loads)
//   warps 1, 3   MMA issuers (even and odd pipeline steps; an elected lane issues); warp 1 owns TMEM allocation
//   warp 2       producer of the packed blobs (1-D bulk copies)
//   warps 4-7    unpack: raw blob -> signed int8 weight rows in TMEM
//   warps 8-15   drain: tcgen05.ld -> convert -> FMA with the group scale; final bf16 store
//
// Split-K variant (SPLIT): when an [M, N] problem has fewer tiles than half the SMs, a tile is given
// to a thread-block cluster of S CTAs, each walking G / S of the K groups (a CTA's time is close to
// proportional to its number of groups, whatever the tile height).  The fp32 partials are reduced
// like the small-M kernel's: after a cluster barrier (every CTA has finished its MMAs, so the
// activation ring is free) each drain thread pushes its partials with st.shared::cluster into the
// ring area of the CTA that owns that share of the tile (slot = pusher's rank), a second cluster
// barrier, and the owner sums its S slots in rank order, applies the token scale and stores bf16.
// The shares are runs of four tokens, so that a push is 16 bytes and needs no division: word by word, each with
// its owner found by two divisions at run time, and the sums stored 2 bytes a lane, the exchange took 10 us of a 208-row
// tile (4096 x 4096 at 200 tokens in three slices 20.2 us, now 13.3; 12288 x 4096 in four with residual 28.3, now 22.2).
// Every wait is bounded; on expiry the CTA records W4A8_ERR_TIMEOUT, frees TMEM and exits.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include "dispatch_rules.h"
#include "ptx_sm100.cuh"
#include "w4a8_internal.cuh"

namespace w4a8 {
namespace {

constexpr int TC_THREADS = 512;
constexpr int WARP_PRODUCER = 0, WARP_MMA = 1, WARP_RAW_PRODUCER = 2, WARP_MMA_ODD = 3, WARP_UNPACK0 = 4, WARP_DRAIN0 = 8;
constexpr int DONE_RING = 8;                     // "group finished" barriers; every role stays within 8 groups of the others
constexpr int NUM_UNPACK_WARPS = 4, NUM_DRAIN_WARPS = 8;
constexpr int RAW_STRIDE = 8576;                 // BLOB_BYTES rounded up to a multiple of 128
constexpr int A_COLS = GROUP / 4;                // 32 TMEM columns hold one group of a weight row (4 bytes per column)
constexpr int TMEM_COLS = 512;
// Cost model of tcgen05_plan (nanoseconds, measured on B200 behind the quantiser, weights cold; 208-, 128-, 64-row
// tiles): per launch; per group a CTA walks; per tile after a CTA's first (its epilogue); for splitting K over a cluster of S
// CTAs (two cluster barriers, exchange and reduction); for the balanced walk (hand-over of two partial tiles, and CTAs out of
// step: its groups in per cent of the plain walk's).  64-row tiles run in the kernel of gemm_tcshort.cu, whose tile is cut to
// 32 columns for up to 32 tokens.
// A tile of few groups is mostly epilogue, so layers of up to 15 groups have constants of their own: fitted to every height
// at 14 token counts from 65 on and six widths, the choice is within 3 % of the best height (with the constants for long K up to
// 16 %: 768 -> 24576 at 96 tokens 11.9 us with 64 rows and 10.8 with 128), up to four groups within 11 %.  From 16 groups on the epilogue is in the fit of the others.
constexpr int TC_MAX_SPLIT = 4;
struct TcCost { long fixed[3], group[3], tile[3]; };
constexpr TcCost TC_COST = {{3500, 3200, 2500}, {525, 440, 255}, {0, 0, 0}}, TC_COST_MEDIUM = {{4000, 2550, 2500}, {525, 440, 255}, {2350, 1450, 1250}},
                 TC_COST_FEW = {{4550, 3750, 2950}, {800, 605, 405}, {2400, 1500, 1250}};
// Layers of up to four groups at more than 32 tokens run their 64-row tiles here: the kernel of gemm_tcshort.cu gains 0.15 us a
// group and loses 0.4 to 0.5 before its first and after its last (measured on B200 behind the quantiser, here against there: 128
// -> 8192 at 64 tokens 4.5 and 5.0 us, 384 -> 24576 at 64 6.5 and 7.3, 512 -> 1024 at 128 5.1 and 5.5; 768 -> 1024 equal, 1024 -> 24576
// at 64 10.1 and 9.7; up to 32 tokens, where its tile has 32 columns, 256 -> 24576 5.9 and 5.7).
constexpr int TC_FEW_GROUPS = 4;
bool few_groups(int M, int G) { return M > 32 && G <= TC_FEW_GROUPS; }
constexpr long TC_GROUP_32_NS = 230;
constexpr long TC_SPLIT_NS[3][TC_MAX_SPLIT + 1] = {{0, 0, 4000, 4500, 5600}, {0, 0, 2800, 2800, 3400}, {0, 0, 1800, 2700, 3500}};
constexpr long TC_BALANCE_NS[3] = {6000, 4000, 4500}, TC_BALANCE_PERCENT[3] = {104, 104, 100};

// Shared-memory rings.  The activation tile comes from L2 through TMA with a latency of roughly
// 2000 cycles, the packed blob from HBM likewise: both rings are deep enough to cover it.
template <int TILE_M>
struct Cfg {
    static constexpr int B_BYTES = TILE_M * GROUP;                            // one activation stage
    static constexpr int SB = TILE_M > 128 ? 5 : (TILE_M == 128 ? 6 : 8);     // activation stages
    static constexpr int SR = TILE_M > 128 ? 8 : (TILE_M == 128 ? 12 : 16);   // packed-blob stages: a short tile finishes a group
                                                                              // quickly, so more blobs must be in flight to cover HBM latency
    static constexpr int NB = 2;                                               // accumulator buffers in flight
    static constexpr int SA_MAX = (TMEM_COLS - NB * TILE_M) / A_COLS;
    static constexpr int SA = SA_MAX > 4 ? 4 : SA_MAX;                        // weight stages in TMEM
    static constexpr int A_COL0 = NB * TILE_M;                                // first weight column (after the accumulators)
    static constexpr int B_OFF = 0;
    static constexpr int RAW_OFF = B_OFF + SB * B_BYTES;
    static constexpr int BAR_OFF = RAW_OFF + SR * RAW_STRIDE;
    static constexpr int NUM_BARS = 2 * SR + SB + SA + NB + DONE_RING + 2 + 2;
    static constexpr int MISC_OFF = (BAR_OFF + NUM_BARS * 8 + 15) & ~15;      // 16-byte aligned: staging is read with 16-byte loads
    static constexpr int W = TILE_M / 2;                                      // accumulator columns (tokens) per drain warp
    static constexpr int NCH = (W + 31) / 32;                                 // 32-column chunks per drain warp (the last may be 8 wide)
    static constexpr int LAST = W - 32 * (NCH - 1);                           // width of the last chunk
    static constexpr int SA_OFF = MISC_OFF + 16;   // per drain warp: token scales as fp32
    static constexpr int OUT_OFF = (SA_OFF + NUM_DRAIN_WARPS * NCH * 32 * 4 + 127) & ~127;   // per drain warp: 32 tokens x 32 channels bf16 (TMA source: 128-byte aligned)
    static constexpr int SMEM_BYTES = OUT_OFF + NUM_DRAIN_WARPS * 2048;
    static constexpr int SMEM_ALLOC = SMEM_BYTES + 1024;       // slack to align the base to 1024 B
    static_assert(TILE_M == 64 || TILE_M == 128 || TILE_M == 208, "token tile");
    static_assert(TILE_M % 16 == 0, "MMA N granularity; 8-row swizzle atoms");
    static_assert(LAST == 32 || LAST == 8, "chunk widths the drain knows how to load");
    static_assert(SA >= 2 && A_COL0 + SA * A_COLS <= TMEM_COLS, "tensor memory");
    static_assert(SB <= DONE_RING && SA <= DONE_RING, "a stage is freed by the group that used it, at most DONE_RING groups ago");
    static_assert(SMEM_ALLOC <= 227 * 1024, "shared memory");
    static_assert(OUT_OFF % 128 == 0 && SA_OFF % 16 == 0 && B_BYTES % 1024 == 0, "alignment");
};

__device__ __forceinline__ uint32_t sub_zero4(uint32_t q, uint32_t kz) {
    // bytes of q in 0..15, bytes of kz = 0x80 - z with z in 0..15: per byte (q + 0x80 - z) ^ 0x80
    // is q - z as a signed int8; no carry crosses a byte (0x71 <= q + 0x80 - z <= 0x8F).  (The per-byte subtract
    // intrinsic __vsub4 in its place was measured 7-10 % slower on the whole kernel: it is not one instruction here.)
    return (q + kz) ^ 0x80808080u;
}

// PC ("per channel"): the scales of a channel are the same in every group, so the integer sums of all
// groups of a tile add up in one accumulator and the tile is drained once (see w4a8_gemm_per_channel).
// BAL: balanced walk (see `segment` below).
// RES: the epilogue adds a residual (its own instantiations: the extra registers of the residual block would
// otherwise spill in the plain kernels).
template <int TILE_M, bool DEBUG, bool SPLIT, bool PC = false, bool BAL = false, bool RES = false>
__global__ void __launch_bounds__(TC_THREADS, 1)
gemm_tcgen05_kernel(const __grid_constant__ CUtensorMap tmap_qa, const __grid_constant__ CUtensorMap tmap_y,
                    const uint8_t* __restrict__ packed,
                    const uint16_t* __restrict__ sa, __nv_bfloat16* y, const __nv_bfloat16* residual,
                    int32_t* __restrict__ debug_partials, uint32_t* __restrict__ status,
                    int M, int N, int K, int m_tiles, int total_tiles, int S,
                    float* __restrict__ handover, uint32_t* __restrict__ handover_flags) {
    // Programmatic dependent launch: the kernel after this one may start its prologue now; this one sets up tensor
    // memory, barriers and its weight stream (weights never depend on the previous kernel) while its predecessor may
    // still run, and the roles that touch activations, token scales, the workspace or the output wait below.
    ptx::pdl_launch_dependents();
    using C = Cfg<TILE_M>;
    static_assert(!SPLIT || C::SB * C::B_BYTES >= (TILE_M / 4 + TC_MAX_SPLIT - 1) * TILE_N * 16, "the split-K exchange buffer lives in the activation ring");
    static_assert(!(SPLIT && PC), "the per-channel form is not split along K");
    static_assert(!BAL || (!SPLIT && !PC), "the balanced walk is for the plain persistent form");
    // Arrivals of one lane, of unpack and drain warps: a branch, or predicated instructions.  Each is the quicker one on its side (B200:
    // 128 rows, per channel 4096 -> 4096 at 1024 tokens 21.1 us with branches, 22.5 predicated, grouped 4096 -> 24576 at 256
    // 43.2 and 45.2; 208 rows at 1024 129.2 and 126.3, per channel 4096 -> 6144 22.3 and 21.8).  With a residual the branch, and no
    // look ahead at the next step's barrier: both cost there, in the balanced walk above all (12288 -> 4096 at 1024 and 4096 tokens
    // 71.1 and 296.9 us with both, 69.5 and 289.5 without; 13824 -> 5120 at 1391 126.2 and 123.6).
    constexpr bool BRANCH = TILE_M <= 128 || RES, LOOK_AHEAD = !RES;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem = smem_raw + (smem_base - ptx::smem_u32(smem_raw));
    const int GK = K / GROUP;                                   // groups of the whole K range (blob and output indexing)
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);     // known to be warp-uniform this way: see the header
    // SPLIT: a cluster of S CTAs per tile (one tile per cluster, no persistence); this CTA walks groups [g_lo, g_lo + G)
    const int slice = SPLIT ? (int)ptx::cluster_ctarank() : 0;
    const int unit = SPLIT ? (int)blockIdx.x / S : (int)blockIdx.x;
    const int num_units = SPLIT ? (int)gridDim.x / S : (int)gridDim.x;
    const int g_lo = SPLIT ? (int)(((long long)slice * GK) / S) : 0;
    const int G = SPLIT ? (int)(((long long)(slice + 1) * GK) / S) - g_lo : GK;

    auto bar = [&](int i) { return smem_base + C::BAR_OFF + 8 * i; };
    // DONE[j % DONE_RING] completes its phase j / DONE_RING when the MMAs of pipeline step j have finished: that
    // one event frees the step's weight stage (unpack warps wait for step it - SA), its activation
    // stage (producer waits for step it - SB) and publishes its accumulator (drain warps wait for it).
    const int RAW_FULL = 0, RAW_EMPTY = C::SR, B_FULL = 2 * C::SR, A_FULL = B_FULL + C::SB, ACC_EMPTY = A_FULL + C::SA,
              DONE = ACC_EMPTY + C::NB, FINAL = DONE + DONE_RING, TILE_DONE = FINAL + 2;
    auto done_bar = [&](uint32_t step) { return bar(DONE + (int)(step % DONE_RING)); };
    auto done_parity = [](uint32_t step) { return (step / DONE_RING) & 1u; };
    volatile uint32_t* tmem_holder = reinterpret_cast<volatile uint32_t*>(smem + C::MISC_OFF);
    volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem + C::MISC_OFF + 4);

    if (warp == WARP_MMA) {
        if (lane == 0) {
            *abort_flag = 0;
            for (int i = 0; i < C::SR; ++i) {
                ptx::mbar_init(bar(RAW_FULL + i), 1);
                ptx::mbar_init(bar(RAW_EMPTY + i), NUM_UNPACK_WARPS);
            }
            for (int i = 0; i < C::SB; ++i) ptx::mbar_init(bar(B_FULL + i), 1);
            for (int i = 0; i < C::SA; ++i) ptx::mbar_init(bar(A_FULL + i), NUM_UNPACK_WARPS);
            for (int i = 0; i < C::NB; ++i) ptx::mbar_init(bar(ACC_EMPTY + i), NUM_DRAIN_WARPS);
            for (int i = 0; i < DONE_RING; ++i) ptx::mbar_init(bar(DONE + i), 1);
            for (int i = 0; i < 2; ++i) ptx::mbar_init(bar(FINAL + i), 1);
            for (int i = 0; i < 2; ++i) ptx::mbar_init(bar(TILE_DONE + i), 2);      // both MMA issuers
            ptx::fence_mbar_init();
        }
        __syncwarp();
        ptx::tmem_alloc(smem_base + C::MISC_OFF, TMEM_COLS);
        ptx::tmem_relinquish();
    }
    if (warp == WARP_PRODUCER && lane == 0) ptx::prefetch_tmap(&tmap_qa);
    if (warp == WARP_DRAIN0 && lane == 0) ptx::prefetch_tmap(&tmap_y);
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_holder;
    // tile of iteration t of this CTA: channel tile and token tile
    auto tile_of = [&](int t, int& ntile, int& mtile) {
        ntile = t / m_tiles;
        mtile = t % m_tiles;
    };

    // The work of a CTA as a list of segments (tile, groups [gb, ge) of it).  Plain persistent walk: whole
    // tiles unit, unit + num_units, ...  Balanced walk (more tiles than CTAs): the tiles x groups units are
    // dealt out in equal contiguous ranges, so a CTA's first and last segment may be part of a tile; the CTA
    // that holds the later groups of such a tile reaches them first (they open its range) and hands its
    // fp32 sums over through global memory to the CTA that holds the earlier groups (they close its range).
    // (warp-uniform on purpose, and said so to the compiler by the shuffles: with the range in ordinary registers the
    // loop counters, ring indices and MMA operands of every role left the uniform datapath: +53 ALU instructions per group
    // and scheduler, 8 to 12 % of the walk: 4096 -> 37888 at 200 tokens, whole tiles only, 43.3 us, now 40.8; plain walk 39.6)
    int bal_tile = 0, bal_gb = 0, bal_left = 0;
    if (BAL) {
        const long lo = ((long)blockIdx.x * total_tiles * G) / gridDim.x, hi = ((long)(blockIdx.x + 1) * total_tiles * G) / gridDim.x;
        bal_tile = __shfl_sync(0xFFFFFFFFu, (int)(lo / G), 0);
        bal_gb = __shfl_sync(0xFFFFFFFFu, (int)(lo % G), 0);
        bal_left = __shfl_sync(0xFFFFFFFFu, (int)(hi - lo), 0) + bal_gb;      // groups to the end of the range, from the first tile's start
    }
    auto segment = [&](int idx, int& tile, int& gb, int& ge) -> bool {
        if (BAL) {
            tile = bal_tile + idx;
            gb = idx == 0 ? bal_gb : 0;
            const int left = bal_left - idx * G;
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
    auto run_lo = [&](int o) { return RUNS * o / S; };
    if (warp < 4) {
        if (TILE_M > 128) asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
        else asm volatile("setmaxnreg.dec.sync.aligned.u32 48;");          // (with 40 the split and the per-channel form spill)
        if (warp == WARP_PRODUCER && lane == 0) {
            // ------------------------------------------------ producer: activation tiles ----
            ptx::pdl_wait();                                    // the activations are the previous kernel's output
            uint32_t it = 0;
            bool ok = true;
            for (int si = 0; ok; ++si) {
                int tile, gb, ge, ntile, mtile;
                if (!segment(si, tile, gb, ge)) break;
                tile_of(tile, ntile, mtile);
                for (int g = gb; g < ge; ++g, ++it) {
                    const uint32_t sb = it % C::SB;
                    if (it >= (uint32_t)C::SB && !(ok = ptx::mbar_wait(done_bar(it - C::SB), done_parity(it - C::SB), abort_flag))) break;
                    ptx::mbar_arrive_expect_tx(bar(B_FULL + sb), C::B_BYTES);
                    ptx::tma_load_2d(smem_base + C::B_OFF + sb * C::B_BYTES, &tmap_qa, (g_lo + g) * GROUP, mtile * TILE_M,
                                     bar(B_FULL + sb));
                }
            }
            if (!ok) {   // let copies already in flight land before shared memory is released
                const uint64_t t0 = ptx::globaltimer_ns();
                while (ptx::globaltimer_ns() - t0 < 200000ull) {}
            }
        } else if (warp == WARP_RAW_PRODUCER && lane == 0) {
            // --------------------------------------------------- producer: packed blobs ----
            uint32_t it = 0;
            bool ok = true;
            for (int si = 0; ok; ++si) {
                int tile, gb, ge, ntile, mtile;
                if (!segment(si, tile, gb, ge)) break;
                tile_of(tile, ntile, mtile);
                const uint8_t* src = packed + ((size_t)ntile * GK + g_lo) * BLOB_BYTES;
                for (int g = gb; g < ge; ++g, ++it) {
                    const uint32_t sr = it % C::SR, pr = (it / C::SR) & 1;
                    if (!(ok = ptx::mbar_wait(bar(RAW_EMPTY + sr), pr ^ 1, abort_flag))) break;
                    ptx::mbar_arrive_expect_tx(bar(RAW_FULL + sr), BLOB_BYTES);
                    ptx::bulk_g2s(smem_base + C::RAW_OFF + sr * RAW_STRIDE, src + (size_t)g * BLOB_BYTES, BLOB_BYTES,
                                  bar(RAW_FULL + sr));
                }
            }
            if (!ok) {
                const uint64_t t0 = ptx::globaltimer_ns();
                while (ptx::globaltimer_ns() - t0 < 200000ull) {}
            }
        } else if (warp == WARP_MMA || warp == WARP_MMA_ODD) {
            // ---------------------------------------------------------------- MMA issuers ----
            // Two warps, one for the even pipeline steps (accumulator buffer 0) and one for the odd
            // ones (buffer 1).  A step costs its issuer several dependent shared-memory and
            // tensor-pipe round trips (three barrier probes, four MMAs, a commit); with two issuers the
            // round trips of one step overlap the MMAs of the other.
            // The whole warp walks the loop and one elected lane issues: with warp-uniform control flow the
            // MMA operands (addresses, descriptors) are computed once per warp in uniform registers, which
            // is where the tensor instructions take them from; issued from inside a one-lane branch, every
            // operand of every MMA went through a register-to-uniform move first.
            const uint32_t par = __shfl_sync(0xFFFFFFFFu, (warp == WARP_MMA) ? 0u : 1u, 0);
            const uint32_t tmem_u = __shfl_sync(0xFFFFFFFFu, tmem_base, 0);
            constexpr uint32_t idesc = ptx::idesc_i8(TILE_N, TILE_M, true, true);
            // descriptor of activation stage 0; a stage and a K slice of 32 bytes are plain
            // additions to its (address >> 4) field
            const uint64_t b_desc0 = ptx::smem_desc_k_sw128(smem_base + C::B_OFF);
            uint32_t it = 0, tcount = 0;
            bool ok = true;
            for (int si = 0; ok; ++si, ++tcount) {
                int tile, gb, ge;
                if (!segment(si, tile, gb, ge)) break;
                // PC: both threads add into the buffer of the tile, which the drain warps left zeroed
                // (integer sums commute, so the order of the two threads' MMAs does not matter)
                const uint32_t buf = PC ? (tcount & 1u) : par;
                const uint32_t d_tmem = tmem_u + buf * TILE_M;
                bool mine = false;
                for (int g = gb; g < ge; ++g, ++it) {
                    if ((it & 1u) != par) continue;
                    const uint32_t sb = it % C::SB, pb = (it / C::SB) & 1;
                    const uint32_t sa_ = it % C::SA, pas = (it / C::SA) & 1;
                    // accumulator drained; activations landed; weights unpacked
                    // Parking waits, one after the other: polling the three barriers in a loop gained nothing at tall
                    // tiles (the accumulator hand-back this warp waits for there is 1 000 cycles away) and cost 3-4 %
                    // at short ones, where the probes queue up in front of the unpack warp's shared-memory accesses
                    // on the same scheduler.  At short tiles the unpacked weights arrive last by far.
                    // (Order as measured: weights first at short tiles; activations first at tall ones, 1.5 % there.)
                    if (TILE_M <= 128) {
                        if (!(ok = ptx::mbar_wait(bar(A_FULL + sa_), pas, abort_flag))) break;
                        if (!(ok = ptx::mbar_wait(bar(B_FULL + sb), pb, abort_flag))) break;
                    } else {
                        if (!(ok = ptx::mbar_wait(bar(B_FULL + sb), pb, abort_flag))) break;
                        if (!(ok = ptx::mbar_wait(bar(A_FULL + sa_), pas, abort_flag))) break;
                    }
                    if (!(ok = ptx::mbar_wait(bar(ACC_EMPTY + buf), (PC ? (tcount >> 1) : (it / C::NB)) & 1, abort_flag))) break;
                    ptx::tc_fence_after_sync();
                    const uint64_t bd = b_desc0 + (uint64_t)(sb * (C::B_BYTES / 16));
                    const uint32_t a_tmem = tmem_u + C::A_COL0 + sa_ * A_COLS;
                    const uint32_t done = done_bar(it);
                    if (ptx::elect_one()) {
#pragma unroll
                        for (int kk = 0; kk < GROUP / 32; ++kk)   // not PC: the first K slice overwrites the buffer
                            ptx::mma_i8_ts(d_tmem, a_tmem + 8 * kk, bd + 2 * kk, idesc, (PC || kk) ? 1u : 0u);
                        ptx::tc_commit(done);                     // stages consumed (not PC: accumulator complete)
                    }
                    __syncwarp();
                    mine = true;
                }
                if (PC && ok) {
                    // the tile is complete when the MMAs of both issuers are: a commit tracks only its own thread's
                    // (elect.sync names the same lane of a full warp every time)
                    if (ptx::elect_one()) {
                        if (mine) ptx::tc_commit(bar(TILE_DONE + buf));
                        else ptx::mbar_arrive(bar(TILE_DONE + buf));
                    }
                    __syncwarp();
                }
            }
            if (ptx::elect_one()) ptx::tc_commit(bar(FINAL + par));
            __syncwarp();
            // nothing may still be executing on the tensor core when TMEM is freed
            ptx::mbar_wait(bar(FINAL + par), 0, abort_flag);
        }
    } else if (warp < WARP_DRAIN0) {
        // short tiles leave the drain registers to spare: the unpack gets them (its loads, arithmetic and
        // TMEM stores then overlap better; measured 4 % on single-tile problems)
        if (TILE_M > 128) asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
        else asm volatile("setmaxnreg.dec.sync.aligned.u32 96;");
        // -------------------------------------------------------------------- unpack ----
        // One weight row (= one TMEM lane) per thread: 64 packed bytes -> 128 signed bytes -> 32
        // TMEM columns of this group's weight stage, k ascending (4 consecutive k per column).
        const int u = tid - WARP_UNPACK0 * 32;
        const int sw0 = blob_chunk_pos(u, 0);
        const uint32_t a_lane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + C::A_COL0;
        uint32_t it = 0;
        bool ok = true;
        for (int si = 0; ok; ++si) {
            int tile, gb, ge;
            if (!segment(si, tile, gb, ge)) break;
            for (int g = gb; g < ge; ++g, ++it) {
                const uint32_t sr = it % C::SR, pr = (it / C::SR) & 1;
                const uint32_t sa_ = it % C::SA;
                if (!(ok = ptx::mbar_wait(bar(RAW_FULL + sr), pr, abort_flag))) break;
                const uint8_t* raw = smem + C::RAW_OFF + sr * RAW_STRIDE;
                const uint32_t z = (raw[BLOB_ZERO_OFF + (u >> 1)] >> ((u & 1) * 4)) & 0xFu;
                const uint32_t kz = 0x80808080u - z * 0x01010101u;       // per byte: 0x80 - z, no borrow
                // chunk p of row u sits at position p ^ ((u >> 1) & 3): eight consecutive rows hit eight bank groups
                const uint4* rawrow = reinterpret_cast<const uint4*>(raw + u * 64);
                const uint4 w0 = rawrow[sw0], w1 = rawrow[sw0 ^ 1], w2 = rawrow[sw0 ^ 2], w3 = rawrow[sw0 ^ 3];
                // the MMAs that read this stage's previous contents have completed
                if (it >= (uint32_t)C::SA && !(ok = ptx::mbar_wait(done_bar(it - C::SA), done_parity(it - C::SA), abort_flag))) break;
                ptx::tc_fence_after_sync();
                const uint32_t a_addr = a_lane + sa_ * A_COLS;
                auto put = [&](const uint4& w, int j) {                  // 16 packed bytes = k 32j .. 32j+31
                    // words 0..3 of a chunk hold the runs of four k (a0, a2), (a1, a3), (a4, a6), (a5, a7) in their
                    // (low, high) nibbles: columns in k order are lo(x), lo(y), hi(x), hi(y), lo(z), lo(w), hi(z), hi(w)
                    ptx::tmem_st_32x8(a_addr + 8 * j,
                                      sub_zero4(w.x & 0x0F0F0F0Fu, kz), sub_zero4(w.y & 0x0F0F0F0Fu, kz),
                                      sub_zero4((w.x >> 4) & 0x0F0F0F0Fu, kz), sub_zero4((w.y >> 4) & 0x0F0F0F0Fu, kz),
                                      sub_zero4(w.z & 0x0F0F0F0Fu, kz), sub_zero4(w.w & 0x0F0F0F0Fu, kz),
                                      sub_zero4((w.z >> 4) & 0x0F0F0F0Fu, kz), sub_zero4((w.w >> 4) & 0x0F0F0F0Fu, kz));
                };
                put(w0, 0);
                put(w1, 1);
                put(w2, 2);
                put(w3, 3);
                ptx::tmem_st_wait();
                ptx::tc_fence_before_sync();
                __syncwarp();
                if (BRANCH) {
                    if (lane == 0) {
                        ptx::mbar_arrive(bar(A_FULL + sa_));
                        ptx::mbar_arrive(bar(RAW_EMPTY + sr));
                    }
                } else {
                    ptx::mbar_arrive_if(bar(A_FULL + sa_), lane == 0);
                    ptx::mbar_arrive_if(bar(RAW_EMPTY + sr), lane == 0);
                }
            }
        }
    } else {
        if (TILE_M > 128) asm volatile("setmaxnreg.inc.sync.aligned.u32 216;");
        else asm volatile("setmaxnreg.inc.sync.aligned.u32 160;");
        // --------------------------------------------------------------------- drain ----
        // Warp (q, h): TMEM lanes 32q..32q+31 (output channels), accumulator columns h*W.. (tokens).
        ptx::pdl_wait();                                        // token scales, hand-over flags, residual and output
        const int q = warp & 3, h = (warp - WARP_DRAIN0) >> 2;
        const int n_local = q * 32 + lane;
        const uint32_t lane_taddr = tmem_base + ((uint32_t)(q * 32) << 16) + h * C::W;
        // PC: this warp's part of an accumulator buffer back to zero (every MMA of a tile adds)
        auto zero_fill = [&](uint32_t taddr) {
#pragma unroll
            for (int c = 0; c < C::W; c += 8) ptx::tmem_st_32x8(taddr + c, 0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u);
            ptx::tmem_st_wait();
        };
        if (PC) {
            zero_fill(lane_taddr);
            zero_fill(lane_taddr + TILE_M);
            ptx::tc_fence_before_sync();
            __syncwarp();
        }
        if (lane == 0) {                                          // the accumulator buffers start out free
            for (int i = 0; i < C::NB; ++i) ptx::mbar_arrive(bar(ACC_EMPTY + i));
        }
        uint32_t it = 0, tcount = 0;
        bool ok = true, ready = false;                            // ready: step `it` is known to be complete
        // token scales (raw fp16 bits) and first group scale of the next segment, requested before the epilogue of
        // the current one so that their latency is not added to the time the tensor pipe waits for this warp
        uint16_t next_sa_bits[C::NCH], next_sw_bits = 0;
        bool have_next = false;
        auto request = [&](int idx) {
            int t2, gb2, ge2, nt2, mt2;
            have_next = segment(idx, t2, gb2, ge2);
            if (!have_next) return;
            tile_of(t2, nt2, mt2);
            const int mb2 = mt2 * TILE_M + h * C::W;
#pragma unroll
            for (int k = 0; k < C::NCH; ++k) {
                const int i = lane + 32 * k;
                next_sa_bits[k] = (i < C::W && mb2 + i < M) ? __ldg(sa + mb2 + i) : (uint16_t)0;
            }
            next_sw_bits = __ldg(reinterpret_cast<const uint16_t*>(packed + ((size_t)nt2 * GK + g_lo + gb2) * BLOB_BYTES +
                                                                   BLOB_SCALE_OFF + 2 * n_local));
        };
        request(0);
        for (int si = 0; ok; ++si, ++tcount) {
            int tile, gb, ge, ntile, mtile;
            if (!segment(si, tile, gb, ge)) break;
            tile_of(tile, ntile, mtile);
            const int n = ntile * TILE_N + n_local;
            const int m_base = mtile * TILE_M + h * C::W;
            const uint8_t* sw_ptr = packed + ((size_t)ntile * GK + g_lo) * BLOB_BYTES + BLOB_SCALE_OFF + 2 * n_local;
            uint64_t facc[C::W / 2];                              // pairs of neighbouring tokens
#pragma unroll
            for (int i = 0; i < C::W / 2; ++i) facc[i] = 0ull;
            auto sum = [&](int i) { const float2 t = ptx::unpack2(facc[i / 2]); return i & 1 ? t.y : t.x; };
            if (BAL && ge < G) {
                // Balanced walk: this CTA's last tile, whose later groups the next CTA summed first (they open its range): the sums
                // start from those.  Fetched here and not after the last group they are off the tail that the launch ends with,
                // and warp by warp (a flag bit each) they need no barrier of the CTA.  (4096 -> 24576 at 200 tokens 32.5 us, now
                // 31.8; 12288 -> 4096 at 1024 with residual 70.5, now 69.1)
                ok = ptx::warp_wait_bit_acquire_gpu(handover_flags + blockIdx.x + 1, 1u << (warp - WARP_DRAIN0), abort_flag);
                if (!ok) break;
                const float* slot = handover + (size_t)(blockIdx.x + 1) * (TILE_M * TILE_N);
#pragma unroll
                for (int i = 0; i < C::W; i += 2) {
                    const float* p = slot + (size_t)(h * C::W + i) * TILE_N + n_local;
                    facc[i / 2] = ptx::pack2(__float_as_uint(__ldcg(p)), __float_as_uint(__ldcg(p + TILE_N)));
                }
                __syncwarp();
                // this warp's bit back to zero for the next call
                if (lane == 0) atomicAnd(handover_flags + blockIdx.x + 1, ~(1u << (warp - WARP_DRAIN0)));
            }
            if (RES) {
                // the residual of this warp's part of the tile (W tokens x 64 bytes) is asked into L2 now; the epilogue's
                // loads then find it there
#pragma unroll
                for (int k = 0; k < C::NCH; ++k) {
                    const int m = m_base + lane + 32 * k;
                    if (lane + 32 * k < C::W && m < M)
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(residual + (size_t)m * N + (size_t)ntile * TILE_N + q * 32));
                }
            }
            // this warp's token scales, widened once per tile (rows past M get 0 and are never stored)
            float* sa_w = reinterpret_cast<float*>(smem + C::SA_OFF) + (warp - WARP_DRAIN0) * (C::NCH * 32);
            __syncwarp();
#pragma unroll
            for (int k = 0; k < C::NCH; ++k)
                if (lane + 32 * k < C::W) sa_w[lane + 32 * k] = __half2float(__ushort_as_half(next_sa_bits[k]));
            __syncwarp();
            uint16_t sw_bits = next_sw_bits;
            if (PC) {
                // One drain per tile: the buffer holds the sum of D over all groups (|sum| < 2^31 for K < 2^13 * 128).  The wait lasts
                // for the whole tile, so it parks: polling, the probes of eight warps queue up in front of the unpack's shared-memory
                // accesses (4096 -> 4096 at 1024 tokens 24.8 us with polling, 22.5 parked; 4096 -> 6144, 208 rows, 23.4 and 21.8).
                const uint32_t buf = tcount & 1u;
                const float sw = __half2float(__ushort_as_half(sw_bits));
                if (!(ok = ptx::warp_mbar_wait(bar(TILE_DONE + buf), (tcount >> 1) & 1, abort_flag))) break;
                ptx::tc_fence_after_sync();
                const uint32_t taddr = lane_taddr + buf * TILE_M;
                uint32_t v[C::NCH][32];
#pragma unroll
                for (int ch = 0; ch < C::NCH; ++ch) {
                    if (ch == C::NCH - 1 && C::LAST == 8) ptx::tmem_ld_32x8(taddr + ch * 32, reinterpret_cast<uint32_t(&)[8]>(v[ch]));
                    else ptx::tmem_ld_32x32(taddr + ch * 32, v[ch]);
                }
                ptx::tmem_ld_wait();
                zero_fill(taddr);
                ptx::tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(bar(ACC_EMPTY + buf));
#pragma unroll
                for (int ch = 0; ch < C::NCH; ++ch) {
#pragma unroll
                    for (int i = 0; i < 32; i += 2) {
                        if (ch * 32 + i < C::W) {
                            const int32_t d0 = (int32_t)v[ch][i], d1 = (int32_t)v[ch][i + 1];
                            // exact while |sum| < 2^24; beyond that one rounding of relative size 2^-24
                            facc[(ch * 32 + i) / 2] = ptx::pack2(__float_as_uint(sw * (float)d0), __float_as_uint(sw * (float)d1));
                            if (DEBUG) {
                                const int m = m_base + ch * 32 + i;
                                if (m < M) debug_partials[(size_t)m * N + n] = d0;
                                if (m + 1 < M) debug_partials[(size_t)(m + 1) * N + n] = d1;
                            }
                        }
                    }
                }
            }
            for (int g = gb; g < (PC ? gb : ge); ++g, ++it) {
                const uint32_t buf = it & (C::NB - 1);
                const float sw = __half2float(__ushort_as_half(sw_bits));
                const uint64_t sw2 = ptx::pack2(__float_as_uint(sw), __float_as_uint(sw));
                if (g + 1 < ge) sw_bits = __ldg(reinterpret_cast<const uint16_t*>(sw_ptr + (size_t)(g + 1) * BLOB_BYTES));
                // (short tiles: this warp mostly waits, and a polling loop's probes queue up in front of the unpack
                // warp's shared-memory accesses on the same scheduler; the parking wait leaves the queue alone)
                if (!ready &&
                    !(ok = (TILE_M <= 128 ? ptx::warp_mbar_wait(done_bar(it), done_parity(it), abort_flag)
                                          : ptx::warp_mbar_wait_hot(done_bar(it), done_parity(it), abort_flag)))) break;
                ptx::tc_fence_after_sync();
                const uint32_t taddr = lane_taddr + buf * TILE_M;
                // All of this warp's columns go to registers with back-to-back loads, then the buffer is
                // handed back: the MMA -> drain -> MMA round trip of a buffer, not the arithmetic
                // below, sets the pace of the pipeline.
                uint32_t v[C::NCH][32];
#pragma unroll
                for (int ch = 0; ch < C::NCH; ++ch) {
                    if (ch == C::NCH - 1 && C::LAST == 8) ptx::tmem_ld_32x8(taddr + ch * 32, reinterpret_cast<uint32_t(&)[8]>(v[ch]));
                    else ptx::tmem_ld_32x32(taddr + ch * 32, v[ch]);
                }
                // the next step's barrier, looked at under the loads' latency (past the last step: a phase that never completes)
                if (LOOK_AHEAD) ready = ptx::warp_mbar_test_wait(done_bar(it + 1), done_parity(it + 1));
                ptx::tmem_ld_wait();
                ptx::tc_fence_before_sync();
                __syncwarp();
                if (!BRANCH) ptx::mbar_arrive_if(bar(ACC_EMPTY + buf), lane == 0);
                else if (lane == 0) ptx::mbar_arrive(bar(ACC_EMPTY + buf));
#pragma unroll
                for (int ch = 0; ch < C::NCH; ++ch) {
#pragma unroll
                    for (int i = 0; i < 32; i += 2) {
                        if (ch * 32 + i < C::W) {
                            ptx::cvt_fma2(facc[(ch * 32 + i) / 2], v[ch][i], v[ch][i + 1], sw2);        // exact converts: |D| < 2^24
                            if (DEBUG) {
                                const int m = m_base + ch * 32 + i;
                                if (m < M) debug_partials[((size_t)m * GK + g_lo + g) * N + n] = (int32_t)v[ch][i];
                                if (m + 1 < M) debug_partials[((size_t)(m + 1) * GK + g_lo + g) * N + n] = (int32_t)v[ch][i + 1];
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
                // t * 128 + n of this CTA's slot, then this warp's bit of the slot's flag word (release).
                float* slot = handover + (size_t)blockIdx.x * (TILE_M * TILE_N);
#pragma unroll
                for (int i = 0; i < C::W; ++i) __stcg(slot + (size_t)(h * C::W + i) * TILE_N + n_local, sum(i));
                __syncwarp();
                if (lane == 0) ptx::red_or_release_gpu_u32(handover_flags + blockIdx.x, 1u << (warp - WARP_DRAIN0));
                continue;                       // the other CTA stores the tile
            }
            if (SPLIT) {
                // every CTA of the cluster is past its last MMA: the activation rings are free and become
                // the exchange buffers; push this thread's partials to the CTAs that own them
                ptx::cluster_sync();
                exchanged = true;
                // The tile's runs of four tokens are dealt out to the S CTAs; a thread pushes 16 bytes (its channel, four
                // tokens) at a time: slot [pusher][run of the owner][channel], channels 4 apart side by side, so that the lane
                // that sums channels 4 l .. 4 l + 3 reads beside its neighbours.
                const int slot_n = (n_local & 3) * 32 + (n_local >> 2);
                const int lo1 = run_lo(1), lo2 = S > 2 ? run_lo(2) : RUNS, lo3 = S > 3 ? run_lo(3) : RUNS;
#pragma unroll
                for (int i = 0; i < C::W; i += 4) {
                    if (m_base + i < M) {
                        const int run = h * (C::W / 4) + i / 4;
                        const int owner = (run >= lo1) + (run >= lo2) + (run >= lo3);
                        const int first = run >= lo3 ? lo3 : (run >= lo2 ? lo2 : (run >= lo1 ? lo1 : 0));
                        const uint32_t at = smem_base + C::B_OFF + (uint32_t)((slice * runs_max + run - first) * TILE_N + slot_n) * 16u;
                        ptx::st_dsmem_f32x4(ptx::map_to_cta(at, (uint32_t)owner), make_float4(sum(i), sum(i + 1), sum(i + 2), sum(i + 3)));
                    }
                }
                // This CTA's share, by the drain warps: a warp takes a run at a time (four tokens x the tile's 128 channels, four
                // to a lane, stores of 256 bytes a row; stores of 2 bytes a lane cost 8 cycles each).  The residual is asked for
                // before the second barrier, so that its round trip runs under the exchange.
                constexpr int ITEMS = (RUNS / 2 + NUM_DRAIN_WARPS - 1) / NUM_DRAIN_WARPS;                // S >= 2
                const int w8 = warp - WARP_DRAIN0, lo = run_lo(slice), cnt = run_lo(slice + 1) - lo;
                const int m_first = mtile * TILE_M + 4 * (lo + w8);                                     // items are eight runs apart
                const size_t at0 = (size_t)m_first * N + (size_t)ntile * TILE_N + 4 * lane;
                uint2 rr[RES ? ITEMS : 1][4];
                if (RES) {
#pragma unroll
                    for (int j = 0; j < ITEMS; ++j)
#pragma unroll
                        for (int t = 0; t < 4; ++t) {
                            rr[j][t] = make_uint2(0u, 0u);
                            if (w8 + 8 * j < cnt && m_first + 32 * j + t < M)
                                rr[j][t] = __ldcg(reinterpret_cast<const uint2*>(residual + at0 + (size_t)(32 * j + t) * N));
                        }
                }
                ptx::cluster_sync();                       // release after the pushes, acquire before the sums
                if (*abort_flag) break;
#pragma unroll
                for (int j = 0; j < ITEMS; ++j) {
                    if (w8 + 8 * j < cnt && m_first + 32 * j < M) {
                        float4 acc[4];                                                  // channel 4 lane + c: four tokens
#pragma unroll
                        for (int c = 0; c < 4; ++c) acc[c] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                        for (int s2 = 0; s2 < S; ++s2) {                                // rank order: deterministic
                            const uint32_t src = smem_base + C::B_OFF + (uint32_t)((s2 * runs_max + w8 + 8 * j) * TILE_N + lane) * 16u;
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                const float4 v = ptx::lds128f(src + c * 512);
                                acc[c].x += v.x; acc[c].y += v.y; acc[c].z += v.z; acc[c].w += v.w;
                            }
                        }
#pragma unroll
                        for (int t = 0; t < 4; ++t) {
                            const int m = m_first + 32 * j + t;
                            if (m < M) {
                                const float ts = __half2float(__ushort_as_half(__ldg(sa + m)));
                                float f[4];
#pragma unroll
                                for (int c = 0; c < 4; ++c) f[c] = t == 0 ? acc[c].x : (t == 1 ? acc[c].y : (t == 2 ? acc[c].z : acc[c].w));
                                uint2 o;
                                if (RES) {
                                    o.x = ptx::pack_bf16x2(fmaf(f[0], ts, __uint_as_float(rr[j][t].x << 16)), fmaf(f[1], ts, __uint_as_float(rr[j][t].x & 0xFFFF0000u)));
                                    o.y = ptx::pack_bf16x2(fmaf(f[2], ts, __uint_as_float(rr[j][t].y << 16)), fmaf(f[3], ts, __uint_as_float(rr[j][t].y & 0xFFFF0000u)));
                                } else {
                                    o.x = ptx::pack_bf16x2(f[0] * ts, f[1] * ts);
                                    o.y = ptx::pack_bf16x2(f[2] * ts, f[3] * ts);
                                }
                                *reinterpret_cast<uint2*>(y + at0 + (size_t)(32 * j + t) * N) = o;
                            }
                        }
                    }
                }
                break;                          // one tile per cluster
            }
            // Epilogue: token scale, bf16, and a transpose through shared memory so that global
            // stores are 16 bytes per lane along the channel dimension (a thread owns a channel,
            // the output is token-major).  Blocks of up to 32 tokens x this warp's 32 channels.
            uint8_t* ob = smem + C::OUT_OFF + (warp - WARP_DRAIN0) * 2048;
            const uint32_t ob_addr = smem_base + C::OUT_OFF + (warp - WARP_DRAIN0) * 2048;
            __nv_bfloat16* yrow = y + (size_t)ntile * TILE_N + q * 32 + 8 * (lane & 3);
            uint4 rv[4];
            // residual rows 8 k + lane / 4 of block b, this lane's 16-byte piece of the warp's 64-byte row (zeros past M or W)
            auto load_res = [&](int b, uint4 (&dst)[4]) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int t = b * 32 + 8 * k + (lane >> 2), m = m_base + t;
                    dst[k] = make_uint4(0u, 0u, 0u, 0u);
                    if (RES && t < C::W && m < M)
                        dst[k] = __ldcg(reinterpret_cast<const uint4*>(residual + (size_t)m * N + (size_t)ntile * TILE_N + q * 32 + 8 * (lane & 3)));
                }
            };
#pragma unroll
            for (int b2 = 0; b2 < C::NCH; ++b2) {
                // The chunk's 32 token scales go to registers first: read one by one between the stores below
                // they would each wait for the store before them (both are shared-memory accesses the compiler
                // must keep in order), a chain of 32 round trips per chunk.
                float sc[32];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const float4 t = *reinterpret_cast<const float4*>(sa_w + b2 * 32 + 4 * k);
                    sc[4 * k] = t.x; sc[4 * k + 1] = t.y; sc[4 * k + 2] = t.z; sc[4 * k + 3] = t.w;
                }
                if (RES) {
                    // The projection's output joins the residual stream, added in fp32 before the one rounding.  A block's
                    // residual (32 tokens x this warp's 32 channels) is fetched in the layout of the stores - 16 bytes per
                    // lane, rows of 64 bytes, one block ahead - and written into the output block, from which each lane
                    // reads its own channel's column back, adds, rounds and overwrites.  y may be the residual buffer:
                    // this warp reads a block before it stores it.
                    if (b2 == 0) load_res(0, rv);
                    uint4 rv_next[4];
                    if (b2 + 1 < C::NCH) load_res(b2 + 1, rv_next);
                    if (lane == 0) ptx::bulk_wait_group_read0();
                    __syncwarp();
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        *reinterpret_cast<uint4*>(ob + (8 * k + (lane >> 2)) * 64 + 16 * (lane & 3)) = rv[k];
                    __syncwarp();
#pragma unroll
                    for (int half = 0; half < 2; ++half) {
                        float rs[16];
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            rs[i] = __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(ob + (16 * half + i) * 64)[lane]);
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            if (b2 * 32 + 16 * half + i < C::W)
                                reinterpret_cast<__nv_bfloat16*>(ob + (16 * half + i) * 64)[lane] =
                                    __float2bfloat16_rn(sum(b2 * 32 + 16 * half + i) * sc[16 * half + i] + rs[i]);
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) rv[k] = rv_next[k];
                } else {
                if (lane == 0) ptx::bulk_wait_group_read0();      // the previous block's TMA store has read `ob`
                __syncwarp();
#pragma unroll
                for (int i = 0; i < 32; ++i)
                    if (b2 * 32 + i < C::W)
                        reinterpret_cast<__nv_bfloat16*>(ob + i * 64)[lane] = __float2bfloat16_rn(sum(b2 * 32 + i) * sc[i]);
                }
                if (b2 < C::NCH - 1 || C::LAST == 32) {
                    // a full block of 32 tokens: one TMA store (rows past M are clipped by the map), the warp moves on
                    ptx::fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) {
                        ptx::tma_store_2d(&tmap_y, ntile * TILE_N + q * 32, m_base + b2 * 32, ob_addr);
                        ptx::bulk_commit_group();
                    }
                } else {
                    // the 8-token tail of a 208-row tile: 16-byte stores per lane
                    __syncwarp();
                    const int row = lane >> 2;
                    const int m = m_base + b2 * 32 + row;
                    if (b2 * 32 + row < C::W && m < M) {
                        const uint4 val = *reinterpret_cast<const uint4*>(ob + row * 64 + 16 * (lane & 3));
                        *reinterpret_cast<uint4*>(yrow + (size_t)m * N) = val;
                    }
                }
            }
        }
        if (lane == 0) ptx::bulk_wait_group0();                   // every tile store of this warp has completed
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

template <int TILE_M, bool DEBUG, bool SPLIT, bool PC = false, bool BAL = false, bool RES = false>
cudaError_t launch_tile(const int8_t* qa, const uint16_t* sa, const void* packed, void* y, const void* residual, int M, int N, int K, int S,
                        void* workspace, int32_t* debug_partials, cudaStream_t stream) {
    using C = Cfg<TILE_M>;
    CUtensorMap tmap, tmap_y;
    cudaError_t te = make_qa_tensor_map(&tmap, qa, M, K, TILE_M);
    if (te != cudaSuccess) return te;
    te = make_y_tensor_map(&tmap_y, y, M, N);
    if (te != cudaSuccess) return te;

    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    static bool attr_done[64] = {false};
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    const int sms = device_sm_count();
    if (!attr_done[dev]) {
        e = cudaFuncSetAttribute(gemm_tcgen05_kernel<TILE_M, DEBUG, SPLIT, PC, BAL, RES>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 C::SMEM_ALLOC);
        if (e != cudaSuccess) return e;
        attr_done[dev] = true;
    }
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
    cfg.blockDim = dim3(TC_THREADS, 1, 1);
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
    return cudaLaunchKernelEx(&cfg, gemm_tcgen05_kernel<TILE_M, DEBUG, SPLIT, PC, BAL, RES>, tmap, tmap_y, static_cast<const uint8_t*>(packed), sa,
                              static_cast<__nv_bfloat16*>(y), static_cast<const __nv_bfloat16*>(residual), debug_partials,
                              reinterpret_cast<uint32_t*>(ws + WS_STATUS_OFF),
                              M, N, K, m_tiles, total, S, reinterpret_cast<float*>(ws + WS_SHARED_OFF),
                              reinterpret_cast<uint32_t*>(ws + WS_COUNTER_OFF));
}

// Clusters of S CTAs of the split-K kernel that the device can hold at once (S CTAs need S free SMs
// of one GPC, so this is less than SMs / S); 0 if the query fails.  Cached per device.
template <int TILE_M>
int max_active_clusters(int S) {
    static int cached[64][TC_MAX_SPLIT + 1] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64 || S < 2 || S > TC_MAX_SPLIT) return 0;
    if (cached[dev][S] == 0) {
        int n = 0;
        if constexpr (TILE_M == 64) {
            n = tcshort_max_clusters(S);
        } else {
            using C = Cfg<TILE_M>;
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3((unsigned)(S * 64), 1, 1);
            cfg.blockDim = dim3(TC_THREADS, 1, 1);
            cfg.dynamicSmemBytes = C::SMEM_ALLOC;
            cudaLaunchAttribute attr;
            attr.id = cudaLaunchAttributeClusterDimension;
            attr.val.clusterDim.x = (unsigned)S;
            attr.val.clusterDim.y = 1;
            attr.val.clusterDim.z = 1;
            cfg.attrs = &attr;
            cfg.numAttrs = 1;
            if (cudaFuncSetAttribute(gemm_tcgen05_kernel<TILE_M, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     C::SMEM_ALLOC) != cudaSuccess ||
                cudaOccupancyMaxActiveClusters(&n, gemm_tcgen05_kernel<TILE_M, false, true>, &cfg) != cudaSuccess)
                n = -1;
        }
        cached[dev][S] = n > 0 ? n : -1;
    }
    return cached[dev][S] > 0 ? cached[dev][S] : 0;
}

template <bool DEBUG, bool RES = false>
cudaError_t launch_plan(int tile_m, int S, bool balanced, const int8_t* qa, const uint16_t* sa, const int32_t* asum, const void* packed, void* y,
                        const void* residual, int M, int N, int K, void* workspace, int32_t* debug_partials, cudaStream_t stream) {
    if (tile_m == 64 && few_groups(M, K / GROUP))       // (neither split nor balanced: the planner does neither with so few groups)
        return launch_tile<64, DEBUG, false, false, false, RES>(qa, sa, packed, y, residual, M, N, K, 1, workspace, debug_partials, stream);
    if (tile_m == 64)
        return launch_gemm_tcshort(S, balanced, qa, sa, asum, packed, y, residual, M, N, K, workspace, debug_partials, stream);
    if (S > 1) {
        if (tile_m == 128) return launch_tile<128, DEBUG, true, false, false, RES>(qa, sa, packed, y, residual, M, N, K, S, workspace, debug_partials, stream);
        return launch_tile<208, DEBUG, true, false, false, RES>(qa, sa, packed, y, residual, M, N, K, S, workspace, debug_partials, stream);
    }
    if (balanced) {
        if (tile_m == 128) return launch_tile<128, DEBUG, false, false, true, RES>(qa, sa, packed, y, residual, M, N, K, 1, workspace, debug_partials, stream);
        return launch_tile<208, DEBUG, false, false, true, RES>(qa, sa, packed, y, residual, M, N, K, 1, workspace, debug_partials, stream);
    }
    if (tile_m == 128) return launch_tile<128, DEBUG, false, false, false, RES>(qa, sa, packed, y, residual, M, N, K, 1, workspace, debug_partials, stream);
    return launch_tile<208, DEBUG, false, false, false, RES>(qa, sa, packed, y, residual, M, N, K, 1, workspace, debug_partials, stream);
}

template <bool DEBUG>
cudaError_t launch_per_channel(int tile_m, const int8_t* qa, const uint16_t* sa, const void* packed, void* y, int M, int N, int K,
                               void* workspace, int32_t* debug_sums, cudaStream_t stream) {
    if (tile_m == 64) return launch_tile<64, DEBUG, false, true>(qa, sa, packed, y, nullptr, M, N, K, 1, workspace, debug_sums, stream);
    if (tile_m == 128) return launch_tile<128, DEBUG, false, true>(qa, sa, packed, y, nullptr, M, N, K, 1, workspace, debug_sums, stream);
    return launch_tile<208, DEBUG, false, true>(qa, sa, packed, y, nullptr, M, N, K, 1, workspace, debug_sums, stream);
}

}  // namespace

// Tile height and K split for an [M, N, K] problem, from a cost model fitted to measurements on B200: a CTA spends
// a fixed time on launch, set-up and pipeline fill, then one per 128-k group of every tile it walks, by height (TC_COST);
// a K split into S slices costs TC_SPLIT_NS for the cluster exchange.  Tall tiles are cheapest per token (2.6,
// 3.6 and 4.2 ns per token and group) and win when there are several waves of them, short ones when a tall tiling would
// leave SMs idle, and a K split when even the shortest tiling does.  (Against an exhaustive sweep of height, split and
// walk at 20 to 400 tokens on eight layers the choice is within 6 % of the best.)
long tcgen05_plan(int M, int N, int K, int sms, int* tile_m, int* split, int* balanced) {
    const int heights[3] = {208, 128, 64};
    const int n_tiles = N / TILE_N, G = K / GROUP;
    const TcCost& cost = few_groups(M, G) ? TC_COST_FEW : (M > 32 && G < 16 ? TC_COST_MEDIUM : TC_COST);
    long best_ns = -1;
    *tile_m = 64;
    *split = 1;
    *balanced = 0;
    for (int i = 0; i < 3; ++i) {
        if (heights[i] > 64 && M <= heights[i + 1]) continue;        // the next height down already covers M in one tile
        const long tiles = (long)((M + heights[i] - 1) / heights[i]) * n_tiles;
        const long waves = (tiles + sms - 1) / sms;
        const long group_ns = M <= 32 ? TC_GROUP_32_NS : cost.group[i];
        const long fixed_ns = cost.fixed[i] + (waves - 1) * cost.tile[i];
        for (int S = 1; S <= TC_MAX_SPLIT; ++S) {
            if (S > 1) {
                if (tiles * S > sms || G / S < 4) break;
                const int room = i == 0 ? max_active_clusters<208>(S) : (i == 1 ? max_active_clusters<128>(S) : max_active_clusters<64>(S));
                if (tiles > room) continue;                          // the clusters must all be resident at once
            }
            const long ns = fixed_ns + waves * group_ns * ((G + S - 1) / S) + TC_SPLIT_NS[i][S];
            if (best_ns < 0 || ns < best_ns) {                        // ties: taller tile, fewer slices
                best_ns = ns; *tile_m = heights[i]; *split = S;
                *balanced = 0;
            }
            // no split, more tiles than SMs: an even share of all tiles x groups units per CTA, at the price of
            // handing partial tiles over between neighbours
            if (S == 1 && G > TC_FEW_GROUPS && tiles > sms && tiles % sms != 0 && sms <= HANDOVER_SLOTS && handover_bytes(M, N, K) > 0) {
                const long nb = fixed_ns + group_ns * ((tiles * G + sms - 1) / sms) * TC_BALANCE_PERCENT[i] / 100 + TC_BALANCE_NS[i];
                if (nb < best_ns) { best_ns = nb; *tile_m = heights[i]; *split = 1; *balanced = 1; }
            }
        }
    }
    return best_ns;                                                   // the estimate, for the caller's choice of kernel family
}

cudaError_t launch_gemm_tcgen05(const int8_t* qa, const uint16_t* sa, const int32_t* asum, const void* packed, void* y, const void* residual,
                                int M, int N, int K, void* workspace, int32_t* debug_partials,
                                cudaStream_t stream) {
    int tile_m = 64, S = 1, balanced = 0;
    tcgen05_plan(M, N, K, device_sm_count(), &tile_m, &S, &balanced);
    if (residual)                                   // (no partials dump in this form)
        return launch_plan<false, true>(tile_m, S, balanced != 0, qa, sa, asum, packed, y, residual, M, N, K, workspace, nullptr, stream);
    if (debug_partials)
        return launch_plan<true>(tile_m, S, balanced != 0, qa, sa, asum, packed, y, nullptr, M, N, K, workspace, debug_partials, stream);
    return launch_plan<false>(tile_m, S, balanced != 0, qa, sa, asum, packed, y, nullptr, M, N, K, workspace, debug_partials, stream);
}

// The same pipeline with one drain per tile: for weights whose scale does not change along K.
// debug_sums, if not null, receives the int32 sum over all groups per (token, channel), [M][N].
cudaError_t launch_gemm_tcgen05_per_channel(const int8_t* qa, const uint16_t* sa, const void* packed, void* y,
                                            int M, int N, int K, void* workspace, int32_t* debug_sums,
                                            cudaStream_t stream) {
    const int tile_m = per_channel_tile_height(M, N / TILE_N, K / GROUP, device_sm_count());
    if (debug_sums)
        return launch_per_channel<true>(tile_m, qa, sa, packed, y, M, N, K, workspace, debug_sums, stream);
    return launch_per_channel<false>(tile_m, qa, sa, packed, y, M, N, K, workspace, nullptr, stream);
}

}  // namespace w4a8
