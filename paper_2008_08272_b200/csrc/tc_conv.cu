// Implicit-GEMM convolution on the tcgen05 tensor cores (TF32 multiply, fp32 accumulate)
// for ONNX Conv (Sec. 4.1) with any kernel size, stride, dilation, padding and groups.
//
// GEMM view: rows = output pixels ("anchors" in slot space, see tc_conv_plan.h), columns =
// output channels, reduction = input channels x filter taps.  The im2col matrix is never
// formed; per block of KB input channels
//   warp 0      stages the raw NCHW rows the tile touches into shared memory by TMA
//               (zero fill outside the tensor);
//   warps 4-15  re-lay them into the K-major "4 channels x slot" operand layout of the MMA,
//               rounding fp32 to TF32 (nearest) and writing zeros for padding;
//   warp 1      streams the pre-packed, pre-rounded weights by bulk copy;
//   warp 2      issues, for every tap, tcgen05.mma on the SAME activation tile at a start address
//               shifted by the tap's slot offset, accumulating in TMEM;
//   warps 16-23 read finished accumulators back (tcgen05.ld), add bias, apply Relu and store NCHW
//               with lanes along consecutive pixels (coalesced); when a tile's accumulators fill at
//               most half of TMEM it holds two sets, so this overlaps the next tile's MMAs.
// CTA pairs (kCtas = 2): two CTAs of a cluster share one tile of 2 x MT x 128 pixels.  Each stages
// its own pixels and HALF of the tile's weight rows; the even CTA issues cta_group::2 MMAs
// (M = 256) that read both CTAs' shared memory and write each CTA's rows into its own TMEM.  Per
// CTA this halves the weight bytes fetched from L2 and the weight bytes the tensor pipe reads from
// shared memory per flop, the two limits of the single-CTA form.  Stage hand-over: the odd CTA's
// epilogue warps arrive directly on the even CTA's barriers, its MMA warp forwards "my weights have
// landed", its relay warp (warp 3) "my operand stage is written", and stage releases come back by
// multicast commit.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "common.h"
#define ONNXB_DEBUG_HOOKS_CONV
#include "debug_hooks.cuh"
#include "pack_weights.cuh"
#include "tc_common.cuh"
#include "tc_conv_plan.h"
#include "tc_host.h"

namespace onnxb {

namespace {

using namespace tc;

// Warps: raw producer, weight producer, MMA issuer, relay, then 12 transform warps and 8 epilogue warps: 768 threads,
// 80 registers each.  The forms of the kernel below stay within them without a spill (those with an addend have one to three words),
// on purpose: with 227 KB of shared memory per CTA next to no L1 is left, and a value spilled in a transform loop is a
// trip to L2 (40 to 90 bytes of spills, while the loops were being written, cost 7 of 51 us on the 64-channel 56x56
// layer at batch 64, 23 of 101 on the 7x7/2 first layer).
constexpr int kXformWarps = 12, kXformThreads = kXformWarps * 32, kEpiWarps = 8;
constexpr int kRelayWarp = 3;               // odd CTA of a pair: passes "operand stage written" on to the issuing CTA
constexpr int kFirstXformWarp = 4, kFirstEpiWarp = kFirstXformWarp + kXformWarps;
constexpr int kThreads = (kFirstEpiWarp + kEpiWarps) * 32;
constexpr int kMaxUnits = 2560;             // (slot, chunk) pairs of an A stage at most
// units of an A stage one transform thread may own (see there): blocks of one chunk, or of several
constexpr int kOwnedThin = (kMaxUnits + kXformThreads - 1) / kXformThreads, kOwnedThick = 2;
constexpr int kMaxRawStages = 4;
constexpr int kMaxAStages = 3;
constexpr int kMaxSpb = 9;                 // K-steps per weight stage (the MMA issue loop is unrolled over them)
constexpr int kMaxBStages = 12;
constexpr int kSmemLimit = 232448;
constexpr int kBarBytes = 512;
constexpr int kSegBytes = 256;             // >= sizeof(TcConvSegs)
constexpr int kBiasBytes = 8 * 128;        // 32 biases per epilogue warp
static_assert(sizeof(TcConvSegs) <= kSegBytes, "segment table does not fit its slot");

enum { kNoAddend, kAddendNear, kAddendFar, kRoundedY };       // kRoundedY: no addend, and Y is rounded to TF32 (a form of its own: three instructions per output)

struct Bars {
    uint64_t raw_full[kMaxRawStages], raw_empty[kMaxRawStages], a_full[kMaxAStages], a_empty[kMaxAStages];
    uint64_t a_done[kMaxAStages];            // odd CTA of a pair: its transform warps have written the stage
    uint64_t b_full[kMaxBStages], b_empty[kMaxBStages];
    uint64_t acc_full[2], acc_empty[2];
    uint64_t seg_full[2], seg_empty[2];      // segment tables, one per tile parity
    uint64_t recv_full;                      // split: all partial sums of this CTA's channels have arrived
    uint32_t tmem_holder;
};
static_assert(sizeof(Bars) <= kBarBytes, "barrier block too large");

// ------------------------------------------------------------------ weight packing
// Packed layout: [group][channel tile][CTA of the pair][channel block][K-step][chunk 0/1][row BNH][4],
// i.e. for each K-step the exact shared-memory image of one CTA's part of the K-major B operand: two
// 16-byte chunks (4 reduction terms each) per output channel, rows 16 bytes apart.  Values are rounded to TF32 (nearest);
// rows past the group's channels, channels past Cg and unpaired taps are zero.
// Launched with programmatic stream serialization: it may become resident while the previous kernel
// of the stream drains, and waits (pdl_wait) before it touches W or the workspace.
__global__ void __launch_bounds__(kPackThreads) pack_weights_kernel(const __grid_constant__ TcConvPlan g, const float *__restrict__ W, float4 *__restrict__ out) {
    pdl_launch_dependents();
    pack_weights(g, W, g.ctiles * g.ctas, g.BNH, g.KB, [&](size_t tile, int cb, int step, int half, int row, const float (&v)[4]) {
        out[(((tile * g.ncb + cb) * g.n_steps + step) * 2 + half) * g.BNH + row] = make_float4(round_tf32(v[0]), round_tf32(v[1]), round_tf32(v[2]), round_tf32(v[3]));
    });
}

// Channel blocks are summed in a rotated order that differs from tile to tile: CTAs working at the
// same time then stream different parts of the (shared) packed weights, instead of all asking the
// same L2 lines at the same moment.
__device__ __forceinline__ int cb_rotation(long long tile, int ncb) { return (int)((tile * 5 + 3) % ncb); }

// TMEM columns of a split tile: its one accumulator, in the sizes that smem_with_tmem knows
__host__ __device__ constexpr uint32_t split_tmem_cols(int BN) { return BN <= 128 ? 128u : 256u; }
// shared memory for its partial sums
__host__ __device__ constexpr int split_recv_bytes(int split, int cols_per) { return split * cols_per * 512; }

// ------------------------------------------------------------------ main kernel
// kAddend: the epilogue also adds a tensor laid out like Y (a residual connection) before the Relu; kAddendFar asks for it ahead
// of time.  Separate instantiations, so that one form's register allocation and instruction schedule do not disturb another's
// (the code that asks ahead, present but not executed, cost others of the layers with an addend up to 13 %).
// kSplit: the problem has few tiles, so a cluster of g.split CTAs shares one: CTA r reduces the channel blocks
// [r * cb_per, (r + 1) * cb_per) and finishes one slice of the tile's channels.  The epilogue warps write each partial
// sum from TMEM straight into the shared memory of the CTA that finishes it (st.async, counted on an mbarrier there);
// that CTA adds them in rank order.  Bound: latency, about 12,700 cycles for one 28x28 image, of which 3,000 are set-up
// and waiting for the previous kernel, 2,800 the first block's way to the tensor core and 1,900 the exchange (reading
// the peers' partial tiles between two cluster barriers took 2,200 more).  One 14x14 image, 256 -> 256 channels: 24 us
// unsplit, 8.6 split over 8; 28x28, 128 channels 15.7 -> 8.3.
// kThin: blocks of one 4-channel chunk (tap pairs).
template <int kCtas, int kAddend, bool kThin, bool kSplit>
__global__ void __launch_bounds__(kThreads, 1)
tc_conv_kernel(const __grid_constant__ CUtensorMap tmX, const TcConvPlan g, const float *__restrict__ X,
               const float *__restrict__ Wpk, const float *__restrict__ bias, const float *__restrict__ R,
               float *__restrict__ Y, unsigned int *err) {
    constexpr int kOwned = kThin ? kOwnedThin : kOwnedThick;
    constexpr bool kAdd = kAddend == kAddendNear || kAddend == kAddendFar, kLinear = kThin && kAddend != kAddendNear;
    // may stage rows (raw_mode 2): the thin ones; but the schedule that the compiler finds for those with an addend, whose epilogue has
    // no register to spare, is the better one with that code in place (64 -> 64 3x3 56x56 batch 32 23.8 against 25.3 us)
    constexpr bool kRows = kThin || kAdd;
    extern __shared__ uint8_t smem_raw[];
    // 1024-byte alignment by pointer arithmetic on the shared array itself, so that the compiler
    // keeps treating everything derived from it as shared memory (LDS/STS, not generic accesses)
    uint8_t *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    uint8_t *a_st = smem;
    uint8_t *raw_st = a_st + (size_t)g.na_stages * g.a_stage_bytes;
    uint8_t *b_st = raw_st + (size_t)g.nr_stages * g.raw_stage_bytes;
    uint8_t *seg_st = b_st + (size_t)g.nb_stages * g.b_stage_bytes;
    uint8_t *bias_st = seg_st + kMaxRawStages * kSegBytes;
    Bars *bars = reinterpret_cast<Bars *>(bias_st + kBiasBytes);
    uint8_t *recv_st = reinterpret_cast<uint8_t *>(bars) + kBarBytes;        // split: partial sums from every CTA

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) LOG(8, 0);
    const int tile_rows = g.MT * 128;
    // CTA pair: rank within the cluster, and the tiles this CTA (pair) walks
    const uint32_t rank = kCtas == 2 ? cluster_ctarank() : 0u;
    const int per_tile = kSplit ? g.split : kCtas;             // CTAs working on one tile
    const long long first_tile = blockIdx.x / per_tile, tile_step = gridDim.x / per_tile;
    const int cb_lo = kSplit ? (int)cluster_ctarank() * g.cb_per : 0;                  // channel blocks of this CTA
    const int cb_cnt = kSplit ? min(g.ncb - cb_lo, g.cb_per) : g.ncb;
    const int cgt = g.ctiles * g.group;        // channel tiles over all groups
    // split: the channels of the tile that this CTA finishes (whole groups of four)
    const int tile_ch = min(g.BN, g.Mg - (int)(first_tile % cgt) % g.ctiles * g.BN), tile_ch4 = (tile_ch + 3) & ~3;
    const int col_lo = kSplit ? (int)cluster_ctarank() * g.cols_per : 0, col_hi = min(tile_ch4, col_lo + g.cols_per);
    // accumulator placement in TMEM: two alternating sets when one set fits in 256 columns
    const bool acc_dbl = g.MT == 1 || g.BN <= 128;
    const uint32_t mt_cols = acc_dbl ? 128u : 256u;     // column distance between a CTA's two accumulators

    if (kSplit && warp == kRelayWarp) {
        // a barrier of each kind per lane: one thread alone takes a thousand cycles for them (which the other
        // forms hide behind the previous kernel)
        if (lane < g.nr_stages) {
            mbar_init(&bars->raw_full[lane], 1);
            mbar_init(&bars->raw_empty[lane], kXformWarps);
        }
        if (lane < g.na_stages) {
            mbar_init(&bars->a_full[lane], kXformWarps);
            mbar_init(&bars->a_empty[lane], 1);
        }
        if (lane < g.nb_stages) {
            mbar_init(&bars->b_full[lane], 1);
            mbar_init(&bars->b_empty[lane], 1);
        }
        if (lane < 2) {
            mbar_init(&bars->acc_full[lane], 1);
            mbar_init(&bars->acc_empty[lane], kEpiWarps);
            mbar_init(&bars->seg_full[lane], 1);
            mbar_init(&bars->seg_empty[lane], kXformWarps);
        }
        if (lane == 31) {
            mbar_init(&bars->recv_full, 1);
            mbar_arrive_expect_tx(&bars->recv_full, (uint32_t)(max(col_hi - col_lo, 0) * 512 * g.split));
        }
        mbar_fence_init();
    }
    if (!kSplit && threadIdx.x == 0) {
        for (int s = 0; s < g.nr_stages; ++s) {
            mbar_init(&bars->raw_full[s], 1);
            mbar_init(&bars->raw_empty[s], kXformWarps);
        }
        for (int s = 0; s < g.na_stages; ++s) {
            // waited on by the issuing CTA only: its own transform warps, plus one message from the peer
            mbar_init(&bars->a_full[s], kCtas == 2 ? (g.relay ? kXformWarps + 1 : 2 * kXformWarps) : kXformWarps);
            mbar_init(&bars->a_done[s], kXformWarps);
            mbar_init(&bars->a_empty[s], 1);
        }
        for (int s = 0; s < g.nb_stages; ++s) {
            // issuing CTA of a pair: its own producer plus the peer's "landed" message
            mbar_init(&bars->b_full[s], (kCtas == 2 && rank == 0) ? 2 : 1);
            mbar_init(&bars->b_empty[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(&bars->acc_full[s], 1);
            mbar_init(&bars->acc_empty[s], kEpiWarps * kCtas);
            mbar_init(&bars->seg_full[s], 1);
            mbar_init(&bars->seg_empty[s], kXformWarps);
        }
        mbar_fence_init();
        if (g.raw_mode == 0) prefetch_tmap(&tmX);
    }
    if (kSplit && threadIdx.x == 0 && g.raw_mode == 0) prefetch_tmap(&tmX);
    if (warp == 2) {
        tmem_alloc(&bars->tmem_holder, kSplit ? split_tmem_cols(g.BN) : 512);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = bars->tmem_holder;
    if (kCtas == 2) cluster_sync_all();     // the peer's barriers exist before anything arrives on them
    if (kSplit) cluster_arrive();           // (waited for when the partial sums go out)
    pdl_launch_dependents();
    // Everything above overlapped the previous kernel's tail, and so does each role's own set-up below:
    // the threads that touch global memory (the two producers, the epilogue warps) wait for the previous
    // kernel just before their first access; the others only ever see what those threads hand them.

    if (warp == 0) {
        // ------------------------------------------------------------ raw activation producer
        if (elect_one()) {
            int rs = 0;
            uint32_t rphase = 0, tile_it = 0;
            const long long HW = (long long)g.H * g.W;
            const long long planes_total = (long long)g.N * g.C;
            const int KB = g.KB, ncb = cb_cnt, box_floats = g.KBR * g.BOXP;
            for (long long t = first_tile; t < g.total_tiles; t += tile_step) {
                const int ct_all = (int)(t % cgt);
                const int grp = ct_all / g.ctiles;
                const long long G0 = ((t / cgt) * kCtas + rank) * tile_rows;
                // The segment table is the same for every channel block of the tile.  Two tables
                // alternate by tile; the transform warps hand a table back once they have turned it
                // into their per-thread offsets, so it is ready long before the tile's data lands.
                const uint32_t sp = tile_it & 1u;
                mbar_wait(&bars->seg_empty[sp], ((tile_it >> 1) & 1u) ^ 1u, err, 20);
                TcConvSegs *segs = reinterpret_cast<TcConvSegs *>(seg_st + sp * kSegBytes);
                tc_conv_segments(g, G0, *segs);
                mbar_arrive(&bars->seg_full[sp]);
                ++tile_it;
                if (tile_it == 1) {
                    pdl_wait();
                    LOG(8, 1);
                }
                const int nseg = segs->nseg;
                const uint32_t tile_bytes = (uint32_t)segs->total_floats * 4u;
                const int rot = kSplit ? cb_lo : cb_rotation(t, ncb);
                for (int cb = 0; cb < ncb; ++cb) {
                    mbar_wait(&bars->raw_empty[rs], rphase ^ 1, err, 11);
                    LOG(0, cb);
                    float *dst = reinterpret_cast<float *>(raw_st + (size_t)rs * g.raw_stage_bytes);
                    const int cbx = kSplit || cb + rot < ncb ? cb + rot : cb + rot - ncb;
                    const int c0 = grp * g.Cg + cbx * KB;
                    if (g.raw_mode == 0) {
                        mbar_arrive_expect_tx(&bars->raw_full[rs], tile_bytes);
                        for (int i = 0; i < nseg; ++i) {
                            // (channel-major: all of it in the first segment)
                            const int plane0 = g.x_cm ? c0 : (segs->n_first + i) * g.C + c0;
                            const int nbox = segs->nbox[i], f0 = segs->f0[i] + (g.x_cm ? segs->n_first * g.H * g.W : 0);
                            float *d = dst + segs->base[i];
                            for (int j = 0; j < nbox; ++j)
                                tma_load_2d(d + j * box_floats, &tmX, &bars->raw_full[rs], f0 + j * g.BOXP, plane0);
                        }
                    } else if (kRows && g.raw_mode == 2) {
                        // the rows of every channel that exists, one copy each
                        const int chans = min(KB, g.Cg - cbx * KB);
                        mbar_arrive_expect_tx(&bars->raw_full[rs], (uint32_t)chans * tile_bytes);
                        for (int i = 0; i < nseg; ++i) {
                            const uint32_t bytes = (uint32_t)segs->nbox[i] * 4u;
                            const float *x = X + ((long long)(segs->n_first + i) * g.C + c0) * HW + segs->f0[i];
                            float *d = dst + segs->base[i];
                            if (bytes)
                                for (int c = 0; c < chans; ++c) bulk_load_1d(d + c * g.BOXP, x + c * HW, bytes, &bars->raw_full[rs]);
                        }
                    } else {
                        // whole-image slabs [channel][H*W]; clip at the end of X
                        uint32_t total = 0;
                        for (int i = 0; i < nseg; ++i) {
                            if (!segs->nbox[i]) continue;
                            long long nch = planes_total - ((long long)(segs->n_first + i) * g.C + c0);
                            if (nch > g.KBR) nch = g.KBR;
                            if (nch > 0) total += (uint32_t)(nch * HW * 4);
                        }
                        mbar_arrive_expect_tx(&bars->raw_full[rs], total);
                        for (int i = 0; i < nseg; ++i) {
                            if (!segs->nbox[i]) continue;
                            const long long plane0 = (long long)(segs->n_first + i) * g.C + c0;
                            long long nch = planes_total - plane0;
                            if (nch > g.KBR) nch = g.KBR;
                            if (nch > 0)
                                bulk_load_1d(dst + segs->base[i], X + plane0 * HW, (uint32_t)(nch * HW * 4),
                                             &bars->raw_full[rs]);
                        }
                    }
                    if (++rs == g.nr_stages) { rs = 0; rphase ^= 1; }
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ weight producer
        if (elect_one()) {
            int bs = 0;
            uint32_t bphase = 0;
            const long long per_ct = (long long)g.ncb * g.n_steps * g.b_step_bytes;   // bytes per channel tile and CTA
            const int nb = g.nb_stages, ncb = cb_cnt, b_steps = g.b_steps, spb = g.spb, n_steps = g.n_steps;
            const uint32_t stage_bytes = (uint32_t)g.b_stage_bytes, step_bytes = (uint32_t)g.b_step_bytes;
            pdl_wait();             // the packed weights may come from the kernel just before this one
            for (long long t = first_tile; t < g.total_tiles; t += g.b_resident ? g.total_tiles : tile_step) {
                const int ct_all = (int)(t % cgt);
                const uint8_t *tile_src = reinterpret_cast<const uint8_t *>(Wpk) + (ct_all * kCtas + (int)rank) * per_ct;
                const int rot = kSplit ? cb_lo : cb_rotation(t, ncb);
                for (int cb = 0; cb < ncb; ++cb) {
                    const int cbx = kSplit || cb + rot < ncb ? cb + rot : cb + rot - ncb;
                    const uint8_t *src = tile_src + (long long)cbx * n_steps * step_bytes;
                    for (int bstep = 0; bstep < b_steps; ++bstep) {
                        const uint32_t bytes = (uint32_t)min(spb, n_steps - bstep * spb) * step_bytes;
                        mbar_wait(&bars->b_empty[bs], bphase ^ 1, err, 12);
                        LOG(1, cb * b_steps + bstep);
                        mbar_arrive_expect_tx(&bars->b_full[bs], bytes);
                        bulk_load_1d(b_st + (size_t)bs * stage_bytes, src, bytes, &bars->b_full[bs]);
                        src += bytes;
                        if (++bs == nb) { bs = 0; bphase ^= 1; }
                    }
                }
            }
        }
    } else if (warp == 2) {
        // ------------------------------------------------------------ MMA issuer
        // One thread issues every MMA.  Operands are no-swizzle K-major: rows 16 bytes apart, 8-row
        // groups 128 bytes apart (SBO), the two 16-byte K chunks of one instruction LBO apart.  For
        // A the per-step table holds offset and LBO (a chunk pitch, or the distance between two taps);
        // all descriptor words are precomputed, a step costs a table read and a few adds.
        if (kCtas == 2 && rank != 0) {
            // Odd CTA of a pair: the even CTA issues the MMAs.  Tell it when each of this CTA's weight
            // stages has landed (everything else reaches its barriers directly).
            if (elect_one()) {
                const uint32_t peer_b_full = map_to_cta(smem_u32(&bars->b_full[0]), 0);
                const int ncb = g.ncb, nb = g.nb_stages, b_steps = g.b_steps;
                int bs = 0;
                uint32_t bphase = 0;
                for (long long t = first_tile; t < g.total_tiles; t += g.b_resident ? g.total_tiles : tile_step) {
                    for (int i = 0; i < ncb * b_steps; ++i) {
                        mbar_wait(&bars->b_full[bs], bphase, err, 19);
                        mbar_arrive_remote(peer_b_full + (uint32_t)bs * 8u);
                        if (++bs == nb) { bs = 0; bphase ^= 1; }
                    }
                }
            }
        } else if (elect_one()) {
            const uint32_t desc_hi = (128u >> 4) | (1u << 14);                 // SBO = 128, descriptor version 1
            const uint32_t a_base16 = (smem_u32(a_st) >> 4) & 0x3FFFu;
            const uint32_t b_lo0 = ((smem_u32(b_st) >> 4) & 0x3FFFu) | (((uint32_t)g.BNH * 16u >> 4) << 16);
            const uint32_t a_stage16 = (uint32_t)g.a_stage_bytes >> 4, b_stage16 = (uint32_t)g.b_stage_bytes >> 4;
            const uint32_t b_step16 = (uint32_t)g.b_step_bytes >> 4;
            const uint32_t idesc = g.idesc;
            const int n_steps = g.n_steps, ncb = cb_cnt, nb = g.nb_stages, spb = g.spb, b_steps = g.b_steps;
            const bool two = g.MT == 2, resident = g.b_resident != 0;
            int as = 0, bs = 0;
            uint32_t aphase = 0, bphase = 0, it = 0;
            PROF_DECL;
            for (long long t = first_tile; t < g.total_tiles; t += tile_step, ++it) {
                const uint32_t ab = acc_dbl ? (it & 1u) : 0u, use = acc_dbl ? (it >> 1) : it;
                const uint32_t d0 = tmem_base + ab * 256u, d1 = d0 + mt_cols;
                if (kCtas == 2) mbar_wait_cluster(&bars->acc_empty[ab], (use & 1u) ^ 1u, err, 13);
                else mbar_wait(&bars->acc_empty[ab], (use & 1u) ^ 1u, err, 13);
                tc_fence_after_sync();
                PROF_MARK(0);
                uint32_t accumulate = 0;
                for (int cb = 0; cb < ncb; ++cb) {
                    if (kCtas == 2) mbar_wait_cluster(&bars->a_full[as], aphase, err, 14);
                    else mbar_wait(&bars->a_full[as], aphase, err, 14);
                    PROF_MARK(1);
                    LOG(2, cb);
                    const uint32_t a_lo = a_base16 + (uint32_t)as * a_stage16;
                    for (int bstep = 0; bstep < b_steps; ++bstep) {
                        if (!resident || it == 0) {
                            if (kCtas == 2) mbar_wait_cluster(&bars->b_full[bs], bphase, err, 15);
                            else mbar_wait(&bars->b_full[bs], bphase, err, 15);
                        }
                        tc_fence_after_sync();
                        PROF_MARK(2);
                        LOG(3, cb * b_steps + bstep);
                        // One thread issues everything, so every instruction here costs its full latency: fetch
                        // the stage's table entries together, then issue the MMAs back to back with nothing
                        // but adds in between (a full stage as straight-line code).
                        const int s0 = bstep * spb, cnt = min(n_steps - s0, spb);
                        uint32_t bl = b_lo0 + (uint32_t)bs * b_stage16;
                        auto mma = [&](uint32_t d, uint32_t al) {
                            if (kCtas == 2) mma_tf32_lohi_pair(d, al, desc_hi, bl, desc_hi, idesc, accumulate);
                            else mma_tf32_lohi(d, al, desc_hi, bl, desc_hi, idesc, accumulate);
                        };
                        auto step = [&](uint32_t sa_j) {
                            mma(d0, a_lo + sa_j);
                            if (two) mma(d1, a_lo + sa_j + 128u);
                            accumulate = 1;
                            bl += b_step16;
                        };
                        if (cnt == kMaxSpb) {
                            uint32_t sa[kMaxSpb];
#pragma unroll
                            for (int j = 0; j < kMaxSpb; ++j) sa[j] = g.step_a[s0 + j];
#pragma unroll
                            for (int j = 0; j < kMaxSpb; ++j) step(sa[j]);
                        } else {
#pragma unroll 4
                            for (int j = 0; j < cnt; ++j) step(g.step_a[s0 + j]);
                        }
                        if (!resident) {
                            if (kCtas == 2) mma_commit_pair(&bars->b_empty[bs]);
                            else mma_commit(&bars->b_empty[bs]);
                        }
                        if (++bs == nb || (resident && bstep == b_steps - 1)) { bs = 0; bphase ^= 1; }
                        PROF_MARK(3);
                    }
                    if (kCtas == 2) mma_commit_pair(&bars->a_empty[as]);
                    else mma_commit(&bars->a_empty[as]);
                    LOG(4, cb);
                    if (++as == g.na_stages) { as = 0; aphase ^= 1; }
                }
                if (kCtas == 2) mma_commit_pair(&bars->acc_full[ab]);
                else mma_commit(&bars->acc_full[ab]);
                PROF_MARK(4);
            }
            PROF_FLUSH(0);
        }
    } else if (warp == kRelayWarp) {
        // ------------------------------------------------------------ operand-stage relay (odd CTA of a pair)
        // The issuing CTA's tensor core reads this CTA's operand stage, so the transform warps' writes must
        // be released at cluster scope before the issuing CTA hears of them.  That fence stalls its thread
        // for about a thousand cycles; done by each transform warp it cost them a quarter of their time.
        // They arrive on a barrier of their own CTA instead (CTA scope: cheap), and this thread, which has
        // nothing else to do, acquires that, fences at cluster scope (release is cumulative: it covers what
        // it acquired) and arrives on the issuing CTA's barrier.
        if (kCtas == 2 && rank != 0 && g.relay && elect_one()) {
            const uint32_t peer_a_full = map_to_cta(smem_u32(&bars->a_full[0]), 0);
            const int ncb = g.ncb, na = g.na_stages;
            int as = 0;
            uint32_t aphase = 0;
            for (long long t = first_tile; t < g.total_tiles; t += tile_step) {
                for (int cb = 0; cb < ncb; ++cb) {
                    mbar_wait(&bars->a_done[as], aphase, err, 22);
                    mbar_arrive_remote_release(peer_a_full + (uint32_t)as * 8u);
                    if (++as == na) { as = 0; aphase ^= 1; }
                }
            }
        }
    } else if (warp < kFirstEpiWarp) {
        // ------------------------------------------------------------ transform warps
        const int xt = (warp - kFirstXformWarp) * 32 + lane;
        const int cp = g.raw_mode == 1 ? g.H * g.W : g.BOXP;    // channel pitch inside the raw stage
        const int per_stage_slots = g.planes * g.SLOTS;
        const int KB = g.KB, ncb = cb_cnt, box_floats = g.KBR * g.BOXP, nr = g.nr_stages;
        // Work units: one slot and `cpu` of its 4-channel chunks (each four raw reads and one 16-byte operand row);
        // unit u = chunk group * slots + slot, and this thread owns units xt, xt + kXformThreads, ...  The offset
        // arithmetic is per unit, not per chunk, and few units keep everything in registers: a spilled value
        // costs a trip to L2 here (shared memory leaves next to no L1).
        const int cpu = kThin ? 1 : g.chunks_per_unit, units = per_stage_slots * (kThin ? 1 : g.chunk_groups);
        const int nu = (units - xt + kXformThreads - 1) / kXformThreads;
        int rs = 0, as = 0;
        uint32_t rphase = 0, aphase = 0, tile_it = 0;
        PROF_DECL;
        const uint32_t a_full_addr = kCtas == 2 ? map_to_cta(smem_u32(&bars->a_full[0]), 0) : 0u;
        // What does not depend on the tile is worked out once: where a unit's operand row goes, and
        // which slot of which parity plane it reads.
        uint32_t udst[kOwned];                     // byte offset of the unit's operand row inside an A stage | chunk group (thin: just xt * 16, and on from there)
        uint32_t ujp[kOwned];                      // slot columns << 16 | slot rows from the tile's first slot (rows << 12 | columns where no rule below compares them)
        uint32_t upix[kOwned];                     // the same distance in pixels, the plane's and the padding's share added: rows << 16 | columns (signed)
        int ulin[kLinear ? kOwned : 1];              // and as one number, rows * W + columns
#pragma unroll
        for (int i = 0; i < kOwned; ++i) {
            udst[i] = kThin ? (uint32_t)xt * 16u + (uint32_t)i * (kXformThreads * 16u) : 0u;
            ujp[i] = 0;
            upix[i] = 0;
            if (kLinear) ulin[i] = 0;
            if (i < nu) {
                const int u = xt + i * kXformThreads;
                const int cg = kThin ? 0 : conv_fdiv(u, g.planes * g.SLOTS, g.dv_pss), idx = u - cg * per_stage_slots;
                // operand rows are 16 bytes apart: the low four bits carry the unit's chunk group
                if (!kThin) udst[i] = ((uint32_t)(cg * cpu) * (uint32_t)g.chunk_pitch + (uint32_t)idx * 16u) | (uint32_t)cg;
                const int pl = conv_fdiv(idx, g.SLOTS, g.dv_SLOTS), j = idx - pl * g.SLOTS;
                // the slot's distance from the tile's first slot, as whole slot rows and columns
                // (both below 2^12: a stage holds at most 2560 slots)
                const int dh = conv_fdiv(j, g.Ws, g.dv_Ws), dw = j - dh * g.Ws;
                ujp[i] = kRows ? (uint32_t)dh | ((uint32_t)dw << 16) : (uint32_t)dw | ((uint32_t)dh << 12);
                // fixed-index reads of the parity tables (a dynamic index into kernel parameters costs an indexed
                // constant load per use)
                const int pa = pl == 0 ? g.pa[0] : pl == 1 ? g.pa[1] : pl == 2 ? g.pa[2] : g.pa[3];
                const int pb = pl == 0 ? g.pb[0] : pl == 1 ? g.pb[1] : pl == 2 ? g.pb[2] : g.pb[3];
                upix[i] = ((uint32_t)(dh * g.sh + pa - g.pt) << 16) | ((uint32_t)(dw * g.sw + pb - g.pl) & 0xFFFFu);
                if (kLinear) ulin[i] = (dh * g.sh + pa - g.pt) * g.W + dw * g.sw + pb - g.pl;
            }
        }
        for (long long t = first_tile; t < g.total_tiles; t += tile_step) {
            int uoff[kOwned];                      // raw float offset of the unit's first channel, -1 = padding
            const int rot = kSplit ? cb_lo : cb_rotation(t, ncb);
            {
                // per-thread offsets of the tile, from its segment table (ready before the data)
                const uint32_t sp = tile_it & 1u;
                mbar_wait(&bars->seg_full[sp], (tile_it >> 1) & 1u, err, 21);
                PROF_MARK(4);
                ++tile_it;
                const TcConvSegs *segs = reinterpret_cast<const TcConvSegs *>(seg_st + sp * kSegBytes);
                const int n0 = segs->n_first, hq0 = segs->hq0, wq0 = segs->wq0;
                // Straight-line code, no branches on a lane's own data: the units' chains of dependent integer
                // operations then overlap instead of running one after the other (this loop, not the data movement,
                // was the larger part of the thin first layer's time).  Slot -> (image, slot row, slot column) without
                // dividing the slot number: the tile's first slot was decomposed once (by the producer, in the
                // segment table), and this unit lies a fixed number of slot rows and columns further on.
                if (kLinear && g.raw_mode == 2 && segs->one_image) {
                    // Nearly every tile of a large image: rows lie as in X, so a pixel's place in X's plane less the
                    // segment's is its offset, and its row exists where that place does (its column exists too).  A third
                    // of the instructions of the general form below, which were nearly half of a thin layer's re-lay: 7x7/2 first
                    // layer at batch 64 67.0 -> 63.8 us, 10 -> 16 channels 3x3 144x144 at batch 56 113.5 -> 99.2.
                    // (saturated: a unit's columns are below 2^12, a slot row of far padding at its end has 2^16 and more)
                    const uint32_t wrap = (uint32_t)min(g.Ws - wq0, 0xFFFF) << 16;
                    const int w0 = wq0 * g.sw, w1 = w0 - g.Ws * g.sw, HW = g.H * g.W;
                    const int p0 = hq0 * g.sh * g.W + w0, p1 = p0 + g.sh * g.W - g.Ws * g.sw, rel = segs->base[0] - segs->f0[0];
#pragma unroll
                    for (int i = 0; i < kOwned; ++i) {
                        const bool carry = ujp[i] >= wrap;
                        const int at = ulin[kLinear ? i : 0] + (carry ? p1 : p0), w = (int)(short)upix[i] + (carry ? w1 : w0);
                        uoff[i] = (unsigned)w < (unsigned)g.W && (unsigned)at < (unsigned)HW ? at + rel : -1;
                    }
                } else {
                    const int nseg = segs->nseg, hbase = hq0 * g.sh, wbase = wq0 * g.sw, Wssw = g.Ws * g.sw, Hssh = g.Hs * g.sh;
                    // the table's first two entries in registers: a tile of a large image touches no more than two
                    const int f0a = segs->f0[0], f0b = segs->f0[1], ba = segs->base[0], bb = segs->base[1];
                    const int images = min(nseg, g.N - n0);
#pragma unroll
                    for (int i = 0; i < kOwned; ++i) {
                        const int ch = kThin ? 0 : (int)(udst[i] & 15u) * cpu;
                        const int carry = wq0 + (int)(kRows ? ujp[i] >> 16 : ujp[i] & 0xFFFu) >= g.Ws ? 1 : 0;
                        const int hq = hq0 + (int)(kRows ? ujp[i] & 0xFFFFu : ujp[i] >> 12) + carry;
                        int k = hq >= g.Hs ? 1 : 0, f0 = k ? f0b : f0a, base = k ? bb : ba;        // images crossed
                        if (nseg > 2) {                                                            // (small images: several)
                            k = conv_fdiv(hq, g.Hs, g.dv_Hs);
                            const int sg = k < nseg ? k : 0;                                       // an entry that exists, whatever k is
                            f0 = segs->f0[sg];
                            base = segs->base[sg];
                        }
                        const int h = hbase + ((int)upix[i] >> 16) + carry * g.sh - k * Hssh;
                        const int w = wbase + (int)(short)upix[i] - carry * Wssw;
                        const bool ok = i < nu && k < images && (unsigned)h < (unsigned)g.H && (unsigned)w < (unsigned)g.W;
                        const int f = h * g.W + w - f0;
                        int o = base + f;                                                          // slabs, rows
                        if (kRows ? g.raw_mode == 0 : g.raw_mode != 1) {
                            if (g.boxp_shift >= 0) {
                                o = base + (f >> g.boxp_shift) * box_floats + (f & (g.BOXP - 1));
                            } else {
                                const int bx = conv_fdiv(ok ? f : 0, g.BOXP, g.dv_BOXP);
                                o = base + bx * box_floats + (f - bx * g.BOXP);
                            }
                        }
                        uoff[i] = ok ? o + ch * 4 * cp : -1;
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars->seg_empty[sp]);
                PROF_MARK(5);
            }
            for (int cb = 0; cb < ncb; ++cb) {
                mbar_wait(&bars->raw_full[rs], rphase, err, 16);
                PROF_MARK(0);
                if (xt == 0) LOG(5, cb);
                mbar_wait(&bars->a_empty[as], aphase ^ 1, err, 17);
                PROF_MARK(1);
                if (xt == 0) LOG(6, cb);
                const float *raw = reinterpret_cast<const float *>(raw_st + (size_t)rs * g.raw_stage_bytes);
                uint8_t *adst = a_st + (size_t)as * g.a_stage_bytes;
                const int cbx = kSplit || cb + rot < ncb ? cb + rot : cb + rot - ncb;
                const int c_left = g.Cg - cbx * KB;    // channels of this block that exist
                if (kThin) {
                    constexpr int kBatch = (kOwned + 1) / 2;
                    // In two batches of units: all reads of a batch first (independent, so their latencies
                    // overlap), then round and store; channels past the end of the group read as zero.
#pragma unroll
                    for (int h0 = 0; h0 < kOwned; h0 += kBatch) {
                        float v[kBatch][4];
#pragma unroll
                        for (int k = 0; k < kBatch; ++k) {
                            const int i = h0 + k;
                            if (i >= kOwned) break;
                            v[k][0] = v[k][1] = v[k][2] = v[k][3] = 0.f;
                            if (i < nu && uoff[i] >= 0) {
                                const float *r = raw + uoff[i];
                                if (c_left > 0) v[k][0] = r[0];
                                if (c_left > 1) v[k][1] = r[cp];
                                if (c_left > 2) v[k][2] = r[2 * cp];
                                if (c_left > 3) v[k][3] = r[3 * cp];
                            }
                        }
#pragma unroll
                        for (int k = 0; k < kBatch; ++k) {
                            const int i = h0 + k;
                            if (i >= kOwned) break;
                            if (i < nu)
                                *reinterpret_cast<float4 *>(adst + (udst[i] & ~15u)) =
                                    make_float4(round_tf32(v[k][0]), round_tf32(v[k][1]), round_tf32(v[k][2]),
                                                round_tf32(v[k][3]));
                        }
                    }
                } else {
                    // Two chunks at a time: their reads first (independent, so their latencies overlap), then round and
                    // store.  Padding units read word 0 and mask it.
#pragma unroll
                    for (int i = 0; i < kOwned; ++i) {
                        if (i < nu) {
                            const bool ok = uoff[i] >= 0;
                            const float *r = raw + (ok ? uoff[i] : 0);
                            uint8_t *d = adst + (udst[i] & ~15u);
                            int left = ok ? c_left - (int)(udst[i] & 15u) * cpu * 4 : 0;     // channels that exist from here on
                            for (int c = 0; c < cpu; c += 2) {
                                float v[8];
#pragma unroll
                                for (int e = 0; e < 8; ++e) v[e] = left > e ? r[e * cp] : 0.f;
                                *reinterpret_cast<float4 *>(d) = make_float4(round_tf32(v[0]), round_tf32(v[1]), round_tf32(v[2]), round_tf32(v[3]));
                                *reinterpret_cast<float4 *>(d + g.chunk_pitch) = make_float4(round_tf32(v[4]), round_tf32(v[5]), round_tf32(v[6]), round_tf32(v[7]));
                                r += 8 * cp;
                                d += 2 * g.chunk_pitch;
                                left -= 8;
                            }
                        }
                    }
                }
                PROF_MARK(2);
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    if (kCtas == 2 && rank != 0) {
                        if (g.relay) mbar_arrive(&bars->a_done[as]);                // the relay warp passes it on
                        else mbar_arrive_remote_release(a_full_addr + (uint32_t)as * 8u);
                    } else {
                        mbar_arrive(&bars->a_full[as]);                             // the issuing CTA's own barrier
                    }
                    mbar_arrive(&bars->raw_empty[rs]);
                }
                PROF_MARK(3);
                if (xt == 0) LOG(7, cb);
                if (++rs == nr) { rs = 0; rphase ^= 1; }
                if (++as == g.na_stages) { as = 0; aphase ^= 1; }
            }

        }
        if (xt == 0) PROF_FLUSH(5);
    } else {
        // ------------------------------------------------------------ epilogue warps
        const int ew = warp - kFirstEpiWarp;       // 0..7
        float *bias_w = reinterpret_cast<float *>(bias_st) + ew * 32;
        const int quarter = warp & 3;              // TMEM lane quarter this warp may read
        const bool two = g.MT == 2;
        const uint32_t acc_empty_addr = kCtas == 2 ? map_to_cta(smem_u32(&bars->acc_empty[0]), 0) : 0u;
        uint32_t it = 0;
        for (long long t = first_tile; t < g.total_tiles; t += tile_step, ++it) {
            const int ct_all = (int)(t % cgt);
            const int grp = ct_all / g.ctiles, ct = ct_all % g.ctiles;
            const long long G0 = ((t / cgt) * kCtas + rank) * tile_rows;
            const uint32_t ab = acc_dbl ? (it & 1u) : 0u, use = acc_dbl ? (it >> 1) : it;
            const int nch = (g.BN + 31) / 32;
            // eight warps: two per TMEM lane quarter, each taking half of the tile
            const int hf = ew >> 2, mt = two ? hf : 0;
            const int ch_lo = two ? 0 : hf ? (nch + 1) / 2 : 0, ch_hi = two || hf ? nch : (nch + 1) / 2;
            const uint32_t PQ4 = g.y_chan4;
            bool valid = false;
            uint32_t off = 0;                          // bytes from Y (and R): the launch keeps them below 2^32
            if (it == 0) pdl_wait();
            if (!kSplit) {
                // What does not depend on the accumulators is fetched while they are being summed: the outputs' places, the first
                // biases and, below, the first addends (each a trip to L2, next to no L1 being left).
                const uint32_t G = (uint32_t)G0 + (uint32_t)(mt * 128 + quarter * 32 + lane);
                valid = G < (uint32_t)g.total_slots;
                if (valid) {
                    const int n = conv_fdiv((int)G, g.L, g.dv_L), u = (int)G - n * g.L;
                    const int p = conv_fdiv(u, g.Ws, g.dv_Ws), q = u - p * g.Ws;
                    valid = p < g.P && q < g.Q;
                    off = (uint32_t)n * g.y_image4 + (uint32_t)(grp * g.Mg + ct * g.BN + ch_lo * 32) * PQ4 + (uint32_t)(p * g.Q + q) * 4u;
                }
            }
            const char *rb = reinterpret_cast<const char *>(R);
            if (kAddend == kAddendFar) {
                // The next tile's addends (the first time this one's too) are asked into L2: eight in flight per lane below, all
                // that its registers hold, are too few for a trip to memory each.  3 -> 64
                // channels 7x7/2 224x224 at batch 32 78.7 -> 65.8 us, 10 -> 80 3x3 130x198 at batch 23 142 -> 122.
                for (long long u = it == 0 ? t : t + tile_step; u <= t + tile_step && u < g.total_tiles; u += tile_step) {
                    const int cta = (int)(u % cgt), gr = cta / g.ctiles, m0 = cta % g.ctiles * g.BN;
                    const uint32_t Gw = (uint32_t)(((u / cgt) * kCtas + rank) * tile_rows) + (uint32_t)(mt * 128 + quarter * 32);
#pragma unroll
                    for (int e = 0; e < 2; ++e) {               // the two lines that the warp's 32 pixels lie in
                        const uint32_t G = Gw + 31u * e;
                        const int n = conv_fdiv((int)G, g.L, g.dv_L), w = (int)G - n * g.L, p = conv_fdiv(w, g.Ws, g.dv_Ws);
                        if (n >= g.N || p >= g.P) continue;
                        const char *at = rb + (uint32_t)(p * g.Q + min(w - p * g.Ws, g.Q - 1)) * 4u;
                        for (int c = m0 + ch_lo * 32 + lane; c < min(g.Mg, m0 + min(g.BN, ch_hi * 32)); c += 32)
                            prefetch_l2(at + ((uint32_t)n * g.y_image4 + (uint32_t)(gr * g.Mg + c) * PQ4));
                    }
                }
            }
            const int tile_left = min(g.Mg - ct * g.BN, g.BN);         // channels of the tile
            float b_next = 0.f, r[2][8];
            auto fetch_bias = [&](int chunk) {
                const int c = chunk * 32 + lane;
                b_next = bias && chunk < ch_hi && c < tile_left ? __ldg(bias + grp * g.Mg + ct * g.BN + c) : 0.f;
            };
            // addends (at Y's own positions) of the eight channels `ahead` of those that `off` has come to, `left` of which exist
            auto fetch_add = [&](float (&to)[8], int ahead, int left) {
                const int lane_left = valid ? left : 0;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    // (the form that does not ask ahead gains from having them issued where they stand, 7 to 20 % on layers with a
                    // large addend; the other, 3 %, from having them where the compiler puts them)
                    if (kAddend == kAddendNear) to[j] = ldg_where(rb + (off + (uint32_t)(ahead + j) * PQ4), ahead + j, lane_left);
                    else to[j] = ahead + j < lane_left ? __ldg(reinterpret_cast<const float *>(rb + (off + (uint32_t)(ahead + j) * PQ4))) : 0.f;
                }
            };
            if (!kSplit) {
                fetch_bias(ch_lo);
                if (kAdd) fetch_add(r[0], 0, min(tile_left, ch_hi * 32) - ch_lo * 32);
            }
            mbar_wait(&bars->acc_full[ab], use & 1u, err, 18);
            tc_fence_after_sync();
            if (ew == 0 && lane == 0) LOG(8, 2);
            if (kSplit) {
                // every group of four channels goes to the CTA that finishes it, as [source CTA][group][pixel][4]:
                // the lanes of a store write consecutive 16-byte pieces
                cluster_wait();                 // (the peers set up long ago)
                const uint32_t to = smem_u32(recv_st) + (cluster_ctarank() * (uint32_t)g.cols_per / 4u * 128u + (uint32_t)(quarter * 32 + lane)) * 16u;
                const uint32_t bar = smem_u32(&bars->recv_full);
                for (int chunk = ew >> 2; chunk < nch; chunk += kEpiWarps / 4) {
                    uint32_t v[32];
                    tmem_ld_32x32(tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(chunk * 32), v);
                    tmem_ld_wait();
                    int dst = chunk * 32 / g.cols_per, in = chunk * 32 - dst * g.cols_per;       // owner, and the place in its slice
#pragma unroll
                    for (int j = 0; j < 32; j += 4) {
                        if (chunk * 32 + j < tile_ch4)
                            st_async_v4(map_to_cta(to + (uint32_t)in * 512u, (uint32_t)dst), v[j], v[j + 1], v[j + 2], v[j + 3], map_to_cta(bar, (uint32_t)dst));
                        in += 4;
                        if (in == g.cols_per) { in = 0; ++dst; }
                    }
                }
            }
            if (!kSplit) {
                const uint32_t acc_col = ab * 256u + (uint32_t)mt * mt_cols;
                char *yb = reinterpret_cast<char *>(Y);
                // fmaxf returns its other argument where one is NaN, and NaN where both are: without Relu nothing is changed.
                // (The constant is hidden from the compiler, which would otherwise choose between x and fmaxf(x, 0) for every
                // output; that took the form with an addend from 145 to 185 us on a 3 -> 64, 7x7/2, 224x224 layer, batch 32.)
                float lowest;
                asm("mov.b32 %0, %1;" : "=f"(lowest) : "r"(g.relu ? 0 : 0x7FC00000));
                for (int chunk = ch_lo; chunk < ch_hi; ++chunk) {
                    uint32_t v[32];
                    tmem_ld_32x32(tmem_base + ((uint32_t)(quarter * 32) << 16) + acc_col + (uint32_t)(chunk * 32), v);
                    const int mg0 = ct * g.BN + chunk * 32;                // first channel (within the group) of the chunk
                    const int cnt = min(g.Mg, (ct + 1) * g.BN) - mg0;      // channels of the chunk that exist (above 32: all)
                    // the chunk's biases through shared memory: eight 16-byte broadcasts instead of 32 shuffles
                    __syncwarp();
                    bias_w[lane] = b_next;
                    __syncwarp();
                    fetch_bias(chunk + 1);
                    tmem_ld_wait();
#pragma unroll
                    for (int j0 = 0; j0 < 32; j0 += 8) {
                        if (kAdd) fetch_add(r[(j0 >> 3) + 1 & 1], 8, min(tile_left, ch_hi * 32) - chunk * 32 - j0);
#pragma unroll
                        for (int j = 0; j < 8; j += 4) {
                            const float4 b4 = *reinterpret_cast<const float4 *>(bias_w + j0 + j);
                            const float b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                float x = __uint_as_float(v[j0 + j + e]) + b[e];
                                if (kAdd) x += r[(j0 >> 3) & 1][j + e];
                                x = fmaxf(x, lowest);
                                if (kAddend == kRoundedY) x = round_tf32(x);
                                if (valid && j0 + j + e < cnt) *reinterpret_cast<float *>(yb + off) = x;
                                off += PQ4;
                            }
                        }
                    }
                }
            }
            tc_fence_before_sync();
            __syncwarp();
            if (ew == 0 && lane == 0) LOG(8, 3);
            if (lane == 0) {
                if (kCtas == 2) mbar_arrive_remote(acc_empty_addr + ab * 8u);
                else mbar_arrive(&bars->acc_empty[ab]);
            }
        }
    }

    if (kSplit) {
        __syncwarp();
        if (warp < kFirstEpiWarp) cluster_wait();
        cluster_arrive();                       // sent
        if (warp >= kFirstXformWarp) {
            // sum this CTA's channels over the sources, in rank order: lanes along pixels, four channels each
            const int tid = threadIdx.x - kFirstXformWarp * 32, row = tid & 127;
            constexpr int kGroups = (kXformWarps + kEpiWarps) / 4;
            const int ct_all = (int)(first_tile % cgt), grp = ct_all / g.ctiles, ct = ct_all % g.ctiles;
            const uint32_t G = (uint32_t)((first_tile / cgt) * 128) + (uint32_t)row;
            const int n = conv_fdiv((int)G, g.L, g.dv_L), u = (int)G - n * g.L;
            const int p = conv_fdiv(u, g.Ws, g.dv_Ws), q = u - p * g.Ws;
            if (G < (uint32_t)g.total_slots && p < g.P && q < g.Q) {
                pdl_wait();                     // long since satisfied
                const long long PQ = g.y_chan4 / 4;
                for (int col = col_lo + (tid >> 7) * 4; col < col_hi; col += kGroups * 4) {
                    const int m = grp * g.Mg + ct * g.BN + col, cnt = tile_ch - col;          // channels that exist (above 4: all)
                    const long long o = (long long)n * (g.y_image4 / 4) + m * PQ + (long long)p * g.Q + q;
                    float b[4], r[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        b[e] = bias && e < cnt ? __ldg(bias + m + e) : 0.f;
                        r[e] = kAdd && e < cnt ? __ldg(R + o + e * PQ) : 0.f;
                    }
                    mbar_wait_cluster(&bars->recv_full, 0, err, 23);
                    const float4 *x = reinterpret_cast<const float4 *>(recv_st) + (col - col_lo) / 4 * 128 + row;
                    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int s = 0; s < 8; ++s)
                        if (s < g.split) {
                            const float4 v = x[s * (g.cols_per / 4) * 128];
                            a.x += v.x; a.y += v.y; a.z += v.z; a.w += v.w;
                        }
                    const float f[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        float y = f[e] + b[e];
                        if (kAdd) y += r[e];
                        if (g.relu) y = fmaxf(y, 0.f);
                        if (kAddend == kRoundedY) y = round_tf32(y);
                        if (e < cnt) Y[o + e * PQ] = y;
                    }
                }
            }
        }
        cluster_wait();                         // no CTA leaves before its peers have sent (they have, unless a wait gave up)
    }
    tc_fence_before_sync();
    __syncthreads();
    if (kCtas == 2) cluster_sync_all();         // no CTA leaves while its peer may still signal it
    if (threadIdx.x == 0) LOG(8, 4);
    if (warp == 2) {
        __syncwarp();
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, kSplit ? split_tmem_cols(g.BN) : 512);
    }
}

// ------------------------------------------------------------------ planning (host)
int pick_conv_bn(int Mg) {
    if (Mg <= 256) return (Mg + 15) / 16 * 16;
    int best = 256, best_pad = 1 << 30;
    for (int bn : {256, 192, 128}) {
        const int padded = (Mg + bn - 1) / bn * bn;
        if (padded < best_pad) { best_pad = padded; best = bn; }
    }
    return best;
}

bool fill_plan(const ConvGeom &c, int ctas, int MT, int BN, int KB, TcConvPlan &g) {
    if (ctas == 2 && BN % 16) return false;      // M = 256 instructions take N in multiples of 16
    g.ctas = ctas;
    g.split = 1;
    g.cb_per = 0;
    g.BNH = BN / ctas;
    g.N = c.N; g.C = c.C; g.H = c.H; g.W = c.W; g.M = c.M; g.Cg = c.Cg; g.Mg = c.Mg;
    g.kH = c.kH; g.kW = c.kW; g.P = c.P; g.Q = c.Q; g.pt = c.pt; g.pl = c.pl;
    g.sh = c.sh; g.sw = c.sw; g.dh = c.dh; g.dw = c.dw; g.group = c.group; g.relu = c.relu;
    g.taps = c.kH * c.kW;
    if (g.taps > kConvMaxTaps) return false;
    ConvAxis ah, aw;
    if (!conv_plan_axis(c.H, c.P, c.pt, c.sh, c.dh, c.kH, ah)) return false;
    if (!conv_plan_axis(c.W, c.Q, c.pl, c.sw, c.dw, c.kW, aw)) return false;
    if (ah.npar * aw.npar > kConvMaxPlanes) return false;
    g.Hs = ah.E; g.Ws = aw.E;
    const long long L = (long long)g.Hs * g.Ws;
    if (L > (1 << 24)) return false;
    g.L = (int)L;
    g.total_slots = (long long)c.N * L;
    if (g.total_slots + 4096 >= (1LL << 31)) return false;        // device code indexes slots in 32 bits
    if ((long long)c.M * c.P * c.Q >= (1LL << 30)) return false;  // and an image's outputs in 32 bits of bytes
    g.planes = 0;
    for (int i = 0; i < ah.npar; ++i)
        for (int j = 0; j < aw.npar; ++j) { g.pa[g.planes] = ah.par[i]; g.pb[g.planes] = aw.par[j]; ++g.planes; }
    g.a_min = ah.par[0]; g.a_max = ah.par[ah.npar - 1];
    const long long maxshift = (long long)ah.Amax * g.Ws + aw.Amax;
    g.MT = MT; g.BN = BN;
    g.ctiles = (c.Mg + BN - 1) / BN;
    const long long slots = (long long)MT * 128 + maxshift;
    if (c.Cg < 16) KB = 4;
    if (slots * g.planes * (KB / 4) > kMaxUnits) return false;
    g.SLOTS = (int)slots;
    // a slot's distance from the tile's first, in pixels, fits 16 signed bits
    if (slots * std::max(c.sh, c.sw) + std::max(c.pt, c.pl) > 32000) return false;
    if ((g.SLOTS + L - 2) / L + 1 > kConvMaxSeg) return false;
    g.plane_pitch = g.SLOTS * 16;
    g.chunk_pitch = g.planes * g.plane_pitch;
    if (g.chunk_pitch >= (1 << 18)) return false;

    // per-tap plane and slot shift, in 16-byte units inside an A stage
    int tap_plane[kConvMaxTaps], tap_off16[kConvMaxTaps];
    for (int r = 0; r < c.kH; ++r)
        for (int s = 0; s < c.kW; ++s) {
            const int a = (r * c.dh) % c.sh, b = (s * c.dw) % c.sw;
            int pl = 0;
            while (g.pa[pl] != a || g.pb[pl] != b) ++pl;
            const int shift = ((r * c.dh) / c.sh) * g.Ws + (s * c.dw) / c.sw;
            tap_plane[r * c.kW + s] = pl;
            tap_off16[r * c.kW + s] = (pl * g.plane_pitch + shift * 16) >> 4;
        }

    // K-steps of one channel block
    if (c.Cg >= 16) {
        // blocks of KB = 16, 32 or 64 channels: KB/8 steps per tap, step j reading chunks 2j and 2j+1
        const int spt = KB / 8;
        g.KB = KB;
        g.n_steps = spt * g.taps;
        if (g.n_steps > kConvMaxSteps) return false;
        const uint32_t lbo16 = (uint32_t)g.chunk_pitch >> 4;
        if ((uint32_t)(KB / 4) * lbo16 >= (1u << 14)) return false;     // every chunk start must fit the address field
        for (int tp = 0; tp < g.taps; ++tp)
            for (int j = 0; j < spt; ++j) {
                const int s = spt * tp + j;
                g.step_a[s] = ((uint32_t)tap_off16[tp] + (uint32_t)j * 2u * lbo16) | (lbo16 << 16);
                g.src_tap[s][0] = g.src_tap[s][1] = (short)tp;
                g.src_c0[s][0] = (short)(j * 8);
                g.src_c0[s][1] = (short)(j * 8 + 4);
            }
    } else {
        // tap pairs: within each plane, taps in order of their offset, two per step
        g.KB = 4;
        g.n_steps = 0;
        for (int pl = 0; pl < g.planes; ++pl) {
            int list[kConvMaxTaps], n = 0;
            for (int tp = 0; tp < g.taps; ++tp)
                if (tap_plane[tp] == pl) list[n++] = tp;
            std::sort(list, list + n, [&](int x, int y) { return tap_off16[x] < tap_off16[y]; });
            for (int i = 0; i < n; i += 2) {
                const int t0 = list[i], t1 = i + 1 < n ? list[i + 1] : -1;
                const uint32_t lbo16 = t1 >= 0 ? (uint32_t)(tap_off16[t1] - tap_off16[t0]) : 0u;
                if (lbo16 >= (1u << 14)) return false;
                const int s = g.n_steps++;
                g.step_a[s] = (uint32_t)tap_off16[t0] | (lbo16 << 16);
                g.src_tap[s][0] = (short)t0;
                g.src_tap[s][1] = (short)t1;
                g.src_c0[s][0] = g.src_c0[s][1] = 0;
            }
        }
    }
    for (int s = g.n_steps; s < kConvMaxSteps; ++s) {
        g.step_a[s] = 0;
        g.src_tap[s][0] = g.src_tap[s][1] = -1;
        g.src_c0[s][0] = g.src_c0[s][1] = 0;
    }
    g.nchunks = g.KB / 4;
    // Chunk groups: the split that gives the busiest transform thread the least work, pairs of chunks at least.
    g.chunk_groups = 1;
    g.chunks_per_unit = g.nchunks;
    if (g.KB > 4) {
        int best = 1 << 30;
        for (int groups = 1; groups * 2 <= g.nchunks; groups *= 2) {
            const long long owned = ((long long)g.planes * g.SLOTS * groups + kXformThreads - 1) / kXformThreads;
            const int work = (int)owned * (g.nchunks / groups) * 4 + (int)owned;        // chunks, and a little per unit
            if (owned <= kOwnedThick && work < best) {
                best = work;
                g.chunk_groups = groups;
                g.chunks_per_unit = g.nchunks / groups;
            }
        }
        if (best == 1 << 30) return false;
    }
    g.ncb = (c.Cg + g.KB - 1) / g.KB;
    const long long ptiles = (g.total_slots + MT * 128 - 1) / (MT * 128);      // per-CTA pixel tiles
    if (ptiles > 0x7fffffffLL) return false;
    g.pix_tiles = (int)((ptiles + ctas - 1) / ctas);
    g.total_tiles = (long long)g.pix_tiles * g.ctiles * c.group;
    // raw staging mode
    const long long HW = (long long)c.H * c.W;
    g.x_cm = c.x_cm;
    const long long y_pitch = channel_pitch(c.N, c.P, c.Q);
    if (c.y_cm && y_pitch * c.M >= (1LL << 30)) return false;         // (one launch: offsets in 32 bits of bytes)
    if (c.x_cm && (!c.y_cm && (long long)c.N * c.M * c.P * c.Q >= (1LL << 30))) return false;
    g.y_image4 = (uint32_t)((c.y_cm ? 1LL : (long long)c.M) * c.P * c.Q * 4);
    g.y_chan4 = (uint32_t)((c.y_cm ? y_pitch : (long long)c.P * c.Q) * 4);
    if (c.x_cm) {
        if (g.KB == 4 || channel_pitch(c.N, c.H, c.W) >= (1LL << 30)) return false;
        g.raw_mode = 0;
    } else if (HW % 4 == 0) {
        // Blocks of 4 channels of images that a tile touches two of at most: a copy per channel (a box per 256 pixels is more
        // copies there, and its places cost the transform a shift and a mask per unit).
        g.raw_mode = g.KB == 4 && (g.SLOTS + L - 2) / L + 1 <= 2 ? 2 : 0;
    } else if (c.Cg % 4 == 0 && c.C % 4 == 0 && HW * g.KB * 4 <= 32768) {
        g.raw_mode = 1;
    } else {
        return false;
    }
    g.a_stage_bytes = g.nchunks * g.chunk_pitch;
    g.a_stage_bytes = (g.a_stage_bytes + 127) / 128 * 128;
    g.b_step_bytes = g.BNH * 32;
    g.idesc = tc::make_idesc_tf32(128 * ctas, BN, 0, 0);
    g.packed_floats = (long long)c.group * g.ctiles * g.ncb * g.n_steps * BN * 8;     // both CTAs' parts
    if (g.packed_floats >= (1LL << 32)) return false;                                  // 32-bit indexing in the packing kernel
    // Raw stage size.  What a tile stages depends on where its first slot lies in an image; of the starts in one
    // slot row the last reaches furthest, and the first image has the most slots after it, so one start per slot
    // row covers all tiles.
    g.KBR = std::min(g.KB, c.Cg);
    // (channel-major: where a range of pixels begins within 16 bytes goes by its image, too)
    auto for_each_start = [&](auto &&f) {
        for (int n = 0; n < (c.x_cm ? std::min(c.N, 4) : 1); ++n)
            for (int r = 0; r < g.Hs; ++r) f(std::min<long long>(n * L + (long long)r * g.Ws + g.Ws - 1, g.total_slots - 1));
    };
    auto stage_floats = [&](int boxp, int &boxes) {
        g.BOXP = boxp;
        int worst = 0;
        boxes = 0;
        for_each_start([&](long long G0) {
            TcConvSegs segs;
            tc_conv_segments(g, G0, segs);
            worst = std::max(worst, segs.total_floats);
            int n = 0;
            for (int i = 0; i < segs.nseg; ++i) n += segs.nbox[i];
            boxes = std::max(boxes, n);
        });
        return worst;
    };
    int worst, boxes;
    if (g.raw_mode == 1) {
        worst = stage_floats(256, boxes);
    } else if (g.raw_mode == 2) {
        g.BOXP = std::max(4, stage_floats(4, boxes));
        worst = g.BOXP * g.KBR;
    } else if (g.KB == 4) {
        // Blocks of 4 channels (the thin first layer of a network) stage little per pixel: 256-pixel boxes, and
        // a power of two spares the transform a division per unit.
        worst = stage_floats(256, boxes);
    } else {
        // Boxes of at most 256 pixels, splitting the widest flat range of an image that a tile needs evenly; every box
        // starts on a 128-byte boundary of shared memory (TMA destination alignment): KB * BOXP * 4 bytes is a
        // multiple of 128.  (Smaller boxes stage less beyond what a tile needs, but cost more than that gains:
        // 64 -> 64 channels at 56x56 44.3 -> 46 us.)
        int widest = 4;
        if (c.x_cm) {
            g.BOXP = 4;                            // (boxes of four: the range itself)
            for_each_start([&](long long G0) {
                TcConvSegs segs;
                tc_conv_segments(g, G0, segs);
                if (segs.nseg > 0) widest = std::max(widest, segs.nbox[0] * 4);
            });
        }
        else for_each_start([&](long long G0) {
            const long long Gend = std::min<long long>(G0 + g.SLOTS, g.total_slots);
            for (long long n = 0; n * L < Gend; ++n) {
                const long long lo = std::max<long long>(G0, n * L), hi = std::min<long long>(Gend, (n + 1) * L);
                if (lo >= hi) continue;
                const int h_min = std::max(0, (int)((lo - n * L) / g.Ws) * c.sh + g.a_min - c.pt);
                const int h_max = std::min(c.H - 1, (int)((hi - 1 - n * L) / g.Ws) * c.sh + g.a_max - c.pt);
                if (h_min <= h_max) widest = std::max(widest, (h_max + 1) * c.W - ((h_min * c.W) & ~3));
            }
        });
        const int align = std::max(4, 32 / g.KB), nbox = (widest + 255) / 256;
        const int boxp = std::min(256, ((widest + nbox - 1) / nbox + align - 1) / align * align);
        worst = stage_floats(boxp, boxes);
    }
    g.raw_stage_bytes = std::max(128, (worst * 4 + 127) / 128 * 128);
    // Raw stages: a third one (the raw tiles come from L2/HBM with a microsecond of latency) when that
    // still leaves 64 KB for the weight ring.
    g.na_stages = 2;
    g.nr_stages = 2;
    g.relay = 0;
    {
        // "ONNXB_CONV_STAGES=a,r" pins the operand / raw stage counts for A/B measurements
        int fa = 0, fr = 0;
        const char *e = getenv("ONNXB_CONV_STAGES");
        if (e && sscanf(e, "%d,%d", &fa, &fr) == 2 && fa >= 2 && fa <= kMaxAStages && fr >= 2 && fr < kMaxRawStages) {
            g.na_stages = fa;
            g.nr_stages = fr;
        } else if (MT == 2 && g.KB >= 16 &&
                   kSmemLimit - (1024 + 3LL * g.a_stage_bytes + kMaxRawStages * kSegBytes + kBiasBytes + kBarBytes) -
                           2LL * g.raw_stage_bytes >= 65536) {
            // Two accumulators per CTA: a third operand stage instead of a third raw stage, and in a CTA pair
            // the odd CTA's "stage written" message through its relay warp.  The message then arrives later,
            // which three stages absorb, and the transform warps no longer wait for their cluster-scope fence.
            // Batch 64, the same tile; two operand and three raw stages without / with the relay, three and two
            // without / with it: 64 -> 64 channels at 56x56 46.6 / 45.5, 47.2 / 38.2 us; 128 -> 128 at 28x28
            // 34.1 / 37.0, 33.4 / 31.8; 256 -> 256 at 14x14 32.6 / 35.1, 31.7 / 31.8.
            g.na_stages = 3;
            g.relay = ctas == 2 ? 1 : 0;
        } else {
            const long long bf = 1024 + 2LL * g.a_stage_bytes + kMaxRawStages * kSegBytes + kBiasBytes + kBarBytes;
            for (int nr = 3; nr <= kMaxRawStages - 1; ++nr)
                if (kSmemLimit - bf - (long long)nr * g.raw_stage_bytes >= 65536) g.nr_stages = nr;
        }
    }
    const long long base_fixed = 1024 + (long long)g.na_stages * g.a_stage_bytes + kMaxRawStages * kSegBytes + kBiasBytes + kBarBytes;
    const long long fixed = base_fixed + (long long)g.nr_stages * g.raw_stage_bytes;
    const long long room = kSmemLimit - fixed;
    // K-steps per weight stage: as many as leave three stages in flight, the block's steps spread evenly.
    g.spb = std::min(g.n_steps, kMaxSpb);
    while (g.spb > 1 && ((long long)g.spb * g.b_step_bytes > 36864 || room < 3LL * g.spb * g.b_step_bytes)) --g.spb;
    g.b_steps = (g.n_steps + g.spb - 1) / g.spb;
    g.spb = (g.n_steps + g.b_steps - 1) / g.b_steps;
    g.b_stage_bytes = g.spb * g.b_step_bytes;
    // One channel block and one channel tile: every tile uses the same weights.  Kept, where they fit.
    g.b_resident = 0;
    if (g.ncb == 1 && g.ctiles * c.group == 1) {
        const int spb = std::min(g.n_steps, kMaxSpb), steps = (g.n_steps + spb - 1) / spb;
        const long long even = (g.n_steps + steps - 1) / steps;
        if (steps <= kMaxBStages && steps * even * g.b_step_bytes <= room) {
            g.b_resident = 1;
            g.spb = (int)even;
            g.b_steps = steps;
            g.b_stage_bytes = g.spb * g.b_step_bytes;
        }
    }
    if (room < 2LL * g.b_stage_bytes && !g.b_resident) return false;
    g.nb_stages = (int)std::min<long long>(kMaxBStages, room / g.b_stage_bytes);
    g.dv_L = conv_divisor(g.L);
    g.dv_Ws = conv_divisor(g.Ws);
    g.dv_Hs = conv_divisor(g.Hs);
    g.boxp_shift = -1;
    for (int b = 0; b < 16; ++b)
        if ((1 << b) == g.BOXP) g.boxp_shift = b;
    g.dv_BOXP = conv_divisor(g.BOXP);
    g.dv_SLOTS = conv_divisor(g.SLOTS);
    g.dv_pss = conv_divisor(g.planes * g.SLOTS);
    return true;
}

// Shares each tile of a plan among a cluster of S: no more stages than a share has blocks, beside room for the partial sums.
bool split_plan(int S, TcConvPlan &p) {
    p.split = S;
    p.cb_per = (p.ncb + S - 1) / S;
    if (p.cb_per * (S - 1) >= p.ncb) return false;                       // every CTA needs a block
    p.cols_per = ((p.BN + S - 1) / S + 3) / 4 * 4;
    p.na_stages = std::min(p.na_stages, p.cb_per);
    p.nr_stages = std::min(p.nr_stages, p.cb_per);
    const long long room = kSmemLimit - 1024 - (long long)p.na_stages * p.a_stage_bytes - (long long)p.nr_stages * p.raw_stage_bytes -
                           kMaxRawStages * kSegBytes - kBiasBytes - kBarBytes - split_recv_bytes(S, p.cols_per);
    p.nb_stages = (int)std::min<long long>({(long long)kMaxBStages, (long long)p.cb_per * p.b_steps, room / p.b_stage_bytes});
    return p.nb_stages >= std::min(2, p.cb_per * p.b_steps);
}

// Estimated SM cycles of a plan, fitted to 2336 measured (shape, tile) pairs: 70 shapes from ResNet-50's 3x3 layers at
// batch 1 to 64 to random ones of 16-384 channels, 3x3 and 5x5, stride 1 and 2, one image and many; the pick is within
// 1 % of the best tile on average.  Per channel block the slowest of: the tensor pipe (0.57 BN cycles per 128 x BN x 8
// share of an instruction, or its operands out of shared memory at 126 bytes/cycle) with 390 cycles per weight stage;
// shared memory as a whole (operand reads, stages written, re-lay) at 115 bytes/cycle; the weight stream out of L2 (32
// bytes/cycle and SM, 3600 over all SMs) or, where the ring is short, its latency of 2100 cycles; the re-lay, 42 cycles
// per chunk of the busiest thread; and the producer's copies, some 330 per image a tile touches.
double tile_cost(const TcConvPlan &p) {
    // tiles in flight (a cluster of 8 does not fit every GPC: 14 of them are resident at once, and 33 of 4)
    const int units = p.split == 8 ? 14 : p.split == 4 ? 33 : 148 / p.ctas / p.split;
    const long long waves = (p.total_tiles + units - 1) / units;
    const double active = (double)std::min<long long>(p.total_tiles, units) * p.ctas * p.split;
    const bool pair = p.ctas == 2;
    const double n_inst = (double)p.n_steps * p.MT, op_bytes = 4096.0 + p.BNH * 32.0;
    const double t_mma = n_inst * std::max(p.BN * 0.568, op_bytes / 126.0) + (p.n_steps + p.spb - 1) / p.spb * 391.0;
    const double owned = (p.planes * p.SLOTS * p.chunk_groups + kXformThreads - 1) / kXformThreads;
    if (p.KB == 4) {
        // Thin layers, fitted to 108 pairs of their own (14 shapes, pick within 1 %): few steps per tile, so the tile's own
        // costs count, the epilogue (17 cycles per channel and accumulator, behind the next tile where the accumulators
        // alternate) and what a pair's CTAs wait for one another (7x7/2 first layer at batch 32: a pair 43.8 us, single CTAs 41.6).
        const double body = p.ncb * (std::max(t_mma, 1000.0) + 800.0 + (pair ? 390.0 : 0.0)) + 1380.0 + 80.0 * owned;
        const double epi = 17.0 * p.MT * p.BN;
        const bool overlapped = p.MT == 1 || p.BN <= 128;
        return waves * (overlapped ? std::max(body, epi) : body + epi) + (overlapped ? epi : 0.0) + 9580.0 + (pair ? 910.0 : 0.0);
    }
    const double w_bytes = p.b_resident ? 0.0 : (double)p.n_steps * p.b_step_bytes;
    const double slots16 = (double)p.planes * p.SLOTS * 16.0 * p.nchunks;
    const double t_smem = (n_inst * op_bytes + w_bytes + 3.0 * slots16) / 115.0;
    const double ring = (double)p.nb_stages * p.b_stage_bytes;
    const double t_w = std::max(w_bytes / std::min(31.5, 3620.0 / active),
                                p.split > 1 && ring >= w_bytes * p.cb_per ? 0.0 : w_bytes * 2090.0 / ring);
    const double t_x = 1075.0 + 42.0 * owned * p.chunks_per_unit + (pair ? 615.0 : 0.0);
    const double t_p = 342.0 + 327.0 * (p.x_cm ? 1 : (p.SLOTS - 1) / p.L + 2);
    const double per_cb = std::max({t_mma, t_smem, t_w, t_x, t_p});
    if (p.split > 1) return (double)waves * (p.cb_per * (per_cb + 896.0) + 28.0 * p.BN + 5190.0) + 7090.0;
    return (double)waves * (p.ncb * (per_cb + (p.na_stages == 3 ? 0.0 : 449.0)) + 1650.0) + 9530.0;
}

}  // namespace

bool tc_conv_plan(const ConvGeom &c, TcConvPlan &plan, bool forced) {
    const long long taps = (long long)c.kH * c.kW;
    if (c.Cg < 16) {
        // tap-pair mode needs at least two taps, and is kept for problems big enough to matter:
        // tiny thin contractions (an MNIST-size first layer) stay on the exact fp32 SIMT kernel
        const double flops = 2.0 * c.N * c.M * c.P * c.Q * c.Cg * (double)taps;
        if (taps < 2 || c.Cg * taps < 32 || (flops < 5e7 && !forced)) return false;
    }
    const int bn0 = pick_conv_bn(c.Mg);
    // candidate tiles (CTAs per tile, accumulators per CTA, channels per tile)
    int cand[96][4];
    int ncand = 0;
    auto add = [&](int ctas, int mt, int bn, int kb) {
        for (int i = 0; i < ncand; ++i)
            if (cand[i][0] == ctas && cand[i][1] == mt && cand[i][2] == bn && cand[i][3] == kb) return;
        cand[ncand][0] = ctas; cand[ncand][1] = mt; cand[ncand][2] = bn; cand[ncand][3] = kb; ++ncand;
    };
    int fc = 0, fm = 0, fb = 0, fk = 16;
    if (const char *e = getenv("ONNXB_CONV_TILE")) {      // "ctas,MT,BN[,KB]": pin the tile for A/B measurements
        if (sscanf(e, "%d,%d,%d,%d", &fc, &fm, &fb, &fk) >= 3 && (fc == 1 || fc == 2) && (fm == 1 || fm == 2) &&
            fb >= 16 && fb <= 256 && fb % 16 == 0 && (fk == 16 || fk == 32 || fk == 64))
            add(fc, fm, fb, fk);
    }
    if (ncand == 0) {
        for (int kb = 16; kb <= 64 && (kb == 16 || kb <= c.Cg); kb *= 2)
            for (int ctas = 2; ctas >= 1; --ctas) {
                for (int bn : {bn0, 128, 96, 64})
                    if (bn <= bn0) {
                        add(ctas, 2, bn, kb);
                        add(ctas, 1, bn, kb);
                    }
            }
    }
    bool have = false;
    double best_cost = 0;
    for (int i = 0; i < ncand; ++i) {
        TcConvPlan p;
        if (!fill_plan(c, cand[i][0], cand[i][1], cand[i][2], cand[i][3], p)) continue;
        const double cost = tile_cost(p);
        if (!have || cost < best_cost * 0.999) {
            have = true;
            best_cost = cost;
            plan = p;
        }
    }
    // Few tiles: let a cluster share each one's channel blocks (not for thin layers, which have one block).
    {
        int pb = 0, pk = 0, ps = 0;         // ONNXB_CONV_SPLIT = "BN,KB,S" pins the shape, "0" rules the split out
        const char *e = getenv("ONNXB_CONV_SPLIT");
        const bool pinned = e && sscanf(e, "%d,%d,%d", &pb, &pk, &ps) == 3;
        const bool ruled_out = (e && !pinned) || getenv("ONNXB_CONV_TILE") || getenv("ONNXB_CONV_STAGES");
        if (c.Cg >= 32 && !ruled_out && (pinned || (have && plan.total_tiles * plan.ctas <= 148))) {
            if (pinned) have = false;
            for (int kb = 16; kb <= 32; kb *= 2)
                for (int bn = 16; bn <= 256; bn *= 2) {
                    const int b = std::min(bn, (c.Mg + 15) / 16 * 16);
                    if (pinned && (bn != pb || kb != pk)) continue;
                    if (!pinned && bn > 16 && b <= bn / 2) break;
                    TcConvPlan whole;
                    if (!fill_plan(c, 1, 1, b, kb, whole)) continue;
                    for (int S = 2; S <= 8; S *= 2) {
                        if (pinned && S != ps) continue;
                        TcConvPlan p = whole;
                        if (!split_plan(S, p)) continue;
                        if (!pinned && p.total_tiles * S > (S == 8 ? 112 : S == 4 ? 132 : 148)) continue;
                        const double cost = tile_cost(p);
                        if (!have || cost < best_cost * 0.999) {
                            have = true;
                            best_cost = cost;
                            plan = p;
                        }
                    }
                }
        }
    }
    if (have) {
        // Thin layers in tap-pair mode, where they run as pairs, are paced by the transform warps: take their fence off
        // them too (4 -> 160 channels, 7x7/2, 112x112, batch 64, one accumulator: 46.0 -> 43.0 us; 3 -> 64 at 224x224,
        // as a pair, 82.6 -> 75.7).  ONNXB_CONV_RELAY = 0 | 1 pins the choice for A/B measurements.
        if (plan.ctas == 2 && plan.KB == 4) plan.relay = 1;
        if (const char *e = getenv("ONNXB_CONV_RELAY"))
            if (e[0] == '0' || e[0] == '1') plan.relay = e[0] - '0';
    }
    return have;
}

// How many CTA pairs (clusters of two) of the pair kernel the device runs at once; queried once.
static int max_pairs() {
    static std::atomic<int> cached{-1};
    int n = cached.load(std::memory_order_acquire);
    if (n >= 0) return n;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * 148);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmemLimit;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, tc_conv_kernel<2, kNoAddend, false, false>, &cfg) != cudaSuccess || n < 1) {
        cudaGetLastError();
        n = tc_host::num_sms() / 2;
    }
    cached.store(n, std::memory_order_release);
    return n;
}

size_t tc_conv_workspace_bytes(const TcConvPlan &plan) { return (size_t)plan.packed_floats * 4; }

static int launch_images(const TcConvPlan &plan, const float *X, const float *B, const float *R, float *Y, const void *workspace,
                         unsigned int *err, cudaStream_t st, bool round_y);

int launch_tc_conv(const TcConvPlan &plan, const float *X, const float *W, const float *B, const float *R, float *Y,
                   void *workspace, void *stream, int phase, bool round_y) {
    using namespace tc_host;
    cudaStream_t st = (cudaStream_t)stream;
    unsigned int *err = device_status_ptr();
    if (!err) return (int)cudaErrorUnknown;

    // 1. pack + round the weights into the workspace (skipped when the caller packed them earlier)
    if (phase != kTcConvRunOnly) {
        const dim3 grid = pack_weights_grid(plan, plan.ctiles * plan.ctas, plan.BNH);
        const cudaError_t e = launch_pdl(pack_weights_kernel, grid, dim3(kPackThreads), 0, st, plan, W, reinterpret_cast<float4 *>(workspace));
        count_launch();
        if (e != cudaSuccess) return (int)e;
    }
    if (phase == kTcConvPackOnly) return 0;
    // 2. the convolution; the kernel reaches outputs by 32-bit byte offsets, so an output of 4 GB and more is computed
    // in several launches, some images each
    const long long image = (long long)plan.M * plan.P * plan.Q;
    const int most = (int)std::min<long long>(plan.N, ((1LL << 30) - 1) / image);
    for (int n0 = 0; n0 < plan.N; n0 += most) {
        TcConvPlan part = plan;
        part.N = std::min(most, plan.N - n0);
        part.total_slots = (long long)part.N * part.L;
        part.pix_tiles = (int)((part.total_slots + part.ctas * part.MT * 128 - 1) / (part.ctas * part.MT * 128));
        part.total_tiles = (long long)part.pix_tiles * part.ctiles * part.group;
        const int e = launch_images(part, X + (long long)n0 * plan.C * plan.H * plan.W, B, R ? R + n0 * image : nullptr, Y + n0 * image,
                                    workspace, err, st, round_y);
        if (e != 0) return e;
    }
    return 0;
}

static int launch_images(const TcConvPlan &plan, const float *X, const float *B, const float *R, float *Y, const void *workspace,
                         unsigned int *err, cudaStream_t st, bool round_y) {
    using namespace tc_host;
    CUtensorMap tmX;
    if (plan.raw_mode == 0) {
        const uint64_t HW = (uint64_t)plan.H * plan.W, N = (uint64_t)plan.N, C = (uint64_t)plan.C;
        const uint64_t dims[2] = {plan.x_cm ? N * HW : HW, plan.x_cm ? C : N * C};
        const uint64_t str[1] = {plan.x_cm ? (uint64_t)channel_pitch(plan.N, plan.H, plan.W) * 4 : HW * 4};
        const uint32_t box[2] = {(uint32_t)plan.BOXP, (uint32_t)plan.KBR};
        if (!make_tmap(&tmX, X, 2, dims, str, box, kTmapSwizzleNone)) return (int)cudaErrorInvalidValue;
    } else {
        memset(&tmX, 0, sizeof tmX);
    }
    const size_t smem = smem_with_tmem(1024 + (size_t)plan.na_stages * plan.a_stage_bytes + (size_t)plan.nr_stages * plan.raw_stage_bytes +
                                           (size_t)plan.nb_stages * plan.b_stage_bytes + kMaxRawStages * kSegBytes + kBiasBytes + kBarBytes +
                                           (plan.split > 1 ? split_recv_bytes(plan.split, plan.cols_per) : 0),
                                       plan.split > 1 ? split_tmem_cols(plan.BN) : 512);
    const bool pair = plan.ctas == 2;
    const bool add = R != nullptr;
    const bool split = plan.split > 1;
    if (round_y && (add || plan.KB == 4)) return (int)cudaErrorInvalidValue;
    const bool thin = plan.KB == 4;
    // Asking ahead for an addend is worth it where L2 is unlikely to hold it still (64 -> 64 channels 3x3 56x56 batch 32, 26 MB:
    // 23.9 -> 25.1 us with it) and the main loop is too short to hide the epilogue (64 -> 64 3x3 112x112 batch 32, 72 steps:
    // 97 -> 102; 32 -> 128, 36 steps of 128 columns: 132 -> 138; 32 -> 64, 36 of 64: 77 -> 69; thin layers:
    // 3 -> 256 7x7 64x64 batch 64 197 -> 173, 12 -> 64 5x5 112x112 batch 32 82 -> 72).
    const bool far = add && 4LL * plan.N * plan.M * plan.P * plan.Q >= (64LL << 20) && (thin || plan.ncb * plan.n_steps * plan.BN <= 2560);
    auto kern = round_y ? (split ? tc_conv_kernel<1, kRoundedY, false, true> : pair ? tc_conv_kernel<2, kRoundedY, false, false> : tc_conv_kernel<1, kRoundedY, false, false>)
                : split ? (add ? tc_conv_kernel<1, kAddendNear, false, true> : tc_conv_kernel<1, kNoAddend, false, true>)
                : thin ? (far   ? (pair ? tc_conv_kernel<2, kAddendFar, true, false> : tc_conv_kernel<1, kAddendFar, true, false>)
                          : add ? (pair ? tc_conv_kernel<2, kAddendNear, true, false> : tc_conv_kernel<1, kAddendNear, true, false>)
                                : (pair ? tc_conv_kernel<2, kNoAddend, true, false> : tc_conv_kernel<1, kNoAddend, true, false>))
                       : (far   ? (pair ? tc_conv_kernel<2, kAddendFar, false, false> : tc_conv_kernel<1, kAddendFar, false, false>)
                          : add ? (pair ? tc_conv_kernel<2, kAddendNear, false, false> : tc_conv_kernel<1, kAddendNear, false, false>)
                                : (pair ? tc_conv_kernel<2, kNoAddend, false, false> : tc_conv_kernel<1, kNoAddend, false, false>));
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
    if (e != cudaSuccess) return (int)e;
    const int sms = num_sms();
    // persistent: one CTA per SM; pairs are clusters of two neighbouring SMs
    const int units = pair ? max_pairs() : sms;
    if (units < 1) return (int)cudaErrorLaunchOutOfResources;
    const int grid = split ? (int)plan.total_tiles * plan.split : (int)std::min<long long>(plan.total_tiles, units) * plan.ctas;
#ifdef ONNXB_PROFILE
    fprintf(stderr, "[plan] ctas %d MT %d BN %d ctiles %d SLOTS %d planes %d Hs %d Ws %d L %d KB %d ncb %d steps %d spb %d tiles %lld grid %d raw_mode %d BOXP %d a_stage %d raw_stage %d b_stage %d nb %d smem %zu\n",
            plan.ctas, plan.MT, plan.BN, plan.ctiles, plan.SLOTS, plan.planes, plan.Hs, plan.Ws, plan.L, plan.KB, plan.ncb,
            plan.n_steps, plan.spb, plan.total_tiles, grid, plan.raw_mode, plan.BOXP, plan.a_stage_bytes,
            plan.raw_stage_bytes, plan.b_stage_bytes, plan.nb_stages, smem);
#endif
    const cudaError_t le =
        pair || split ? launch_pdl_cluster(kern, split ? (unsigned)plan.split : 2u, dim3(grid), dim3(kThreads), smem, st, tmX, plan, X,
                                  reinterpret_cast<const float *>(workspace), B, R, Y, err)
             : launch_pdl(kern, dim3(grid), dim3(kThreads), smem, st, tmX, plan, X,
                          reinterpret_cast<const float *>(workspace), B, R, Y, err);
    count_launch();
    return (int)le;
}

}  // namespace onnxb
