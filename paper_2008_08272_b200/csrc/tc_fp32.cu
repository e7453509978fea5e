// fp32 contractions on the TF32 tensor cores: ONNX Gemm (Sec. 3.4.3) and ONNX Conv (Sec. 4.1) for the
// problems that are computed in fp32 because TMA cannot describe an operand (rows that are no multiples
// of 16 bytes, images of odd size), once they are large enough to be worth a tensor-core launch.
//
// Every fp32 operand is split into hi = TF32(x) and lo = TF32(x - hi), which together carry all but the
// last bit of x, and a product is hi*hi + lo*hi + hi*lo (the missing lo*lo is below 2^-24 of the term).
// The tensor core truncates when it adds into its accumulator (measured on exact TF32 operands: the
// relative error of a dot product grows as 2.4e-9 * K, always towards zero), so an accumulator only ever
// covers 32 terms, the large products apart from the small ones; the epilogue warps add these partial sums in fp32
// registers, rounding to nearest, as the FMA kernels do.
//
// What is split where.  Gemm's operands and a convolution's filters are split by a launch of their own into the
// workspace (filters that are constants once, when they are packed), laid out as the tensor core reads them, so that
// one bulk copy brings a block of 32 terms: split by the warps of every tile that reads them, through registers by
// 4-byte loads, the same blocks took 1800 to 3100 cycles against the 768 of their MMAs.  The pixels of a convolution are
// split by five warps on their way into shared memory, ONCE for all taps of a filter: a tile is 128 consecutive slots of the
// padded images with the halo behind them, one 16-byte row per slot and four channels, and a tap reads the same rows from
// another start (plan of the slots: conv_plan_axis, fill, fill_steps).  The MMA's rows are the pixels, or
// the columns of Gemm (what is contiguous in Y: TMEM lanes then store consecutive addresses), its columns the
// channels, or the rows of Gemm.
//
// Bound: the tensor core, three products of 128 x BN x 8 per 8 terms, each reading its operands out of shared memory at
// 128 bytes per cycle (64 cycles at BN = 128, 56 at 96, 48 at 64).
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>
#include <cstdlib>

#include "common.h"
#include "pack_weights.cuh"
#include "tc_common.cuh"
#include "tc_host.h"

namespace onnxb {

namespace {

using namespace tc;

constexpr int kGroupSteps = 4;                  // K-steps of eight terms per partial sum
constexpr int kEpiWarps = 16, kCopyWarp = 16, kMmaWarp = 17, kRawWarp = 18, kFirstXform = 19, kXformWarps = 5;
constexpr int kGemmThreads = kRawWarp * 32, kConvThreads = (kFirstXform + kXformWarps) * 32, kXformThreads = kXformWarps * 32;
constexpr int kBatch = 5;                       // of which so many are in flight
constexpr int kMaxOwned = 3 * kBatch;                   // (slot, chunk) pairs of a stage that a transform thread owns
constexpr int kMaxAStages = 3, kMaxBStages = 8, kRawStages = 2;
constexpr uint32_t kTmemCols = 512;
constexpr int kMaxAccs = 8;
constexpr int kSmemLimit = 232448, kBarBytes = 768;             // barriers, and two tables of a tile's rows
struct Bars {
    uint64_t raw_full[kRawStages], raw_empty[kRawStages], seg_full[2], seg_empty[2];
    uint64_t a_full[kMaxAStages], a_empty[kMaxAStages], b_full[kMaxBStages], b_empty[kMaxBStages], acc_full[kMaxAccs], acc_empty[kMaxAccs];
    uint32_t tmem_holder;
};
static_assert(sizeof(Bars) + 2 * sizeof(Fp32ConvSegs) <= kBarBytes, "barrier block too large");

// One operand of Gemm (or the pixels of a 1x1 convolution, which has no taps to share them), split: [tile][block of 32 terms][K-step][4-term chunk][hi, lo][row of the tile][4] for the column operand (one
// instruction multiplies by both parts), [hi, lo][4-term chunk] for the row operand.  Lanes run along
// what is contiguous in the operand: eight rows of 16 terms, or 32 rows.
struct PackOperand {
    const float *src;
    float4 *dst;
    int n, tile_rows, k_contig;
    unsigned chunk_at, lo_at;    // where the second chunk and the lo part lie, in rows of the tile
    long long ld;                // stride of the index that is not contiguous
    unsigned items;              // rows, padded to whole tiles, x chunks
    // pixels: row j is pixel j % PQ of image j / PQ
    int PQ, Q, row_step, col_step;
    long long image;
    ConvDivisor dv_PQ, dv_Q;
};
__device__ __forceinline__ long long pixel_offset(const PackOperand &o, int j) {
    const int n = conv_fdiv(j, o.PQ, o.dv_PQ), u = j - n * o.PQ, p = conv_fdiv(u, o.Q, o.dv_Q);
    return n * o.image + (long long)p * o.row_step + (long long)(u - p * o.Q) * o.col_step;
}
// Per epilogue warp: eight columns of its rows on their way out, and the biases of its columns.
constexpr int kOutFloats = 8 * 32 + 32, kOutBytes = kEpiWarps * kOutFloats * 4;

struct Args {
    const float4 *Rp, *Cp;       // packed operands: rows (Gemm), columns
    const float *R, *C;          // the operands themselves: rows (Gemm; else X), columns
    long long r_si, r_sk, c_si, c_sk;
    float *Y;
    int rows, cols, K;           // Gemm: N, M, K; convolution: -, channels and terms of a group
    int BN, tiles_r, tiles_c, relu;
    long long tiles;
    int nblk, blk_per, split;    // blocks of the reduction, and how many of them each of `split` CTAs of a cluster sums
    int nb_stages, b_stage_bytes, na_stages, a_bytes, raw_bytes;
    // Gemm epilogue: alpha * D + beta * Cadd
    float alpha, beta;
    const float *Cadd;
    long long cadd_si, cadd_sj;
    // Conv; a 1x1 convolution by packed pixels (PQ > 0) is a Gemm with these in its epilogue
    const float *bias, *Radd;
    PackOperand px;
    Fp32ConvPlan p;
};

__device__ __forceinline__ void tmem_ld_32x16(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ float ld_dsmem(uint32_t addr) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}

// hi to nearest; lo's rounding is completed by the tensor core, which ignores the low 13 bits.  A value that is
// not finite leaves lo = NaN, one that rounds to infinity lo = the opposite infinity, and either way every output it
// takes part in is NaN: the epilogue then sums that output from the operands themselves.  (Whatever a NaN x becomes in
// hi: x - hi is the NaN of GPU arithmetic, 0x7FFFFFFF, which half an ulp more would turn into a zero.  The larger of
// the two as signed integers keeps it, and is the sum for every other value; all 2^32 compared.)
__device__ __forceinline__ void split_tf32(float x, float &hi, float &lo) {
    hi = __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xFFFFE000u);
    int r;
    asm("{\n.reg .s32 t;\nadd.s32 t, %1, 0x1000;\nmax.s32 %0, t, %1;\n}" : "=r"(r) : "r"(__float_as_int(x - hi)));
    lo = __int_as_float(r);
}
__device__ __forceinline__ void split4(const float (&v)[4], float4 &hi, float4 &lo) {
    split_tf32(v[0], hi.x, lo.x);
    split_tf32(v[1], hi.y, lo.y);
    split_tf32(v[2], hi.z, lo.z);
    split_tf32(v[3], hi.w, lo.w);
}

// ------------------------------------------------------------------ packing
__device__ __forceinline__ void pack_item(const PackOperand &o, int K, int nblk, unsigned i) {
    const unsigned chunks = (unsigned)nblk * 8u;
    unsigned row, c;
    if (o.k_contig) {                              // 32 items: 8 rows x 4 chunks
        const unsigned w = i >> 5, l = i & 31u, cw = chunks / 4u;
        row = w / cw * 8u + (l >> 2);
        c = w % cw * 4u + (l & 3u);
    } else {
        const unsigned padded = o.items / chunks;
        c = i / padded;
        row = i - c * padded;
    }
    const unsigned tile = row / (unsigned)o.tile_rows, r = row - tile * (unsigned)o.tile_rows;
    const float *src = o.src + (o.k_contig ? (long long)row * o.ld : o.PQ ? pixel_offset(o, (int)row) : (long long)row);
    const long long ks = o.k_contig ? 1 : o.ld;
    float v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int k = (int)c * 4 + e;
        v[e] = (int)row < o.n && k < K ? __ldg(src + k * ks) : 0.f;
    }
    float4 hi, lo;
    split4(v, hi, lo);
    const unsigned step = c >> 1, k = c & 1u, tr = (unsigned)o.tile_rows;
    float4 *d = o.dst + ((size_t)tile * nblk * kGroupSteps + step) * 4u * tr + k * o.chunk_at + r;
    d[0] = hi;
    d[o.lo_at] = lo;
}
__global__ void __launch_bounds__(256) pack_split_kernel(const __grid_constant__ PackOperand a, const __grid_constant__ PackOperand b, int K, int nblk) {
    pdl_launch_dependents();
    pdl_wait();
    for (unsigned i = blockIdx.x * 256u + threadIdx.x; i < a.items + b.items; i += gridDim.x * 256u) {
        if (i < a.items) pack_item(a, K, nblk, i);
        else pack_item(b, K, nblk, i - a.items);
    }
}

// The filters of a convolution, split: [group][channel tile][block][K-step][chunk][hi, lo][channel of the tile][4].
__global__ void __launch_bounds__(kPackThreads) pack_filters_split_kernel(const __grid_constant__ Fp32ConvPlan p, const float *__restrict__ W, float4 *__restrict__ out) {
    pdl_launch_dependents();
    pack_weights(p, W, p.tiles_c, p.BN, p.nch * 4, [&](size_t tile, int cb, int step, int half, int row, const float (&v)[4]) {
        float4 hi, lo;
        split4(v, hi, lo);
        float4 *d = out + (((tile * p.ncb + cb) * p.n_steps + step) * 2 + half) * 2 * p.BN + row;
        d[0] = hi;
        d[p.BN] = lo;
    });
}

// ------------------------------------------------------------------ tiles and pixels
struct Tile {
    int grp, r, c0;              // row tile (of pixels or of Gemm's columns), first column
};
template <bool kConv>
__device__ __forceinline__ Tile tile_of(const Args &g, long long t) {
    // column tiles fastest: CTAs running at the same time share a row tile's operand in L2
    const int ct = (int)(t % g.tiles_c);
    const long long u = t / g.tiles_c;
    Tile r;
    r.grp = kConv ? (int)(u / g.tiles_r) : 0;
    r.r = kConv ? (int)(u % g.tiles_r) : (int)u;
    r.c0 = ct * g.BN;
    return r;
}
// Image, slot row and slot column of a slot.
__device__ __forceinline__ void slot_of(const Fp32ConvPlan &p, int G, int &n, int &hq, int &wq) {
    n = conv_fdiv(G, p.L, p.dv_L);
    const int u = G - n * p.L;
    hq = conv_fdiv(u, p.Ws, p.dv_Ws);
    wq = u - hq * p.Ws;
}
// Image, output row and column of a tile's row m; false where that is no output of the tile.
__device__ __forceinline__ bool pixel_of(const Fp32ConvPlan &p, int rt, int m, int &n, int &pp, int &q) {
    slot_of(p, fp32_conv_first_slot(p, rt) + m, n, pp, q);
    return n < p.N && pp < p.P && q < p.Q && (!p.per_image || n == conv_fdiv(rt, p.per_image, p.dv_per_image));
}
// Where column 0 of Gemm's row j lies in Y, and the distance to the next.
__device__ __forceinline__ void row_of(const Args &g, int j, long long &ybase, long long &ystep) {
    ybase = j;
    ystep = g.rows;
    if (g.px.PQ) {
        const int n = conv_fdiv(j, g.px.PQ, g.px.dv_PQ);
        ybase += (long long)n * (g.cols - 1) * g.px.PQ;
        ystep = g.px.PQ;
    }
}
// One output from the operands themselves, for those the split cannot carry.
template <bool kConv>
__device__ __noinline__ float dot_plain(const Args &g, int grp, int i, int j, int n, int pp, int q) {
    float d = 0.f;
    if (!kConv) {
        const float *r = g.R + (g.px.PQ ? pixel_offset(g.px, j) : j * g.r_si);
        for (int k = 0; k < g.K; ++k) d = fmaf(__ldg(g.C + i * g.c_si + k * g.c_sk), __ldg(r + k * g.r_sk), d);
        return d;
    }
    const Fp32ConvPlan &p = g.p;
    for (int k = 0; k < g.K; ++k) {
        const int c = k / p.taps, rs = k - c * p.taps, r = rs / p.kW, s = rs - r * p.kW;
        const int h = pp * p.sh - p.pt + r * p.dh, w = q * p.sw - p.pl + s * p.dw;
        const bool in = (unsigned)h < (unsigned)p.H && (unsigned)w < (unsigned)p.W;
        const float x = in ? __ldg(g.R + (((long long)n * p.C + (long long)grp * p.Cg + c) * p.H + h) * p.W + w) : 0.f;
        d = fmaf(__ldg(g.C + (long long)(grp * g.cols + i) * g.K + k), x, d);
    }
    return d;
}

__device__ __forceinline__ Fp32ConvSegs *segs_of(Bars *bars, uint32_t i) { return reinterpret_cast<Fp32ConvSegs *>(bars + 1) + i; }

// ------------------------------------------------------------------ main kernel
template <bool kConv>
__global__ void __launch_bounds__(kConv ? kConvThreads : kGemmThreads, 1)
tc_fp32_kernel(const __grid_constant__ Args g, unsigned int *err) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *b_st = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    uint8_t *a_st = b_st + (size_t)g.nb_stages * g.b_stage_bytes;
    float *raw_st = reinterpret_cast<float *>(a_st + (kConv ? (size_t)g.na_stages * g.a_bytes : 0));
    float *out_st = raw_st + (kConv ? (size_t)kRawStages * (g.raw_bytes / 4) : 0);
    Bars *bars = reinterpret_cast<Bars *>(out_st + kEpiWarps * kOutFloats);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_steps = kConv ? g.p.n_steps : kGroupSteps, spg = kConv ? g.p.spg : kGroupSteps, n_groups = kConv ? g.p.n_groups : 1;
    // a cluster's CTAs share a tile's blocks
    const int rank = g.split > 1 ? (int)cluster_ctarank() : 0;
    const int blk_lo = rank * g.blk_per, nblk = min(g.nblk - blk_lo, g.blk_per);
    // accumulators: the large products' columns, then the small ones'
    const uint32_t acc_cols = g.BN <= 32 ? 64u : g.BN <= 64 ? 128u : 256u, n_acc = kTmemCols / acc_cols;
    const long long first = blockIdx.x / (unsigned)g.split, step_t = gridDim.x / (unsigned)g.split;

    if (warp == kCopyWarp) {
        if (lane < g.nb_stages) {
            mbar_init(&bars->b_full[lane], 1);
            mbar_init(&bars->b_empty[lane], 1);
        }
        if (kConv && lane < g.na_stages) {
            mbar_init(&bars->a_full[lane], kXformWarps);
            mbar_init(&bars->a_empty[lane], 1);
        }
        if (kConv && lane < 2) {
            mbar_init(&bars->raw_full[lane], 1);
            mbar_init(&bars->raw_empty[lane], kXformWarps);
            mbar_init(&bars->seg_full[lane], 1);
            mbar_init(&bars->seg_empty[lane], kXformWarps);
        }
        if (lane < kMaxAccs) {
            mbar_init(&bars->acc_full[lane], 1);
            mbar_init(&bars->acc_empty[lane], kEpiWarps);
        }
        mbar_fence_init();
    }
    if (warp == kMmaWarp) {
        tmem_alloc(&bars->tmem_holder, kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = bars->tmem_holder;
    pdl_launch_dependents();

    if (warp == kCopyWarp) {
        // ------------------------------------------------------------ packed operands, one group of K-steps per stage
        if (elect_one()) {
            const uint32_t c_step = (uint32_t)g.BN * 64u, r_step = 128u * 64u;
            int bs = 0;
            uint32_t phase = 0;
            pdl_wait();
            for (long long t = first; t < g.tiles; t += step_t) {
                const Tile tl = tile_of<kConv>(g, t);
                const long long ct = (long long)tl.grp * g.tiles_c + tl.c0 / g.BN;
                const uint8_t *c = reinterpret_cast<const uint8_t *>(g.Cp) + (ct * g.nblk + blk_lo) * n_steps * c_step;
                const uint8_t *r = reinterpret_cast<const uint8_t *>(g.Rp) + (kConv ? 0 : ((long long)tl.r * g.nblk + blk_lo) * (kGroupSteps * r_step));
                for (int b = 0; b < nblk; ++b)
                    for (int s0 = 0; s0 < n_steps; s0 += spg) {
                        const uint32_t cnt = (uint32_t)min(spg, n_steps - s0);
                        uint8_t *d = b_st + (size_t)bs * g.b_stage_bytes;
                        mbar_wait(&bars->b_empty[bs], phase ^ 1u, err, 40);
                        mbar_arrive_expect_tx(&bars->b_full[bs], cnt * (kConv ? c_step : c_step + r_step));
                        bulk_load_1d(d, c, cnt * c_step, &bars->b_full[bs]);
                        c += cnt * c_step;
                        if (!kConv) {
                            bulk_load_1d(d + kGroupSteps * c_step, r, kGroupSteps * r_step, &bars->b_full[bs]);
                            r += kGroupSteps * r_step;
                        }
                        if (++bs == g.nb_stages) { bs = 0; phase ^= 1u; }
                    }
            }
        }
    } else if (warp == kMmaWarp) {
        // ------------------------------------------------------------ MMAs, issued by one thread
        if (elect_one()) {
            const uint32_t desc_hi = (128u >> 4) | (1u << 14);             // groups of eight rows 128 bytes apart
            const uint32_t a_part = kConv ? (uint32_t)g.a_bytes >> 5 : 256u, b_step = (uint32_t)g.BN * 4u;
            const uint32_t b_lbo = 2u * (uint32_t)g.BN << 16;
            const uint32_t idesc2 = make_idesc_tf32(128, 2 * g.BN, 0, 0), idesc1 = make_idesc_tf32(128, g.BN, 0, 0);
            // (in a cluster an address carries its CTA's rank above the descriptor's 14 bits)
            const uint32_t st16 = (smem_u32(b_st) >> 4) & 0x3FFFu, b_stage16 = (uint32_t)g.b_stage_bytes >> 4;
            const uint32_t as16 = (smem_u32(a_st) >> 4) & 0x3FFFu, a_stage16 = (uint32_t)g.a_bytes >> 4;
            int bs = 0, as = 0;
            uint32_t bphase = 0, aphase = 0, ab = 0, accphase = 0;
            for (long long t = first; t < g.tiles; t += step_t) {
                for (int b = 0; b < nblk; ++b) {
                    if (kConv) mbar_wait(&bars->a_full[as], aphase, err, 41);
                    for (int s0 = 0; s0 < n_steps; s0 += spg) {
                        const int cnt = min(spg, n_steps - s0);
                        const uint32_t d = tmem_base + ab * acc_cols;
                        const uint32_t stage = st16 + (uint32_t)bs * b_stage16, bl = stage | b_lbo;
                        // rows' descriptor of step j: start address and the distance of its two 16-byte chunks
                        uint32_t al[kGroupSteps];
#pragma unroll
                        for (int j = 0; j < kGroupSteps; ++j)
                            al[j] = kConv ? as16 + (uint32_t)as * a_stage16 + g.p.step_a[min(s0 + j, n_steps - 1)] : (stage + kGroupSteps * b_step + (uint32_t)j * 512u) | (128u << 16);
                        mbar_wait(&bars->acc_empty[ab], accphase ^ 1u, err, 42);
                        mbar_wait(&bars->b_full[bs], bphase, err, 43);
                        tc_fence_after_sync();
#pragma unroll
                        for (int j = 0; j < kGroupSteps; ++j)
                            if (j < cnt) {
                                // hi by hi and by lo in one instruction, into the accumulator's two halves, then lo by hi
                                const uint32_t bj = bl + (uint32_t)j * b_step;
                                mma_tf32_lohi(d, al[j], desc_hi, bj, desc_hi, idesc2, j > 0);
                                mma_tf32_lohi(d + (uint32_t)g.BN, al[j] + a_part, desc_hi, bj, desc_hi, idesc1, 1);
                            }
                        mma_commit(&bars->b_empty[bs]);
                        mma_commit(&bars->acc_full[ab]);
                        if (++ab == n_acc) { ab = 0; accphase ^= 1u; }
                        if (++bs == g.nb_stages) { bs = 0; bphase ^= 1u; }
                    }
                    if (kConv) {
                        mma_commit(&bars->a_empty[as]);
                        if (++as == g.na_stages) { as = 0; aphase ^= 1u; }
                    }
                }
            }
        }
    } else if (kConv && warp == kRawWarp) {
        // ------------------------------------------------------------ raw rows: one copy per channel and image, a lane each
        // Rows of X have any alignment, copies whole 16-byte pieces: a copy starts up to three elements early and ends up to three
        // late, and lands as far from a 16-byte boundary as it lies in X.  The last elements of X, where they are no whole
        // piece, are brought by plain loads.
        const Fp32ConvPlan &p = g.p;
        const int HW = p.H * p.W, x_whole = (p.N * p.C * HW) & ~3, x_end = p.N * p.C * HW;
        int rs = 0;
        uint32_t phase = 0, tile_it = 0;
        for (long long t = first; t < g.tiles; t += step_t, ++tile_it) {
            const Tile tl = tile_of<kConv>(g, t);
            Fp32ConvSegs *segs = segs_of(bars, tile_it & 1u);
            mbar_wait(&bars->seg_empty[tile_it & 1u], ((tile_it >> 1) & 1u) ^ 1u, err, 46);
            if (lane == 0) {
                fp32_conv_segments(p, tl.r, tl.grp, *segs);
                mbar_arrive(&bars->seg_full[tile_it & 1u]);
            }
            __syncwarp();
            if (tile_it == 0) pdl_wait();
            const int nseg = segs->nseg;
            for (int b = blk_lo; b < blk_lo + nblk; ++b) {
                const int chans = min(p.nch * 4, p.Cg - b * p.nch * 4), copies = chans * nseg;
                mbar_wait(&bars->raw_empty[rs], phase ^ 1u, err, 47);
                float *stage = raw_st + (size_t)rs * (g.raw_bytes / 4);
                // (at most 32 * 4 copies)
                int from[4], to[4], bytes[4], sum = 0;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int u = lane + k * 32, c = u / nseg, i = u - c * nseg;
                    bytes[k] = 0;
                    if (u < copies && segs->len[i] > 0) {
                        const int e = ((segs->n_first + i) * p.C + tl.grp * p.Cg + b * p.nch * 4 + c) * HW + segs->f0[i], d = c * p.pitch + segs->at[i];
                        const int last = e + segs->len[i];
                        from[k] = e & ~3;
                        to[k] = d - (e & 3);
                        bytes[k] = (fp32_conv_copy_end(last, x_whole) - from[k]) * 4;
                        if (last > x_whole)
                            for (int x = max(e, x_whole); x < x_end; ++x) stage[d + x - e] = __ldg(g.R + x);
                    }
                    sum += bytes[k];
                }
                sum = (int)__reduce_add_sync(0xffffffffu, (unsigned)sum);
                __syncwarp();                        // (the plain stores come before the arrival)
                if (lane == 0) mbar_arrive_expect_tx(&bars->raw_full[rs], (uint32_t)sum);
                __syncwarp();
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (bytes[k] > 0) bulk_load_1d(stage + to[k], g.R + from[k], (uint32_t)bytes[k], &bars->raw_full[rs]);
                if (++rs == kRawStages) { rs = 0; phase ^= 1u; }
            }
        }
    } else if (kConv && warp >= kFirstXform) {
        // ------------------------------------------------------------ pixels: split and laid out once for all taps
        const Fp32ConvPlan &p = g.p;
        const int tid = threadIdx.x - kFirstXform * 32, slots = p.planes * p.SLOTS, units = slots * p.nch;
        const uint32_t a_part = (uint32_t)g.a_bytes >> 1;
        int off[kMaxOwned];                  // of the unit's first channel in a raw stage, -1: padding
        int as = 0, rs = 0;
        uint32_t aphase = 0, rphase = 0, tile_it = 0;
        for (long long t = first; t < g.tiles; t += step_t, ++tile_it) {
            const Tile tl = tile_of<kConv>(g, t);
            const int G0 = fp32_conv_first_slot(p, tl.r);
            const Fp32ConvSegs *segs = segs_of(bars, tile_it & 1u);
            mbar_wait(&bars->seg_full[tile_it & 1u], (tile_it >> 1) & 1u, err, 48);
#pragma unroll
            for (int e = 0; e < kMaxOwned; ++e) {
                off[e] = -1;
                const int u = tid + e * kXformThreads;
                if (u < units) {
                    const int ch = conv_fdiv(u, slots, p.dv_slots), s = u - ch * slots, pl = conv_fdiv(s, p.SLOTS, p.dv_SLOTS);
                    int n, hq, wq;
                    slot_of(p, G0 + s - pl * p.SLOTS, n, hq, wq);
                    const int h = hq * p.sh + p.pa[pl] - p.pt, w = wq * p.sw + p.pb[pl] - p.pl, i = n - segs->n_first;
                    if (i < segs->nseg && (unsigned)h < (unsigned)p.H && (unsigned)w < (unsigned)p.W)
                        off[e] = ch * 4 * p.pitch + segs->at[i] + h * p.W + w - segs->f0[i];
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars->seg_empty[tile_it & 1u]);
            for (int b = blk_lo; b < blk_lo + nblk; ++b) {
                const float *raw = raw_st + (size_t)rs * (g.raw_bytes / 4);
                uint8_t *d = a_st + (size_t)as * g.a_bytes;
                const int c_left = (p.Cg - b * p.nch * 4) * p.pitch;       // channels that exist, as a distance in the stage
                mbar_wait(&bars->raw_full[rs], rphase, err, 49);
                mbar_wait(&bars->a_empty[as], aphase ^ 1u, err, 44);
#pragma unroll
                for (int e0 = 0; e0 < kMaxOwned; e0 += kBatch) {
                    if (e0 * kXformThreads >= units) break;
                    float v[kBatch][4];
#pragma unroll
                    for (int x = 0; x < kBatch; ++x)
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            // (a channel's own offset is below the pitch)
                            const int o = off[e0 + x] + k * p.pitch;
                            v[x][k] = off[e0 + x] >= 0 && o < c_left ? raw[o] : 0.f;
                        }
#pragma unroll
                    for (int x = 0; x < kBatch; ++x) {
                        const int u = tid + (e0 + x) * kXformThreads;
                        if (u < units) {
                            float4 hi, lo;
                            split4(v[x], hi, lo);
                            *reinterpret_cast<float4 *>(d + u * 16) = hi;
                            *reinterpret_cast<float4 *>(d + a_part + u * 16) = lo;
                        }
                    }
                }
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&bars->a_full[as]);
                    mbar_arrive(&bars->raw_empty[rs]);
                }
                if (++as == g.na_stages) { as = 0; aphase ^= 1u; }
                if (++rs == kRawStages) { rs = 0; rphase ^= 1u; }
            }
        }
    } else if (warp < kEpiWarps) {
        // ------------------------------------------------------------ partial sums and epilogue
        // Sixteen warps, four to a TMEM lane quarter, each with every fourth 16-column chunk of the tile.
        const int quarter = warp & 3, first_chunk = warp >> 2, chunks = g.BN / 16;
        const int nch = first_chunk < chunks ? (chunks - first_chunk + 3) / 4 : 0;             // (one or two)
        uint32_t ab = 0, accphase = 0;
        const int n_flush = nblk * n_groups;
        float *out = out_st + warp * kOutFloats, *bias = out + 8 * 32;
        pdl_wait();
        for (long long t = first; t < g.tiles; t += step_t) {
            const Tile tl = tile_of<kConv>(g, t);
            {
                const int col = tl.c0 + (first_chunk + (lane >> 4) * 4) * 16 + (lane & 15);
                __syncwarp();
                bias[lane] = g.bias && col < min(g.cols, tl.c0 + g.BN) ? __ldg(g.bias + tl.grp * g.cols + col) : 0.f;
            }
            float acc[32];
#pragma unroll
            for (int e = 0; e < 32; ++e) acc[e] = 0.f;
            for (int f = 0; f < n_flush; ++f) {
                mbar_wait(&bars->acc_full[ab], accphase, err, 45);
                tc_fence_after_sync();
                const uint32_t ta = tmem_base + ab * acc_cols + ((uint32_t)(quarter * 32) << 16) + (uint32_t)first_chunk * 16u;
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    if (c < nch) {
                        uint32_t x[16], y[16];
                        tmem_ld_32x16(ta + (uint32_t)g.BN + c * 64u, x);
                        tmem_ld_32x16(ta + c * 64u, y);
                        tmem_ld_wait();
#pragma unroll
                        for (int e = 0; e < 16; ++e) acc[c * 16 + e] += __uint_as_float(x[e]) + __uint_as_float(y[e]);
                    }
                }
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars->acc_empty[ab]);
                if (++ab == n_acc) { ab = 0; accphase ^= 1u; }
            }
            if (g.split > 1) {
                // every MMA has completed and every stage been read: the partial tile takes the ring's place, [column][row]
                float *part = reinterpret_cast<float *>(b_st) + first_chunk * (16 * 128) + quarter * 32 + lane;
#pragma unroll
                for (int e = 0; e < 32; ++e)
                    if (e < nch * 16) part[((e >> 4) * 64 + (e & 15)) * 128] = acc[e];
                break;
            }
            const int m = quarter * 32 + lane;
            int n = 0, pp = 0, q = 0, j = tl.r * 128 + m;
            bool rowok;
            long long ybase, ystep;
            if (kConv) {
                rowok = pixel_of(g.p, tl.r, m, n, pp, q);
                ystep = (long long)g.p.P * g.p.Q;
                ybase = rowok ? ((long long)n * g.p.M + (long long)tl.grp * g.cols) * ystep + (long long)pp * g.p.Q + q : 0;
            } else {
                rowok = j < g.rows;
                row_of(g, j, ybase, ystep);
            }
            // Out by way of shared memory, eight columns at a time: the accumulators' indices are constants, and a copy of the
            // code below for every one of them ran at the rate of cold instruction fetches (96 columns: 9400 cycles).
            // (a residual addend lies as Y does)
            const float *const addend = g.Radd ? g.Radd : g.Cadd;
            const bool has_add = addend != nullptr;
            const long long add_step = g.Radd ? ystep : g.cadd_si;
            bool bad = false;
#pragma unroll 1
            for (int c = 0; c < 2 * nch; ++c) {
                const int i0 = tl.c0 + (first_chunk + (c >> 1) * 4) * 16 + (c & 1) * 8, cnt = g.cols - i0;      // columns (above 8: all)
                const float *add = !has_add ? g.Y : addend + i0 * add_step + (g.Radd ? ybase : j * g.cadd_sj);
                float r[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    r[e] = has_add && rowok && e < cnt ? __ldg(add) : 0.f;
                    add += add_step;
                }
                __syncwarp();
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (k == c) {
#pragma unroll
                        for (int e = 0; e < 8; ++e) out[e * 32 + lane] = acc[k * 8 + e];
                    }
                __syncwarp();
                float *y = g.Y + ybase + (long long)i0 * ystep;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const float d = out[e * 32 + lane];
                    float v = kConv ? (d + bias[c * 8 + e]) + r[e] : fmaf(g.alpha, d, g.beta * r[e]) + bias[c * 8 + e];
                    if (g.relu) v = v > 0.f ? v : 0.f;
                    if (rowok && e < cnt) {
                        bad |= d != d;
                        *y = v;
                    }
                    y += ystep;
                }
            }
            if (bad) {      // an operand the split cannot carry (see split_tf32): this row again, term by term
                for (int c = 0; c < nch * 16; ++c) {
                    const int i = tl.c0 + (first_chunk + (c >> 4) * 4) * 16 + (c & 15);
                    if (i >= g.cols) break;
                    float v = dot_plain<kConv>(g, tl.grp, i, j, n, pp, q);
                    const float r = has_add ? __ldg(addend + i * add_step + (g.Radd ? ybase : j * g.cadd_sj)) : 0.f;
                    v = kConv ? (v + bias[c]) + r : fmaf(g.alpha, v, g.beta * r) + bias[c];
                    if (g.relu) v = v > 0.f ? v : 0.f;
                    g.Y[ybase + (long long)i * ystep] = v;
                }
            }
        }
    }

    if (g.split > 1) {
        // Each CTA adds its share of the columns over the cluster's partial tiles, in rank order.
        __syncwarp();
        cluster_sync_all();
        pdl_wait();
        const Tile tl = tile_of<kConv>(g, first);
        const int m = threadIdx.x & 127, per = (g.BN + g.split - 1) / g.split, groups = (int)blockDim.x / 128;
        const int lo = rank * per, hi = min(min(g.BN, lo + per), g.cols - tl.c0), j = tl.r * 128 + m;
        int n = 0, pp = 0, q = 0;
        bool rowok = (int)threadIdx.x < groups * 128;
        long long ybase, ystep;
        if (kConv) {
            rowok = pixel_of(g.p, tl.r, m, n, pp, q) && rowok;
            ystep = (long long)g.p.P * g.p.Q;
            ybase = rowok ? ((long long)n * g.p.M + (long long)tl.grp * g.cols) * ystep + (long long)pp * g.p.Q + q : 0;
        } else {
            rowok = rowok && j < g.rows;
            row_of(g, j, ybase, ystep);
        }
        const uint32_t base = smem_u32(b_st);
        for (int c = lo + (int)threadIdx.x / 128; rowok && c < hi; c += groups) {
            const int i = tl.c0 + c;
            float add = 0.f, r = 0.f, d = 0.f;
            if (g.bias) add = __ldg(g.bias + tl.grp * g.cols + i);
            if (g.Radd) r = __ldg(g.Radd + ybase + (long long)i * ystep);
            else if (g.Cadd) r = __ldg(g.Cadd + i * g.cadd_si + j * g.cadd_sj);
            float x[8];
#pragma unroll
            for (int s = 0; s < 8; ++s) x[s] = s < g.split ? ld_dsmem(map_to_cta(base + (uint32_t)(c * 128 + m) * 4u, (uint32_t)s)) : 0.f;
#pragma unroll
            for (int s = 0; s < 8; ++s)
                if (s < g.split) d += x[s];
            if (d != d) d = dot_plain<kConv>(g, tl.grp, i, j, n, pp, q);
            float v = kConv ? (d + add) + r : fmaf(g.alpha, d, g.beta * r) + add;
            if (g.relu) v = v > 0.f ? v : 0.f;
            g.Y[ybase + (long long)i * ystep] = v;
        }
        cluster_sync_all();                         // no CTA leaves while a peer still reads its partial tile
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == kMmaWarp) {
        __syncwarp();
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, kTmemCols);
    }
}

// ------------------------------------------------------------------ planning (host)
// Cycles of a K-step's two instructions: the tensor pipe, or their operands out of shared memory.
double step_cycles(int bn) { return std::max(bn * 1.0, 32.0 + bn * 0.5) + std::max(bn * 0.5, 32.0 + bn * 0.25); }
// Cycles of a partial sum over `steps` K-steps: its MMAs, the epilogue warps adding it up, or its bytes out of L2.
double group_cycles(int bn, int steps, double bytes) { return std::max({steps * step_cycles(bn) * 1.08 + 60.0, 400.0 + 3.0 * bn, bytes / 60.0}); }
// Cycles of a tile's outputs on their way out (the store path: rows of any alignment).
double out_cycles(int bn) { return 1500.0 + 60.0 * bn; }
int cluster_units(int split) { return split == 8 ? 14 : split == 4 ? 33 : 148 / split; }
// A cluster's exchange, and what starting another round of clusters costs.
double split_cycles(int split, double rounds) { return split > 1 ? 2500.0 + 9000.0 * (rounds - 1.0) : 0.0; }

}  // namespace

// Tile width and split of a Gemm's K blocks with the shortest estimated time in cycles (of the packing launch too).
double tc_fp32_gemm_plan(int M, int N, int K, Fp32GemmPlan &out) {
    const int nblk = (K + 31) / 32;
    const long long tiles_r = (N + 127) / 128;
    double best = -1;
    int pb = 0, ps = 0;                              // ONNXB_FP32_GEMM = "BN,split" pins the plan for A/B measurements
    const char *e = getenv("ONNXB_FP32_GEMM");
    if (!e || sscanf(e, "%d,%d", &pb, &ps) != 2) pb = 0;
    for (int bn = 16; bn <= 128 && bn <= (M + 15) / 16 * 16; bn += 16) {
        const long long tiles = tiles_r * ((M + bn - 1) / bn);
        const double blk = group_cycles(bn, kGroupSteps, (128.0 + bn) * 256.0);
        for (int s = 1; s <= 8; s *= 2) {
            const int per = (nblk + s - 1) / s;
            if (per * (s - 1) >= nblk || tiles * s > 2147483647LL) continue;
            if (pb && (bn != pb || s != ps)) continue;
            const double rounds = (double)((tiles + cluster_units(s) - 1) / cluster_units(s));
            const double packed = 8.0 * 32 * nblk * (tiles_r * 128.0 + (double)((M + bn - 1) / bn) * bn);
            const double cost = rounds * (per * blk + out_cycles(bn)) + split_cycles(s, rounds) + 9000.0 + 4000.0 + packed / 1500.0;
            if (best < 0 || cost < best) {
                best = cost;
                out = {bn, s};
            }
        }
    }
    return best;
}

size_t tc_fp32_gemm_workspace(int M, int N, int K, const Fp32GemmPlan &p) {
    return ((size_t)(N + 127) / 128 * 128 + (size_t)(M + p.BN - 1) / p.BN * p.BN) * ((size_t)(K + 31) / 32 * 32) * 8;
}

namespace {

size_t stage_smem(const Args &a, bool conv) {
    return 128 + (size_t)a.nb_stages * a.b_stage_bytes + (conv ? (size_t)a.na_stages * a.a_bytes + (size_t)kRawStages * a.raw_bytes : 0) + kOutBytes + kBarBytes;
}
template <bool kConv>
int launch(Args &a, cudaStream_t st) {
    unsigned int *err = device_status_ptr();
    if (!err) return (int)cudaErrorUnknown;
    auto kern = tc_fp32_kernel<kConv>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
    if (e != cudaSuccess) return (int)e;
    const size_t smem = smem_with_tmem(stage_smem(a, kConv), kTmemCols);
    const dim3 block(kConv ? kConvThreads : kGemmThreads);
    const cudaError_t le =
        a.split > 1 ? tc_host::launch_pdl_cluster(kern, (unsigned)a.split, dim3((unsigned)(a.tiles * a.split)), block, smem, st, a, err)
                    : tc_host::launch_pdl(kern, dim3((unsigned)std::min<long long>(a.tiles, tc_host::num_sms())), block, smem, st, a, err);
    count_launch();
    return (int)le;
}

}  // namespace

namespace {

// Packs both operands and multiplies: `a` holds the problem and its epilogue, `r` and `c` the operands but for where their copies go.
int pack_and_multiply(Args &a, PackOperand r, PackOperand c, const Fp32GemmPlan &plan, void *workspace, cudaStream_t st) {
    const int nblk = (a.K + 31) / 32;
    a.BN = plan.BN; a.tiles_r = (a.rows + 127) / 128; a.tiles_c = (a.cols + plan.BN - 1) / plan.BN;
    a.tiles = (long long)a.tiles_r * a.tiles_c;
    a.nblk = nblk; a.split = plan.split; a.blk_per = (nblk + plan.split - 1) / plan.split;
    a.b_stage_bytes = kGroupSteps * 64 * (128 + plan.BN);
    a.nb_stages = std::min({kMaxBStages, (kSmemLimit - 128 - kOutBytes - kBarBytes) / a.b_stage_bytes, std::max(2, a.blk_per)});
    r.n = a.rows; r.tile_rows = 128; r.chunk_at = 128; r.lo_at = 256;
    r.items = (unsigned)a.tiles_r * 128u * (unsigned)nblk * 8u;
    r.dst = static_cast<float4 *>(workspace);
    c.n = a.cols; c.tile_rows = plan.BN; c.chunk_at = 2u * (unsigned)plan.BN; c.lo_at = (unsigned)plan.BN;
    c.items = (unsigned)(a.tiles_c * plan.BN) * (unsigned)nblk * 8u;
    c.dst = r.dst + (size_t)r.items * 2;
    a.R = r.src; a.C = c.src; a.Rp = r.dst; a.Cp = c.dst;
    const unsigned blocks = std::min((r.items + c.items + 255) / 256, 148u * 16);
    const cudaError_t e = tc_host::launch_pdl(pack_split_kernel, dim3(blocks), dim3(256), 0, st, r, c, a.K, nblk);
    count_launch();
    if (e != cudaSuccess) return (int)e;
    return launch<false>(a, st);
}

}  // namespace

int launch_tc_fp32_gemm(const GemmProblem &p, const Fp32GemmPlan &plan, const float *A, const float *B, const float *C, float *Y,
                        void *workspace, void *stream) {
    Args a{};
    a.Y = Y; a.rows = p.N; a.cols = p.M; a.K = p.K; a.relu = p.relu;
    a.r_si = p.transB ? p.K : 1; a.r_sk = p.transB ? 1 : p.N;
    a.c_si = p.transA ? 1 : p.K; a.c_sk = p.transA ? p.M : 1;
    a.alpha = p.alpha; a.beta = p.beta; a.Cadd = C; a.cadd_si = p.c_stride_i; a.cadd_sj = p.c_stride_j;
    PackOperand r{}, c{};
    r.src = B; r.k_contig = p.transB != 0; r.ld = p.transB ? p.K : p.N;
    c.src = A; c.k_contig = p.transA == 0; c.ld = p.transA ? p.M : p.K;
    return pack_and_multiply(a, r, c, plan, workspace, (cudaStream_t)stream);
}

// An unpadded 1x1 convolution of one group: the pixels it reads are packed like Gemm's columns.
int launch_tc_fp32_conv1x1(const ConvGeom &g, const Fp32GemmPlan &plan, const float *X, const float *W, const float *B, const float *R,
                           float *Y, void *workspace, void *stream) {
    Args a{};
    a.Y = Y; a.rows = g.N * g.P * g.Q; a.cols = g.M; a.K = g.C; a.relu = g.relu;
    a.r_sk = (long long)g.H * g.W; a.c_si = g.C; a.c_sk = 1;
    a.alpha = 1.f; a.beta = 1.f; a.bias = B; a.Radd = R;
    PackOperand r{}, c{};
    r.src = X; r.ld = a.r_sk; r.image = a.r_sk * g.C;
    r.PQ = g.P * g.Q; r.Q = g.Q; r.row_step = g.sh * g.W; r.col_step = g.sw;
    r.dv_PQ = conv_divisor(r.PQ); r.dv_Q = conv_divisor(r.Q);
    a.px = r;
    c.src = W; c.k_contig = 1; c.ld = g.C;
    return pack_and_multiply(a, r, c, plan, workspace, (cudaStream_t)stream);
}

// ---- convolutions
namespace {

// Fills the shared-memory side of a plan; false where it does not fit.
bool conv_stages(const Fp32ConvPlan &p, Args &a) {
    a.a_bytes = p.planes * p.SLOTS * p.nch * 32;
    a.raw_bytes = (p.nch * 4 * p.pitch * 4 + 127) / 128 * 128;
    a.b_stage_bytes = p.spg * p.BN * 64;
    const long long room = kSmemLimit - 128 - kOutBytes - kBarBytes - (long long)kRawStages * a.raw_bytes;
    const int per = (p.ncb + p.split - 1) / p.split;
    a.na_stages = std::min(per, room - 3LL * a.a_bytes >= 4LL * a.b_stage_bytes ? 3 : 2);
    a.nb_stages = (int)std::min<long long>({kMaxBStages, (room - (long long)a.na_stages * a.a_bytes) / std::max(1, a.b_stage_bytes), std::max(2, per * p.n_groups)});
    if (room < (long long)a.na_stages * a.a_bytes || a.nb_stages < 2) return false;
    return p.split == 1 || a.nb_stages * a.b_stage_bytes + a.na_stages * a.a_bytes >= p.BN * 512;
}

double conv_cost(const Fp32ConvPlan &p) {
    const long long tiles = (long long)p.tiles_r * p.tiles_c * p.group;
    const double rounds = (double)((tiles + cluster_units(p.split) - 1) / cluster_units(p.split));
    const int units = p.planes * p.SLOTS * p.nch, per = (p.ncb + p.split - 1) / p.split;
    // Per block the slower of its partial sums (each some 90 cycles longer than Gemm's) and its transform, 320 cycles per unit
    // of a thread; a tile's offsets are another 650 per unit.  Within 15 % of ten measured layers but one (25 %).
    const double owned = (units + kXformThreads - 1) / kXformThreads;
    double mma = 0;
    for (int s = 0; s < p.n_steps; s += p.spg) {
        const int cnt = std::min(p.spg, p.n_steps - s);
        mma += group_cycles(p.BN, cnt, cnt * p.BN * 64.0) * 1.07 + 90.0;
    }
    return rounds * (per * (std::max(mma, 320.0 * owned) + 400.0) + 650.0 * owned + out_cycles(p.BN)) + split_cycles(p.split, rounds) + 9000.0;
}

bool fill(const ConvGeom &c, const ConvAxis &ah, const ConvAxis &aw, int nch, int bn, int split, Fp32ConvPlan &p) {
    p.N = c.N; p.C = c.C; p.H = c.H; p.W = c.W; p.M = c.M; p.Cg = c.Cg; p.Mg = c.Mg; p.kW = c.kW; p.P = c.P; p.Q = c.Q;
    p.pt = c.pt; p.pl = c.pl; p.sh = c.sh; p.sw = c.sw; p.dh = c.dh; p.dw = c.dw; p.group = c.group; p.taps = c.kH * c.kW;
    p.Hs = ah.E; p.Ws = aw.E; p.BN = bn; p.nch = nch; p.split = split;
    p.planes = ah.npar * aw.npar;
    p.a_min = ah.par[0]; p.a_max = ah.par[ah.npar - 1];
    const long long L = (long long)p.Hs * p.Ws, slots = 128 + (long long)ah.Amax * p.Ws + aw.Amax;
    if (L > (1 << 24) || c.N * L + slots + 4096 >= (1LL << 31)) return false;
    if (slots * p.planes * nch > kMaxOwned * kXformThreads) return false;
    p.L = (int)L;
    p.SLOTS = (int)slots;
    // tiles of one image each where those are fewer: they leave out what lies between the images
    const long long across = (c.N * L + 127) / 128, each = ((c.P - 1LL) * p.Ws + c.Q + 127) / 128;
    p.per_image = c.N * each < across ? (int)each : 0;
    p.tiles_r = (int)(p.per_image ? c.N * each : across);
    const long long nseg = (slots + L - 2) / L + 1, rows = std::min((slots + p.Ws - 2) / p.Ws + 1, nseg * p.Hs) * c.sh;
    if (nseg > kFp32MaxSeg || nseg * nch * 4 > 128) return false;
    long long pitch = std::min(rows, nseg * c.H) * c.W + nseg * 10 + 4;      // (a segment's place is rounded up and shifted, its copies end late)
    while ((pitch - (long long)c.H * c.W) % 4 != 0) ++pitch;
    if (pitch * nch * 16 > kSmemLimit) return false;
    p.pitch = (int)pitch;
    p.ncb = (c.Cg + 4 * nch - 1) / (4 * nch);
    if (split > 1 && (p.ncb + split - 1) / split * (split - 1) >= p.ncb) return false;
    p.tiles_c = (c.Mg + bn - 1) / bn;
    p.n_steps = (nch * p.taps + 1) / 2;
    if (p.n_steps > kFp32MaxSteps) return false;
    p.n_groups = (p.n_steps + kGroupSteps - 1) / kGroupSteps;
    p.spg = (p.n_steps + p.n_groups - 1) / p.n_groups;
    p.n_groups = (p.n_steps + p.spg - 1) / p.spg;
    if (2LL * p.group * p.tiles_c * p.ncb * p.n_steps * bn >= (1LL << 31)) return false;
    return (long long)p.tiles_r * p.tiles_c * p.group * split <= 2147483647LL;
}

// Where every (chunk, tap) pair of a block lies in its stage, two to a K-step, in the order of their places.
bool fill_steps(const ConvGeom &c, const ConvAxis &ah, const ConvAxis &aw, Fp32ConvPlan &p) {
    for (int i = 0; i < ah.npar; ++i)
        for (int j = 0; j < aw.npar; ++j) {
            p.pa[i * aw.npar + j] = (short)ah.par[i];
            p.pb[i * aw.npar + j] = (short)aw.par[j];
        }
    // Pairs of one tap's neighbouring chunks; the taps of a last odd chunk pair up among themselves, each with one half the taps
    // further on.
    struct Atom {
        int at, tap, c0;
    } atoms[2 * kFp32MaxSteps];
    auto atom = [&](int ch, int tap) {
        const int r = tap / c.kW, s = tap - r * c.kW, a = r * c.dh % c.sh, b = s * c.dw % c.sw;
        int pl = 0;
        while (p.pa[pl] != a || p.pb[pl] != b) ++pl;
        return Atom{(ch * p.planes + pl) * p.SLOTS + r * c.dh / c.sh * p.Ws + s * c.dw / c.sw, tap, ch * 4};
    };
    int n = 0;
    for (int ch = 0; ch + 1 < p.nch; ch += 2)
        for (int tap = 0; tap < p.taps; ++tap) {
            atoms[n++] = atom(ch, tap);
            atoms[n++] = atom(ch + 1, tap);
        }
    if (p.nch % 2) {
        Atom rest[2 * kFp32MaxSteps];
        for (int tap = 0; tap < p.taps; ++tap) rest[tap] = atom(p.nch - 1, tap);
        std::sort(rest, rest + p.taps, [](const Atom &x, const Atom &y) { return x.at < y.at; });
        const int half = (p.taps + 1) / 2;
        for (int i = 0; i < half; ++i) {
            atoms[n++] = rest[i];
            if (i + half < p.taps) atoms[n++] = rest[i + half];
        }
    }
    for (int s = 0; s < p.n_steps; ++s) {
        const Atom &x = atoms[2 * s];
        const bool two = 2 * s + 1 < n;
        const int gap = two ? atoms[2 * s + 1].at - x.at : 0;
        if (gap < 0 || gap >= (1 << 14)) return false;
        p.step_a[s] = (uint32_t)x.at | (uint32_t)gap << 16;
        p.src_tap[s][0] = (short)x.tap;
        p.src_c0[s][0] = (short)x.c0;
        p.src_tap[s][1] = (short)(two ? atoms[2 * s + 1].tap : -1);      // a lone last one is read twice, its second weights are zero
        p.src_c0[s][1] = (short)(two ? atoms[2 * s + 1].c0 : 0);
    }
    p.dv_L = conv_divisor(p.L);
    p.dv_Ws = conv_divisor(p.Ws);
    p.dv_slots = conv_divisor(p.planes * p.SLOTS);
    if (p.per_image) p.dv_per_image = conv_divisor(p.per_image);
    p.dv_SLOTS = conv_divisor(p.SLOTS);
    return true;
}

}  // namespace

// Plan with the shortest estimated time, and that time in cycles; negative: none.
double tc_fp32_conv_plan(const ConvGeom &c, Fp32ConvPlan &plan) {
    ConvAxis ah, aw;
    if (!conv_plan_axis(c.H, c.P, c.pt, c.sh, c.dh, c.kH, ah) || !conv_plan_axis(c.W, c.Q, c.pl, c.sw, c.dw, c.kW, aw)) return -1;
    if (ah.npar * aw.npar > kFp32MaxPlanes || (long long)c.kH * c.kW > 2 * kFp32MaxSteps) return -1;
    int f[3] = {-1, 0, 0};                           // ONNXB_FP32_TILE = "chunks,BN,split" pins the plan for A/B measurements
    if (const char *e = getenv("ONNXB_FP32_TILE"))
        if (sscanf(e, "%d,%d,%d", &f[0], &f[1], &f[2]) != 3) f[0] = -1;
    double best = -1;
    for (int nch = 1; nch <= 16 && nch <= (c.Cg + 3) / 4; ++nch)
        for (int bn = 16; bn <= 128 && bn <= (c.Mg + 15) / 16 * 16; bn += 16)
            for (int split = 1; split <= 8; split *= 2) {
                if (f[0] >= 0 && (nch != f[0] || bn != f[1] || split != f[2])) continue;
                Fp32ConvPlan p{};
                Args a{};
                if (!fill(c, ah, aw, nch, bn, split, p) || !conv_stages(p, a)) continue;
                const double cost = conv_cost(p);
                if (best < 0 || cost < best) {
                    best = cost;
                    plan = p;
                }
            }
    return best >= 0 && fill_steps(c, ah, aw, plan) ? best : -1;
}

size_t tc_fp32_conv_workspace(const Fp32ConvPlan &p) { return (size_t)p.group * p.tiles_c * p.ncb * p.n_steps * p.BN * 64; }

int launch_tc_fp32_conv(const ConvGeom &g, const Fp32ConvPlan &p, const float *X, const float *W, const float *B, const float *R, float *Y,
                        void *packed, void *stream, int phase) {
    cudaStream_t st = (cudaStream_t)stream;
    if (phase != kTcConvRunOnly) {
        const cudaError_t e = tc_host::launch_pdl(pack_filters_split_kernel, pack_weights_grid(p, p.tiles_c, p.BN), dim3(kPackThreads), 0, st, p, W,
                                                  static_cast<float4 *>(packed));
        count_launch();
        if (e != cudaSuccess) return (int)e;
    }
    if (phase == kTcConvPackOnly) return 0;
    Args a{};
    a.Cp = static_cast<const float4 *>(packed);
    a.R = X; a.C = W; a.Y = Y; a.cols = g.Mg; a.K = g.Cg * p.taps;
    a.BN = p.BN; a.tiles_r = p.tiles_r; a.tiles_c = p.tiles_c; a.relu = g.relu;
    a.tiles = (long long)p.tiles_r * p.tiles_c * p.group;
    a.nblk = p.ncb; a.split = p.split; a.blk_per = (p.ncb + p.split - 1) / p.split;
    a.bias = B; a.Radd = R; a.p = p;
    if (!conv_stages(p, a)) return (int)cudaErrorInvalidConfiguration;
    return launch<true>(a, st);
}

}  // namespace onnxb
