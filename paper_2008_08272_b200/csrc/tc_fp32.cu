// fp32 contractions on the TF32 tensor cores: ONNX Gemm (Sec. 3.4.3) and ONNX Conv (Sec. 4.1) for the
// problems that are computed in fp32 because TMA cannot describe an operand (rows that are no multiples
// of 16 bytes, images of odd size), once they are large enough to be worth a tensor-core launch.
//
// Every fp32 operand is split into hi = TF32(x) and lo = TF32(x - hi), which together carry all but the
// last bit of x, and a product is hi*hi + lo*hi + hi*lo (the missing lo*lo is below 2^-24 of the term).
// The tensor core truncates when it adds into its accumulator (measured on exact TF32 operands: the
// relative error of a dot product grows as 2.4e-9 * K, always towards zero), so an accumulator only ever
// covers 32 terms, its two small products first; the epilogue warps add these partial sums in fp32
// registers, rounding to nearest, as the FMA kernels do.
//
// Bound: shared memory.  A 128 x 128 x 8 instruction reads 8 KB of operands in its 64 cycles (the full
// 128 B/clk) and the split operands of a K block of 32 are another 64 KB of writes: about 1300 cycles per
// block against 768 of MMA, 400 FMA per cycle and SM, three times what the FMA pipe can do.  Operands are
// fetched by plain 4-byte loads (no alignment is known), always one half block ahead, and written as the
// no-swizzle K-major layout [4-term chunk][row][16 bytes]; the chunk pitch is 16 bytes more than the
// rows need, so that stores with lanes along K (one word per lane) hit 32 different banks.
//
// The MMA's rows are the index that is contiguous in Y (pixels, or columns of Gemm), its columns the other
// one (channels, or rows of Gemm): TMEM lanes then store consecutive addresses.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "common.h"
#include "tc_common.cuh"
#include "tc_host.h"

namespace onnxb {

namespace {

using namespace tc;

constexpr int kBK = 32, kStages = 3;
// 16 warps, so that a thread may hold 128 registers: the first epilogue warp issues the MMAs as well
constexpr int kProducerWarps = 8, kEpiWarps = 8, kMmaWarp = kProducerWarps;
constexpr int kThreads = (kProducerWarps + kEpiWarps) * 32;
constexpr uint32_t kChunkPitch = 128 * 16 + 16;             // one 4-term chunk of up to 128 rows
constexpr uint32_t kPart = (kBK / 4) * kChunkPitch;         // one operand's hi or lo block
constexpr uint32_t kStageBytes = 4 * kPart;                 // row hi, row lo, column hi, column lo
constexpr int kTabBytes = kProducerWarps * 16 * 16;         // per producer warp: 16 reduction terms' offsets
constexpr uint32_t kTmemCols = 256;                         // two accumulators
constexpr size_t kSmem = 128 + (size_t)kStages * kStageBytes + kTabBytes + 256;
static_assert(kSmem >= kSmemMoreTmem, "see smem_with_tmem");

struct Bars {
    uint64_t full[kStages], empty[kStages], acc_full[2], acc_empty[2];
    uint32_t tmem_holder;
};
static_assert(sizeof(Bars) <= 256, "barrier block too large");

enum { kKContig = 0, kMnContig = 1, kPixels = 2 };

struct Args {
    const float *R, *C;          // row operand, column operand
    float *Y;
    int rows, cols, K;           // per group for a convolution
    long long r_ld, c_ld;        // stride of the index that is not contiguous
    int BN, tiles_c, relu;
    long long tiles;
    // Gemm epilogue: alpha * D + beta * Cadd
    float alpha, beta;
    const float *Cadd;
    long long c_si, c_sj;
    // Conv
    const float *bias, *Radd;
    int Cch, H, W, PQ, Q, sh, sw, dh, dw, pt, pl, taps, kW, Mtot, tiles_r;
    ConvDivisor dv_PQ, dv_Q, dv_taps, dv_kW;
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

// hi to nearest; lo's rounding is completed by the tensor core, which ignores the low 13 bits.  A value that is
// not finite leaves lo = NaN, one that rounds to infinity lo = the opposite infinity, and either way every output it
// takes part in is NaN: the epilogue then sums that output from the operands themselves.  (Whatever a NaN x becomes in
// hi: x - hi is the NaN of GPU arithmetic, 0x7FFFFFFF, which half an ulp more would turn into a zero.  The larger of
// the two as signed integers keeps it, and is the sum for every other value; all 2^32 compared.  It costs 0.2 us of
// 86 on the dilated grouped 75x61 layer, a comparison and a selection for hi 2.1.)
__device__ __forceinline__ void split_tf32(float x, float &hi, float &lo) {
    hi = __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xFFFFE000u);
    int r;
    asm("{\n.reg .s32 t;\nadd.s32 t, %1, 0x1000;\nmax.s32 %0, t, %1;\n}" : "=r"(r) : "r"(__float_as_int(x - hi)));
    lo = __int_as_float(r);
}

// Where one tile's operands lie, for one producer thread.
struct Src {
    const float *p;              // k-contiguous: first row of this warp, + lane; else: this thread's row / column
    int left;                    // rows (columns) from there to the end of the operand
    uint32_t m_lo, m_hi;         // pixels: which filter taps lie inside the image
};

template <int MODE>
__device__ __forceinline__ void src_setup(const Args &g, bool rowop, int grp, int first, int warp, int lane, int tid, Src &s) {
    const float *base = rowop ? g.R : g.C;
    const long long ld = rowop ? g.r_ld : g.c_ld;
    const int n = rowop ? g.rows : g.cols;
    s.m_lo = s.m_hi = 0;
    if (MODE == kKContig) {
        s.p = base + (long long)(grp * (rowop ? 0 : g.cols) + first + warp) * ld + lane;
        s.left = n - first - warp;
    } else if (MODE == kMnContig) {
        s.p = base + first + (tid & 127);
        s.left = n - first - (tid & 127);
    } else {
        const int j = first + (tid & 127);
        s.left = n - j;
        const int jj = s.left > 0 ? j : 0;
        const int img = conv_fdiv(jj, g.PQ, g.dv_PQ), u = jj - img * g.PQ;
        const int p = conv_fdiv(u, g.Q, g.dv_Q), q = u - p * g.Q;
        const int h = p * g.sh - g.pt, w = q * g.sw - g.pl;
        s.p = base + (((long long)img * g.Cch + (long long)grp * (g.K / g.taps)) * g.H + h) * g.W + w;
        unsigned long long m = 0, cols = 0;
        for (int x = 0; x < g.kW; ++x) cols |= (unsigned long long)((unsigned)(w + x * g.dw) < (unsigned)g.W) << x;
        for (int y = 0; y * g.kW < g.taps; ++y)
            if ((unsigned)(h + y * g.dh) < (unsigned)g.H) m |= cols << (y * g.kW);
        if (s.left > 0) {                           // past the last pixel: every term is outside the image
            s.m_lo = (uint32_t)m;
            s.m_hi = (uint32_t)(m >> 32);
        }
    }
}

// Loads this thread's 16 values of K block kb (zeros outside the operand).
template <int MODE>
__device__ __forceinline__ void src_load(const Args &g, bool rowop, const Src &s, int kb, int width, int warp, int lane,
                                         int tid, int4 *tab, float (&v)[16]) {
    const long long ld = rowop ? g.r_ld : g.c_ld;
    const int k0 = kb * kBK;
    if (MODE == kKContig) {
        // lane = term, 16 rows 8 apart
        const bool kok = k0 + lane < g.K;
        const float *p = s.p + k0;
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            v[e] = kok && e * 8 < s.left && warp + e * 8 < width ? __ldg(p) : 0.f;
            p += 8 * ld;
        }
    } else if (MODE == kMnContig) {
        const int kh = k0 + (tid >> 7) * 16;
        const float *p = s.p + (long long)kh * ld;
        const bool ok = s.left > 0 && (tid & 127) < width;
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            v[e] = ok && kh + e < g.K ? __ldg(p) : 0.f;
            p += ld;
        }
    } else {
        // the warp's 16 terms: offset in X and the tap's bit (lanes 0-15 work them out; tc_fp32_conv_fits: 31 bits hold it)
        const int k = k0 + (tid >> 7) * 16 + (lane & 15);
        int4 t = make_int4(0, 0, 0, 0);
        if (k < g.K) {
            const int c = conv_fdiv(k, g.taps, g.dv_taps), rs = k - c * g.taps;
            const int r = conv_fdiv(rs, g.kW, g.dv_kW), q = rs - r * g.kW;
            t = make_int4(c * g.H * g.W + r * g.dh * g.W + q * g.dw, rs < 32 ? (int)(1u << rs) : 0,
                          rs < 32 ? 0 : (int)(1u << (rs - 32)), 0);
        }
        __syncwarp();
        if (lane < 16) tab[lane] = t;
        __syncwarp();
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            const int4 o = tab[e];
            v[e] = ((s.m_lo & (uint32_t)o.y) | (s.m_hi & (uint32_t)o.z)) ? __ldg(s.p + o.x) : 0.f;
        }
    }
}

template <int MODE>
__device__ __forceinline__ void src_store(uint8_t *hi, const float (&v)[16], int width, int warp, int lane, int tid) {
    if (MODE == kKContig) {
        uint8_t *d = hi + (uint32_t)(lane >> 2) * kChunkPitch + (uint32_t)warp * 16u + (uint32_t)(lane & 3) * 4u;
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            if (e * 8 < width) {
                float h, l;
                split_tf32(v[e], h, l);
                *reinterpret_cast<float *>(d + e * 128) = h;
                *reinterpret_cast<float *>(d + e * 128 + kPart) = l;
            }
        }
    } else {
        uint8_t *d = hi + (uint32_t)(tid >> 7) * 4u * kChunkPitch + (uint32_t)(tid & 127) * 16u;
        if ((tid & 127) < width) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float h[4], l[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) split_tf32(v[4 * c + e], h[e], l[e]);
                *reinterpret_cast<float4 *>(d + c * kChunkPitch) = make_float4(h[0], h[1], h[2], h[3]);
                *reinterpret_cast<float4 *>(d + c * kChunkPitch + kPart) = make_float4(l[0], l[1], l[2], l[3]);
            }
        }
    }
}

struct Tile {
    int grp, r0, c0;
};
__device__ __forceinline__ Tile tile_of(const Args &g, long long t) {
    // column tiles fastest: CTAs running at the same time share a row tile's operand in L2
    const int ct = (int)(t % g.tiles_c);
    const long long u = t / g.tiles_c;
    Tile r;
    r.grp = (int)(u / g.tiles_r);
    r.r0 = (int)(u % g.tiles_r) * 128;
    r.c0 = ct * g.BN;
    return r;
}

// One operand value of an output, for the scalar path of tiles whose values the split cannot carry.
template <int MODE>
__device__ float fetch(const Args &g, bool rowop, int grp, int idx, int k) {
    const float *base = rowop ? g.R : g.C;
    const long long ld = rowop ? g.r_ld : g.c_ld;
    if (MODE == kKContig) return __ldg(base + (long long)(grp * (rowop ? 0 : g.cols) + idx) * ld + k);
    if (MODE == kMnContig) return __ldg(base + (long long)k * ld + idx);
    const int img = idx / g.PQ, u = idx - img * g.PQ, p = u / g.Q, q = u - p * g.Q;
    const int c = k / g.taps, rs = k - c * g.taps, r = rs / g.kW, s = rs - r * g.kW;
    const int h = p * g.sh - g.pt + r * g.dh, w = q * g.sw - g.pl + s * g.dw;
    if ((unsigned)h >= (unsigned)g.H || (unsigned)w >= (unsigned)g.W) return 0.f;
    return __ldg(base + (((long long)img * g.Cch + (long long)grp * (g.K / g.taps) + c) * g.H + h) * g.W + w);
}

template <int RM, int CM>
__global__ void __launch_bounds__(kThreads, 1)
tc_fp32_kernel(const __grid_constant__ Args g, unsigned int *err) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *stages = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    int4 *tabs = reinterpret_cast<int4 *>(stages + (size_t)kStages * kStageBytes);
    Bars *bars = reinterpret_cast<Bars *>(reinterpret_cast<uint8_t *>(tabs) + kTabBytes);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nkb = (g.K + kBK - 1) / kBK;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&bars->full[s], kProducerWarps);
            mbar_init(&bars->empty[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(&bars->acc_full[s], 1);
            mbar_init(&bars->acc_empty[s], kEpiWarps);
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

    if (warp < kProducerWarps) {
        // ------------------------------------------------------------ operand producers
        const int tid = threadIdx.x;
        int4 *tab = tabs + warp * 16;
        float vr[16], vc[16];
        Src sr, sc;
        long long t = blockIdx.x;
        if (t < g.tiles) {
            pdl_wait();
            Tile tl = tile_of(g, t);
            src_setup<RM>(g, true, tl.grp, tl.r0, warp, lane, tid, sr);
            src_setup<CM>(g, false, tl.grp, tl.c0, warp, lane, tid, sc);
            src_load<RM>(g, true, sr, 0, 128, warp, lane, tid, tab, vr);
            src_load<CM>(g, false, sc, 0, g.BN, warp, lane, tid, tab, vc);
            int st = 0, kb = 0;
            uint32_t phase = 0;
            while (true) {
                // what comes after this block: the tile's next block, or the next tile's first
                int nkb_i = kb + 1;
                long long nt = t;
                if (nkb_i == nkb) {
                    nkb_i = 0;
                    nt += gridDim.x;
                    if (nt < g.tiles) {
                        tl = tile_of(g, nt);
                        src_setup<RM>(g, true, tl.grp, tl.r0, warp, lane, tid, sr);
                        src_setup<CM>(g, false, tl.grp, tl.c0, warp, lane, tid, sc);
                    }
                }
                uint8_t *sp = stages + (size_t)st * kStageBytes;
                mbar_wait(&bars->empty[st], phase ^ 1u, err, 40);
                src_store<RM>(sp, vr, 128, warp, lane, tid);
                if (nt < g.tiles) src_load<RM>(g, true, sr, nkb_i, 128, warp, lane, tid, tab, vr);
                src_store<CM>(sp + 2 * kPart, vc, g.BN, warp, lane, tid);
                if (nt < g.tiles) src_load<CM>(g, false, sc, nkb_i, g.BN, warp, lane, tid, tab, vc);
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars->full[st]);
                if (++st == kStages) { st = 0; phase ^= 1u; }
                if (nkb_i == 0 && nt >= g.tiles) break;
                t = nt;
                kb = nkb_i;
            }
        }
    } else {
        // ------------------------------------------------------------ partial sums and epilogue
        const int quarter = warp & 3, half = (warp - kProducerWarps) >> 2;
        const int chunks = (g.BN + 15) / 16;                        // 16-column chunks of the tile
        const int c_lo = half ? (chunks + 1) / 2 : 0, nch = half ? chunks / 2 : (chunks + 1) / 2;
        // MMAs of one K block, issued by one thread of the first epilogue warp, a block ahead of the sums
        const long long my_tiles = blockIdx.x < g.tiles ? (g.tiles - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
        const long long n_blk = my_tiles * nkb;
        const bool issuer = warp == kMmaWarp && elect_one();
        const uint32_t desc_hi = (128u >> 4) | (1u << 14);
        const uint32_t a0 = ((smem_u32(stages) >> 4) & 0x3FFFu) | ((kChunkPitch >> 4) << 16);
        const uint32_t idesc = make_idesc_tf32(128, g.BN, 0, 0);
        int st = 0;
        uint32_t phase = 0;
        auto issue = [&](uint32_t blk) {
            if (issuer) {
                const uint32_t ab = blk & 1u;
                mbar_wait(&bars->acc_empty[ab], ((blk >> 1) & 1u) ^ 1u, err, 41);
                mbar_wait(&bars->full[st], phase, err, 42);
                tc_fence_after_sync();
                const uint32_t d = tmem_base + ab * 128u;
                const uint32_t a = a0 + (uint32_t)st * (kStageBytes >> 4);
                const uint32_t part = kPart >> 4, two = 2u * kChunkPitch >> 4;
#pragma unroll
                for (int j = 0; j < kBK / 8; ++j) {
                    // the two small products first, while the accumulator is small
                    const uint32_t o = a + (uint32_t)j * two;
                    mma_tf32_lohi(d, o + part, desc_hi, o + 2 * part, desc_hi, idesc, j > 0);
                    mma_tf32_lohi(d, o, desc_hi, o + 3 * part, desc_hi, idesc, 1);
                }
#pragma unroll
                for (int j = 0; j < kBK / 8; ++j) {
                    const uint32_t o = a + (uint32_t)j * two;
                    mma_tf32_lohi(d, o, desc_hi, o + 2 * part, desc_hi, idesc, 1);
                }
                mma_commit(&bars->empty[st]);
                mma_commit(&bars->acc_full[ab]);
                if (++st == kStages) { st = 0; phase ^= 1u; }
            }
            __syncwarp();
        };
        if (warp == kMmaWarp && n_blk > 0) issue(0);
        uint32_t blk = 0, tile_it = 0;
        for (long long t = blockIdx.x; t < g.tiles; t += gridDim.x, ++tile_it) {
            const Tile tl = tile_of(g, t);
            float acc[64];
#pragma unroll
            for (int e = 0; e < 64; ++e) acc[e] = 0.f;
            for (int kb = 0; kb < nkb; ++kb, ++blk) {
                if (warp == kMmaWarp && (long long)blk + 1 < n_blk) issue(blk + 1);
                const uint32_t ab = blk & 1u;
                mbar_wait(&bars->acc_full[ab], (blk >> 1) & 1u, err, 43);
                tc_fence_after_sync();
                const uint32_t ta = tmem_base + ab * 128u + ((uint32_t)(quarter * 32) << 16) + (uint32_t)c_lo * 16u;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    if (c < nch) {
                        uint32_t v[16];
                        tmem_ld_32x16(ta + c * 16u, v);
                        tmem_ld_wait();
#pragma unroll
                        for (int e = 0; e < 16; ++e) acc[c * 16 + e] += __uint_as_float(v[e]);
                    }
                }
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars->acc_empty[ab]);
            }
            if (tile_it == 0) pdl_wait();       // long since satisfied: the producers passed theirs before the first load
            const int j = tl.r0 + quarter * 32 + lane;
            const bool rowok = j < g.rows;
            const int cc0 = tl.c0 + c_lo * 16;                      // first column (within the group) of this warp
            const int ncol = min(g.cols - cc0, nch * 16);
            bool bad = false;
            long long ybase, ystep;
            if (RM == kPixels) {
                const int jj = rowok ? j : 0, img = conv_fdiv(jj, g.PQ, g.dv_PQ);
                ybase = ((long long)img * g.Mtot + (long long)tl.grp * g.cols) * g.PQ + (jj - img * g.PQ);
                ystep = g.PQ;
            } else {
                ybase = j;
                ystep = g.rows;
            }
            auto finish = [&](float d, int i, float add, float r) {
                float v = RM == kPixels ? (d + add) + r : fmaf(g.alpha, d, add);
                if (g.relu) v = v > 0.f ? v : 0.f;
                g.Y[ybase + (long long)i * ystep] = v;
            };
            auto addend = [&](int i, float &add, float &r) {
                add = r = 0.f;
                if (RM == kPixels) {
                    if (g.bias) add = __ldg(g.bias + tl.grp * g.cols + i);
                    if (g.Radd) r = __ldg(g.Radd + ybase + (long long)i * ystep);
                } else if (g.Cadd) {
                    add = g.beta * __ldg(g.Cadd + i * g.c_si + j * g.c_sj);
                }
            };
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                float add[8], r[8];
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    if (rowok && c * 8 + e < ncol) addend(cc0 + c * 8 + e, add[e], r[e]);
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    if (rowok && c * 8 + e < ncol) {
                        bad |= acc[c * 8 + e] != acc[c * 8 + e];
                        finish(acc[c * 8 + e], cc0 + c * 8 + e, add[e], r[e]);
                    }
            }
            if (bad) {      // an operand the split cannot carry (see split_tf32): this row again, term by term
                for (int c = 0; c < ncol; ++c) {
                    float d = 0.f, add, r;
                    for (int k = 0; k < g.K; ++k)
                        d = fmaf(fetch<CM>(g, false, tl.grp, cc0 + c, k), fetch<RM>(g, true, tl.grp, j, k), d);
                    addend(cc0 + c, add, r);
                    finish(d, cc0 + c, add, r);
                }
            }
        }
    }

    tc_fence_before_sync();
    __syncthreads();
    if (warp == kMmaWarp) {
        __syncwarp();
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, kTmemCols);
    }
}

// Tile width with the shortest estimated time (cycles, fitted to measurements from 0.4 to 14 GFLOP): rounds
// of 148 tiles x (K blocks of 1800 to 3100 cycles, more for pixels, whose loads need more work; and the
// tile's own start and epilogue).  Within 4 % of 34 measured problems on average.
struct Pick {
    int bn;
    double cost;
};
Pick pick_width(long long rows, int cols, int K, int groups, bool pixels) {
    Pick best{0, 0};
    for (int bn = 16; bn <= 128 && bn <= (cols + 15) / 16 * 16; bn += 16) {
        const long long tiles = (rows + 127) / 128 * ((cols + bn - 1) / bn) * groups;
        const double rounds = (double)((tiles + 147) / 148);
        const double blk = pixels ? 2120.0 + 8.0 * bn : 1750.0 + 5.0 * bn;
        const double cost = rounds * ((K + kBK - 1) / kBK * blk + 12000.0) + 4500.0;
        if (best.bn == 0 || cost < best.cost) best = {bn, cost};
    }
    return best;
}

template <int RM, int CM>
int launch(Args &a, int groups, cudaStream_t st) {
    unsigned int *err = device_status_ptr();
    if (!err) return (int)cudaErrorUnknown;
    a.tiles_r = (a.rows + 127) / 128;
    const int sms = tc_host::num_sms();
    a.BN = pick_width(a.rows, a.cols, a.K, groups, RM == kPixels).bn;
    a.tiles_c = (a.cols + a.BN - 1) / a.BN;
    a.tiles = (long long)a.tiles_r * a.tiles_c * groups;
    auto kern = tc_fp32_kernel<RM, CM>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
    if (e != cudaSuccess) return (int)e;
    const cudaError_t le = tc_host::launch_pdl(kern, dim3((unsigned)std::min<long long>(a.tiles, sms)), dim3(kThreads), kSmem,
                                               st, a, err);
    count_launch();
    return (int)le;
}

}  // namespace

double tc_fp32_cost(long long rows, int cols, int K, int groups, bool pixels) {
    return pick_width(rows, cols, K, groups, pixels).cost;
}

int launch_tc_fp32_gemm(const GemmProblem &p, const float *A, const float *B, const float *C, float *Y, void *stream) {
    Args a{};
    a.R = B; a.C = A; a.Y = Y; a.rows = p.N; a.cols = p.M; a.K = p.K;
    a.r_ld = p.transB ? p.K : p.N;
    a.c_ld = p.transA ? p.M : p.K;
    a.alpha = p.alpha; a.beta = p.beta; a.Cadd = C; a.c_si = p.c_stride_i; a.c_sj = p.c_stride_j; a.relu = p.relu;
    cudaStream_t st = (cudaStream_t)stream;
    if (p.transB) return p.transA ? launch<kKContig, kMnContig>(a, 1, st) : launch<kKContig, kKContig>(a, 1, st);
    return p.transA ? launch<kMnContig, kMnContig>(a, 1, st) : launch<kMnContig, kKContig>(a, 1, st);
}

// At most 64 taps (a bit each), and offsets of a window's terms from its start that are 32-bit integers: beyond, and only where
// the image is mostly padding, a dilated row of taps lies 2^31 elements and more further on.  (Sums modulo 2^32 as in
// the FMA kernel take an addition more per load: 86.3 -> 87.3 us on the dilated grouped 75x61 layer.)
bool tc_fp32_conv_fits(const ConvGeom &g) {
    const long long last = (g.Cg - 1LL) * g.H * g.W + (g.kH - 1LL) * g.dh * g.W + (g.kW - 1LL) * g.dw;
    return g.kH * g.kW <= 64 && last <= 2147483647LL;
}

int launch_tc_fp32_conv(const ConvGeom &g, const float *X, const float *W, const float *B, const float *R, float *Y,
                        void *stream) {
    Args a{};
    a.R = X; a.C = W; a.Y = Y; a.rows = g.N * g.P * g.Q; a.cols = g.Mg; a.K = g.Cg * g.kH * g.kW;
    a.c_ld = a.K;
    a.bias = B; a.Radd = R; a.relu = g.relu;
    a.Cch = g.C; a.H = g.H; a.W = g.W; a.PQ = g.P * g.Q; a.Q = g.Q;
    a.sh = g.sh; a.sw = g.sw; a.dh = g.dh; a.dw = g.dw; a.pt = g.pt; a.pl = g.pl;
    a.taps = g.kH * g.kW; a.kW = g.kW; a.Mtot = g.M;
    a.dv_PQ = conv_divisor(a.PQ); a.dv_Q = conv_divisor(a.Q); a.dv_taps = conv_divisor(a.taps); a.dv_kW = conv_divisor(a.kW);
    return launch<kPixels, kKContig>(a, g.group, (cudaStream_t)stream);
}

}  // namespace onnxb
