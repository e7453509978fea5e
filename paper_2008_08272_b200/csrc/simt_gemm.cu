// fp32 (FMA) tiled contraction: ONNX Gemm (Sec. 3.4.3) and ONNX Conv (Sec. 4.1) for the problems
// that stay in fp32: contractions too thin for the tensor cores, or operands TMA cannot describe (rows
// that are no multiples of 16 bytes, images of odd size).
//
// One kernel serves both operators as D (M x N) = A (M x K) * B (K x N):
//   Gemm  A', B' in any of the four storage orders;
//   Conv  A = the filters W[m][k] (k = (c*kH + r)*kW + s, exactly ONNX's layout), B = the pixels, column
//         j = (image, p, q), whose row k is fetched from X through a small table of the K block's
//         (channel, tap) offsets: the unfolded matrix is never formed.
//
// Bound: the FMA pipe (148 SMs x 128 FMA x 1.965 GHz = 74.4 TFLOP/s).  What it takes to get near it:
// packed fma.rn.f32x2 (two FMAs per issue slot, so the operand reads and address work fit beside them), 8x8
// or 8x4 outputs per thread, operands staged by cp.async (4 bytes: rows have no alignment) three K blocks
// deep, and the reduction split over a cluster's CTAs where the tiles alone leave SMs idle (partial tiles
// are summed through distributed shared memory in rank order, so the result does not depend on timing).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>
#include <cstdlib>

#include "common.h"
#include "tc_common.cuh"
#include "tc_host.h"

namespace onnxb {

namespace {

constexpr int kBK = 16;        // reduction terms per stage
constexpr int kStages = 3;

enum { kKContig = 0, kMnContig = 1, kPixels = 2 };

struct SgemmArgs {
    const float *A, *B;
    float *Y;
    int M, N, K;                       // per group for a convolution
    long long a_ld, b_ld;              // stride of the non-contiguous index
    int tiles_m, tiles_n, relu;
    // Gemm epilogue: alpha * D + beta * C
    float alpha, beta;
    const float *C;
    long long c_si, c_sj;
    // Conv
    const float *bias, *R;
    int Cch, H, W, PQ, Q, sh, sw, dh, dw, pt, pl, taps, kW, Mtot;
    ConvDivisor dv_PQ, dv_Q, dv_taps, dv_kW;
};

__device__ __forceinline__ void cp_async4(uint32_t dst, const float *src, bool live) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(live ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void fma2(unsigned long long &d, unsigned long long a, unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long dup2(float a) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
    return r;
}
__device__ __forceinline__ float ld_dsmem(uint32_t addr) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}

template <int BM, int BN>
__host__ __device__ constexpr size_t sgemm_smem() {
    const size_t ring = (size_t)kStages * kBK * (BM + 4 + BN + 4) * 4, out = (size_t)BM * (BN + 4) * 4;
    return (ring > out ? ring : out) + (kStages + 1) * kBK * 16;
}

// Threads form (BM/TM) x (BN/TN); a warp covers 4 x 8 of them.  A thread's rows are tm*4 + {0..3} and, for
// TM = 8, the same in the tile's lower half (likewise its columns), so that every fragment read is a 16-byte
// shared-memory load whose lanes touch consecutive pieces.
template <int BM, int BN, int TM, int TN, int AM, int BMODE>
__global__ void __launch_bounds__((BM / TM) * (BN / TN), (BM / TM) * (BN / TN) == 256 ? 2 : 4)
sgemm_kernel(const __grid_constant__ SgemmArgs g, int split) {
    constexpr int NT_M = BM / TM, NT_N = BN / TN, NTHR = NT_M * NT_N;
    constexpr int PA = BM + 4, PB = BN + 4;
    constexpr int WARPS_N = NT_N / 8;
    extern __shared__ __align__(16) float sm[];
    float *As = sm, *Bs = sm + kStages * kBK * PA;
    int4 *ktab = reinterpret_cast<int4 *>(reinterpret_cast<uint8_t *>(sm) + sgemm_smem<BM, BN>() - (kStages + 1) * kBK * 16);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = (int)(blockIdx.x % (unsigned)split);
    unsigned tile = blockIdx.x / (unsigned)split;
    const int tile_m = (int)(tile % (unsigned)g.tiles_m);
    tile /= (unsigned)g.tiles_m;
    const int tile_n = (int)(tile % (unsigned)g.tiles_n), grp = (int)(tile / (unsigned)g.tiles_n);
    const int i0 = tile_m * BM, j0 = tile_n * BN;
    const int ktiles = (g.K + kBK - 1) / kBK;
    const int kt_per = (ktiles + split - 1) / split;
    const int kt_lo = rank * kt_per, kt_hi = min(ktiles, kt_lo + kt_per);

    // ---- what this thread loads
    constexpr int A_ROWS_STEP = NTHR / kBK, A_N = BM / A_ROWS_STEP;          // k-contiguous: lanes along k
    constexpr int A_KSTEP = NTHR / BM > 0 ? NTHR / BM : 1;                    // m-contiguous: lanes along m
    constexpr int A_MREP = NTHR >= BM ? 1 : BM / NTHR;
    constexpr int B_ROWS_STEP = NTHR / kBK, B_N = BN / B_ROWS_STEP;
    constexpr int B_KSTEP = NTHR / BN > 0 ? NTHR / BN : 1;
    constexpr int B_NREP = NTHR >= BN ? 1 : BN / NTHR;
    const float *Ag = g.A + (BMODE == kPixels ? (long long)grp * g.M * g.K : 0);
    const uint32_t as_u32 = tc::smem_u32(As), bs_u32 = tc::smem_u32(Bs);

    // pixel columns of a convolution: where the column's window starts in X.  This offset and those of the table below
    // are summed modulo 2^32: under a dilation of 2^19 either may lie billions of elements outside X, but the sum, used
    // only for taps inside the image, is an element of X, and X has fewer than 2^31.
    unsigned px_base[B_NREP];
    int px_h[B_NREP], px_w[B_NREP];
    if (BMODE == kPixels) {
#pragma unroll
        for (int e = 0; e < B_NREP; ++e) {
            const int j = j0 + tid % BN + e * NTHR;
            if (j < g.N) {
                const int n = conv_fdiv(j, g.PQ, g.dv_PQ), u = j - n * g.PQ;
                const int p = conv_fdiv(u, g.Q, g.dv_Q), q = u - p * g.Q;
                px_h[e] = p * g.sh - g.pt;
                px_w[e] = q * g.sw - g.pl;
                px_base[e] = (unsigned)(n * g.Cch + grp * (g.K / g.taps)) * (unsigned)(g.H * g.W) + (unsigned)px_h[e] * (unsigned)g.W +
                             (unsigned)px_w[e];
            } else {
                px_h[e] = px_w[e] = -(1 << 30);
                px_base[e] = 0;
            }
        }
    }
    // offsets of one K block's rows: {offset in X, r*dh, s*dw}; rows past K point far outside the image
    auto write_ktab = [&](int kt) {
        if (BMODE == kPixels && tid < kBK) {
            const int k = kt * kBK + tid;
            int4 e = make_int4(0, -(1 << 30), -(1 << 30), 0);
            if (k < g.K) {
                const int c = conv_fdiv(k, g.taps, g.dv_taps), rs = k - c * g.taps;
                const int r = conv_fdiv(rs, g.kW, g.dv_kW), s = rs - r * g.kW;
                const unsigned rh = (unsigned)(r * g.dh), sw = (unsigned)(s * g.dw);
                e = make_int4((int)((unsigned)(c * g.H * g.W) + rh * (unsigned)g.W + sw), (int)rh, (int)sw, 0);
            }
            ktab[(kt % (kStages + 1)) * kBK + tid] = e;
        }
    };
    auto load_tile = [&](int kt, int st) {
        const int k0 = kt * kBK;
        if (AM == kKContig) {
            const int kk = tid % kBK, r0 = tid / kBK;
            const bool kok = k0 + kk < g.K;
            const float *src = Ag + (long long)(i0 + r0) * g.a_ld + k0 + kk;
            uint32_t dst = as_u32 + (uint32_t)((st * kBK + kk) * PA + r0) * 4u;
#pragma unroll
            for (int e = 0; e < A_N; ++e) {
                const bool ok = kok && i0 + r0 + e * A_ROWS_STEP < g.M;
                cp_async4(dst, ok ? src : g.A, ok);
                src += (long long)A_ROWS_STEP * g.a_ld;
                dst += A_ROWS_STEP * 4u;
            }
        } else {
#pragma unroll
            for (int e = 0; e < A_MREP; ++e) {
                const int ii = tid % BM + e * NTHR, kk0 = NTHR >= BM ? tid / BM : 0;
                const bool iok = i0 + ii < g.M;
                const float *src = Ag + (long long)(k0 + kk0) * g.a_ld + i0 + ii;
                uint32_t dst = as_u32 + (uint32_t)((st * kBK + kk0) * PA + ii) * 4u;
#pragma unroll
                for (int kk = 0; kk < kBK; kk += A_KSTEP) {
                    const bool ok = iok && k0 + kk0 + kk < g.K;
                    cp_async4(dst, ok ? src : g.A, ok);
                    src += (long long)A_KSTEP * g.a_ld;
                    dst += A_KSTEP * PA * 4u;
                }
            }
        }
        if (BMODE == kKContig) {
            const int kk = tid % kBK, r0 = tid / kBK;
            const bool kok = k0 + kk < g.K;
            const float *src = g.B + (long long)(j0 + r0) * g.b_ld + k0 + kk;
            uint32_t dst = bs_u32 + (uint32_t)((st * kBK + kk) * PB + r0) * 4u;
#pragma unroll
            for (int e = 0; e < B_N; ++e) {
                const bool ok = kok && j0 + r0 + e * B_ROWS_STEP < g.N;
                cp_async4(dst, ok ? src : g.B, ok);
                src += (long long)B_ROWS_STEP * g.b_ld;
                dst += B_ROWS_STEP * 4u;
            }
        } else {
            const int4 *tab = ktab + (kt % (kStages + 1)) * kBK;
#pragma unroll
            for (int e = 0; e < B_NREP; ++e) {
                const int jj = tid % BN + e * NTHR, kk0 = NTHR >= BN ? tid / BN : 0;
                uint32_t dst = bs_u32 + (uint32_t)((st * kBK + kk0) * PB + jj) * 4u;
                if (BMODE == kMnContig) {
                    const bool jok = j0 + jj < g.N;
                    const float *src = g.B + (long long)(k0 + kk0) * g.b_ld + j0 + jj;
#pragma unroll
                    for (int kk = 0; kk < kBK; kk += B_KSTEP) {
                        const bool ok = jok && k0 + kk0 + kk < g.K;
                        cp_async4(dst, ok ? src : g.B, ok);
                        src += (long long)B_KSTEP * g.b_ld;
                        dst += B_KSTEP * PB * 4u;
                    }
                } else {
#pragma unroll
                    for (int kk = 0; kk < kBK; kk += B_KSTEP) {
                        const int4 t = tab[kk0 + kk];
                        const bool ok = (unsigned)(px_h[e] + t.y) < (unsigned)g.H && (unsigned)(px_w[e] + t.z) < (unsigned)g.W;
                        cp_async4(dst, ok ? g.B + (px_base[e] + (unsigned)t.x) : g.B, ok);
                        dst += B_KSTEP * PB * 4u;
                    }
                }
            }
        }
    };

    // ---- main loop
    const int wm = warp / WARPS_N, wn = warp % WARPS_N;
    const int tm = wm * 4 + ((lane & 1) | ((lane >> 4) << 1)), tn = wn * 8 + ((lane >> 1) & 7);
    unsigned long long acc[TM][TN / 2];
#pragma unroll
    for (int a = 0; a < TM; ++a)
#pragma unroll
        for (int b = 0; b < TN / 2; ++b) acc[a][b] = 0ull;

    tc::pdl_launch_dependents();
    tc::pdl_wait();
    if (BMODE == kPixels) {
        for (int s = 0; s < kStages; ++s) write_ktab(kt_lo + s);
        __syncthreads();
    }
#pragma unroll
    for (int s = 0; s < kStages - 1; ++s) {
        if (kt_lo + s < kt_hi) load_tile(kt_lo + s, s);
        cp_async_commit();
    }
    int st = 0;
    for (int kt = kt_lo; kt < kt_hi; ++kt) {
        cp_async_wait<kStages - 2>();
        __syncthreads();
        {
            const int nk = kt + kStages - 1;
            if (nk < kt_hi) load_tile(nk, st == 0 ? kStages - 1 : st - 1);
            cp_async_commit();
            write_ktab(kt + kStages);
        }
        const float *as = As + st * kBK * PA + tm * 4, *bs = Bs + st * kBK * PB + tn * 4;
#pragma unroll
        for (int kk = 0; kk < kBK; ++kk) {
            float av[TM];
            unsigned long long bv[TN / 2];
#pragma unroll
            for (int h = 0; h < TM / 4; ++h) {
                const float4 t = *reinterpret_cast<const float4 *>(as + kk * PA + h * (BM / 2));
                av[4 * h] = t.x; av[4 * h + 1] = t.y; av[4 * h + 2] = t.z; av[4 * h + 3] = t.w;
            }
#pragma unroll
            for (int h = 0; h < TN / 4; ++h) {
                const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(bs + kk * PB + h * (BN / 2));
                bv[2 * h] = t.x; bv[2 * h + 1] = t.y;
            }
#pragma unroll
            for (int a = 0; a < TM; ++a) {
                const unsigned long long aa = dup2(av[a]);
#pragma unroll
                for (int b = 0; b < TN / 2; ++b) fma2(acc[a][b], aa, bv[b]);
            }
        }
        if (++st == kStages) st = 0;
    }

    // ---- epilogue: the tile goes through shared memory so that lanes store consecutive columns; with a
    // split reduction every CTA of the cluster sums its share of the rows over all partial tiles
    cp_async_wait<0>();
    __syncthreads();
#pragma unroll
    for (int a = 0; a < TM; ++a) {
        const int row = (a / 4) * (BM / 2) + tm * 4 + a % 4;
#pragma unroll
        for (int h = 0; h < TN / 4; ++h)
            *reinterpret_cast<ulonglong2 *>(sm + row * PB + h * (BN / 2) + tn * 4) = make_ulonglong2(acc[a][2 * h], acc[a][2 * h + 1]);
    }
    if (split > 1) tc::cluster_sync_all();
    else __syncthreads();

    constexpr int CPT = NTHR >= BN ? 1 : BN / NTHR;                // columns per thread
    constexpr int RSTEP = NTHR >= BN ? NTHR / BN : 1;
    constexpr int UR = 8;                                          // rows in flight per thread (addend loads overlap)
    const int rows = (BM + split - 1) / split, r_lo = rank * rows, r_hi = min(min(BM, r_lo + rows), g.M - i0);
    const uint32_t sm_u32 = tc::smem_u32(sm);
#pragma unroll
    for (int e = 0; e < CPT; ++e) {
        const int jj = tid % BN + e * NTHR, j = j0 + jj;
        if (j >= g.N) continue;
        long long ybase, ystep;
        if (BMODE == kPixels) {
            const int n = conv_fdiv(j, g.PQ, g.dv_PQ);
            ybase = ((long long)n * g.Mtot + (long long)grp * g.M) * g.PQ + (j - n * g.PQ);
            ystep = g.PQ;
        } else {
            ybase = j;
            ystep = g.N;
        }
        for (int r0 = r_lo + (NTHR >= BN ? tid / BN : 0); r0 < r_hi; r0 += RSTEP * UR) {
            float add[UR], v[UR];
#pragma unroll
            for (int u = 0; u < UR; ++u) {
                const int r = r0 + u * RSTEP, i = i0 + r;
                add[u] = v[u] = 0.f;
                if (r < r_hi) {
                    if (BMODE == kPixels) {
                        if (g.bias) add[u] = __ldg(g.bias + grp * g.M + i);
                        if (g.R) v[u] = __ldg(g.R + ybase + (long long)i * ystep);
                    } else if (g.C) {
                        add[u] = g.beta * __ldg(g.C + i * g.c_si + j * g.c_sj);
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < UR; ++u) {
                const int r = r0 + u * RSTEP;
                if (r < r_hi) {
                    float d = 0.f;
                    if (split == 1) {
                        d = sm[r * PB + jj];
                    } else {
                        for (int s = 0; s < split; ++s)
                            d += ld_dsmem(tc::map_to_cta(sm_u32 + (uint32_t)(r * PB + jj) * 4u, (uint32_t)s));
                    }
                    d = BMODE == kPixels ? (d + add[u]) + v[u] : fmaf(g.alpha, d, add[u]);
                    if (g.relu) d = d > 0.f ? d : 0.f;
                    g.Y[ybase + (long long)(i0 + r) * ystep] = d;
                }
            }
        }
    }
    if (split > 1) tc::cluster_sync_all();      // no CTA leaves while a peer still reads its partial tile
}

// ------------------------------------------------------------------ tiny Gemms: one warp per output
// A few hundred to a few thousand dot products (a 10-class head behind a small network): everything is
// latency, so no staging and no barrier; lanes split the reduction, a shuffle tree joins it.
template <int AM, int BMODE>
__global__ void __launch_bounds__(128)
gemm_dot_kernel(const __grid_constant__ SgemmArgs g) {
    tc::pdl_launch_dependents();
    const int warp = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (warp >= g.M * g.N) return;
    const int i = warp / g.N, j = warp - i * g.N;
    const float *a = g.A + (AM == kKContig ? i * g.a_ld : i), *b = g.B + (BMODE == kKContig ? j * g.b_ld : j);
    const long long as = AM == kKContig ? 1 : g.a_ld, bs = BMODE == kKContig ? 1 : g.b_ld;
    tc::pdl_wait();
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    int k = lane;
    for (; k + 224 < g.K; k += 256) {           // eight loads of each operand in flight
        float x[8], y[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) { x[u] = __ldg(a + (k + 32 * u) * as); y[u] = __ldg(b + (k + 32 * u) * bs); }
#pragma unroll
        for (int u = 0; u < 8; ++u) s[u & 3] = fmaf(x[u], y[u], s[u & 3]);
    }
    for (; k < g.K; k += 32) s[0] = fmaf(__ldg(a + k * as), __ldg(b + k * bs), s[0]);
    float v = (s[0] + s[1]) + (s[2] + s[3]);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    if (lane == 0) {
        v *= g.alpha;
        if (g.C) v = fmaf(g.beta, __ldg(g.C + i * g.c_si + j * g.c_sj), v);
        if (g.relu) v = v > 0.f ? v : 0.f;
        g.Y[(long long)i * g.N + j] = v;
    }
}

// ------------------------------------------------------------------ host side
struct Shape {
    int bm, bn, threads;
    double eff;                // measured share of the FMA pipe with the SMs full (Gemm; 0.63 of it for pixels)
};
constexpr int kShapes = 5;
constexpr Shape kShape[kShapes] = {{128, 128, 256, 0.73}, {64, 128, 128, 0.68}, {64, 64, 128, 0.59}, {16, 128, 128, 0.45},
                                   {32, 32, 64, 0.50}};

template <int AM, int BMODE, int I, int BM, int BN, int TM, int TN>
cudaError_t launch_shape(const SgemmArgs &a, int split, long long tiles, cudaStream_t st) {
    static_assert(kShape[I].bm == BM && kShape[I].bn == BN && kShape[I].threads == (BM / TM) * (BN / TN), "shape table");
    // Blocks placed while the previous kernel still holds its SMs crowd on those that happen to have room: so much shared memory is
    // asked for that no SM takes more than its share (clusters, which do not fit every GPC, one more).  From a graph Gemm 157 x 225 x 786
    // 10.5 -> 8.6 us, 541 x 87 x 705 10.3 -> 6.7, 1001 x 130 x 333 13.8 -> 12.1; 12 -> 40 channels 3x3 33x31 at batch 3 10.6 -> 9.2; the one
    // of 60 that lost, 885 x 63 x 115, 4.6 -> 4.8.  From 148 blocks on in place of 100: 355 x 49 x 571 10.0 us for 6.9; from the first on
    // seven of 60 are 4 to 6 % shorter; to 8 per SM no difference; two more for clusters: 649 x 103 x 227 8.9 for 6.6.  Two streams with a
    // Gemm each: 157 x 225 x 786 14.1 -> 11.8, 301 x 403 x 131 8.6 -> 9.3.
    size_t smem = sgemm_smem<BM, BN>();
    const long long ctas = tiles * split, sms = tc_host::num_sms(), share = (ctas + sms - 1) / sms + (split > 1 ? 1 : 0);
    if (ctas > 100 && share <= 4) smem = std::max(smem, smem_for_share(share));
    auto kern = sgemm_kernel<BM, BN, TM, TN, AM, BMODE>;
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e != cudaSuccess) return e;
    }
    const dim3 grid((unsigned)(tiles * split)), block(kShape[I].threads);
    return split > 1 ? tc_host::launch_pdl_cluster(kern, (unsigned)split, grid, block, smem, st, a, split)
                     : tc_host::launch_pdl(kern, grid, block, smem, st, a, split);
}

// Tile and split: the shortest estimated time, in cycles, fitted to a sweep of every shape and split over 34
// problems from 0.2 MFLOP to 14 GFLOP (the pick is within 6 % of the best on average).  An SM shares its FMA
// pipe among its CTAs, so what counts is the work of the fullest SM over the rate its resident warps reach; a
// CTA's start and epilogue come on top, a launch costs 7200 and a cluster's reduction 2000 more.
struct Pick {
    int shape, split;
    double cost;
};
Pick search_shape(int M, int N, int K, int groups, bool pixels) {
    Pick best{-1, 1, 0};
    const long long ktiles = (K + kBK - 1) / kBK;
    int ps = -1, pk = 1;       // ONNXB_FP32 = "shape,split" pins both
    if (const char *pin = getenv("ONNXB_FP32"))
        if (sscanf(pin, "%d,%d", &ps, &pk) != 2) ps = -1;
    for (int s = 0; s < kShapes; ++s) {
        const Shape &h = kShape[s];
        const long long tiles = (long long)((M + h.bm - 1) / h.bm) * ((N + h.bn - 1) / h.bn) * groups;
        for (int split = 1; split <= 8; ++split) {
            if (ps >= 0 && (s != ps || split != pk)) continue;
            if (split > 1 && ktiles < split && ps < 0) break;
            const long long ctas = tiles * split;
            if (ctas > 2147483647LL) continue;
            const long long per_sm = (ctas + 147) / 148;
            const double kt = (double)((ktiles + split - 1) / split);
            const double warps = std::min((double)per_sm * (h.threads / 32), 16.0);
            const double eff = h.eff * (pixels ? 0.63 : 1.0) * std::min(1.0, 0.28 + 0.72 * warps / 14.0);
            const double busy = (double)per_sm * h.bm * h.bn * kt * kBK / (128.0 * eff);
            const double each = (double)per_sm * (400.0 + h.bm * h.bn / 3.7 + (split > 1 ? 260.0 : 0.0));
            const double cost = std::max(busy, kt * 230.0) + each + 7200.0 + (split > 1 ? 2000.0 : 0.0);
            if (best.shape < 0 || cost < best.cost) best = {s, split, cost};
        }
    }
    return best;
}

// What a launch of Gemm is: a tile shape and split, or the tensor-core kernel.  The search costs some 2 us of host
// time, as much as the launch itself, so each thread remembers the choices of the last few problems.  ONNXB_FP32 = "tc"
// pins the tensor-core kernel (but for the dot-product kernel's problems), any other value the FMA one.
struct Choice {
    int M, N, K, groups, pixels;
    Pick pick;
    Fp32GemmPlan plan;
    bool tc;
};
// Whether a problem may go to the tensor cores, faster there or not.  The split operands' own error does not grow with the
// reduction, the FMA kernel's chain of additions does: relative to the result (2-norm, against 64 bits) split operands err by
// 1.2 to 1.4e-7 up to some 1000 terms, the FMA kernel by 1.1e-7 where a CTA adds 35 terms, 1.5e-7 at 69, 2.1e-7 at 144.  So
// the tensor cores are for what an FMA kernel's CTA would add some 60 terms of; and, with fewer, for problems of much work per
// output tile (12,000 cycles' worth: 4119 x 1513 x 56 33 us by FMA, 20 there; 5230 x 5956 x 33 stays).  One round of 128 x 128 tiles
// of 17 to 32 terms also stays, by the estimates (563 x 3424 x 27: 10.6 us against 10.7; 15.2 and 9.7 measured), and is the more
// exact for it (0.9e-7 against 1.3e-7).
bool tc_is_as_exact(int M, int N, long long K, int groups, bool pixels, const Pick &fma) {
    if (K >= 64LL * fma.split - 8) return true;
    for (int bn = 16; bn <= 128 && bn <= (M + 15) / 16 * 16; bn += 16) {
        const long long tiles = (N + 127LL) / 128 * ((M + bn - 1) / bn) * groups;
        const double blk = pixels ? 2120.0 + 8.0 * bn : 1750.0 + 5.0 * bn;
        if ((double)((tiles + 147) / 148) * ((double)((K + 31) / 32) * blk + 12000.0) + 4500.0 < fma.cost) return true;
    }
    return false;
}

constexpr double kGemmScale = 0.85;        // the tensor-core estimate runs high by this (18 problems: 0.75 to 0.9)
Choice choose(int M, int N, int K, int groups, bool pixels) {
    thread_local Choice memo[64] = {};
    const char *pin = getenv("ONNXB_FP32");
    const unsigned h = ((unsigned)M * 2654435761u ^ (unsigned)N * 2246822519u ^ (unsigned)K * 3266489917u ^ (unsigned)groups * 668265263u ^
                        (unsigned)pixels) >> 7;
    Choice &c = memo[h % 64];
    if (!pin && c.M == M && c.N == N && c.K == K && c.groups == groups && c.pixels == (int)pixels) return c;
    Choice r{M, N, K, groups, (int)pixels, search_shape(M, N, K, groups, pixels), {0, 0}, false};
    if (!pixels) {
        const double tc = tc_fp32_gemm_plan(M, N, K, r.plan);
        // (the packed copies are addressed in 32 bits of 16-byte pieces)
        const bool fits = tc >= 0 && tc_fp32_gemm_workspace(M, N, K, r.plan) < (1ull << 33);
        r.tc = fits && (pin ? pin[0] == 't' : kGemmScale * tc < r.pick.cost && tc_is_as_exact(M, N, K, 1, false, r.pick));
    }
    if (!pin) c = r;
    return r;
}

template <int AM, int BMODE>
int launch_sgemm(SgemmArgs &a, int groups, const Pick &pick, cudaStream_t st) {
    const int best = pick.shape, best_split = pick.split;
    if (best < 0) return (int)cudaErrorInvalidConfiguration;
    a.tiles_m = (a.M + kShape[best].bm - 1) / kShape[best].bm;
    a.tiles_n = (a.N + kShape[best].bn - 1) / kShape[best].bn;
    const long long tiles = (long long)a.tiles_m * a.tiles_n * groups;
    cudaError_t e;
    switch (best) {
        case 0: e = launch_shape<AM, BMODE, 0, 128, 128, 8, 8>(a, best_split, tiles, st); break;
        case 1: e = launch_shape<AM, BMODE, 1, 64, 128, 8, 8>(a, best_split, tiles, st); break;
        case 2: e = launch_shape<AM, BMODE, 2, 64, 64, 8, 4>(a, best_split, tiles, st); break;
        case 3: e = launch_shape<AM, BMODE, 3, 16, 128, 4, 4>(a, best_split, tiles, st); break;
        default: e = launch_shape<AM, BMODE, 4, 32, 32, 4, 4>(a, best_split, tiles, st); break;
    }
    count_launch();
    return (int)e;
}

}  // namespace

// Up to this size the dot-product kernel beats any tiled launch (64 x 10 x 256: one launch of about 3 us).
bool simt_gemm_is_tiny(long long M, long long N, long long K) { return M * N <= 4096 && M * N * K <= (1 << 20); }

int launch_simt_gemm(const GemmProblem &p, const float *A, const float *B, const float *C, float *Y, void *workspace,
                     size_t workspace_bytes, void *stream) {
    SgemmArgs a{};
    a.A = A; a.B = B; a.Y = Y; a.M = p.M; a.N = p.N; a.K = p.K;
    a.a_ld = p.transA ? p.M : p.K;
    a.b_ld = p.transB ? p.K : p.N;
    a.alpha = p.alpha; a.beta = p.beta; a.C = C; a.c_si = p.c_stride_i; a.c_sj = p.c_stride_j; a.relu = p.relu;
    cudaStream_t st = (cudaStream_t)stream;
    if (simt_gemm_is_tiny(p.M, p.N, p.K)) {
        auto kern = p.transA ? (p.transB ? gemm_dot_kernel<kMnContig, kKContig> : gemm_dot_kernel<kMnContig, kMnContig>)
                             : (p.transB ? gemm_dot_kernel<kKContig, kKContig> : gemm_dot_kernel<kKContig, kMnContig>);
        const cudaError_t e = tc_host::launch_pdl(kern, dim3((unsigned)((p.M * p.N + 3) / 4)), dim3(128), 0, st, a);
        count_launch();
        return (int)e;
    }
    const Choice ch = choose(a.M, a.N, a.K, 1, false);
    const Pick pick = ch.pick;
    if (ch.tc && workspace && workspace_bytes > 0 && workspace_bytes >= tc_fp32_gemm_workspace(p.M, p.N, p.K, ch.plan))
        return launch_tc_fp32_gemm(p, ch.plan, A, B, C, Y, workspace, stream);
    if (p.transA)
        return p.transB ? launch_sgemm<kMnContig, kKContig>(a, 1, pick, st) : launch_sgemm<kMnContig, kMnContig>(a, 1, pick, st);
    return p.transB ? launch_sgemm<kKContig, kKContig>(a, 1, pick, st) : launch_sgemm<kKContig, kMnContig>(a, 1, pick, st);
}

size_t simt_gemm_workspace_bytes(int M, int N, int K) {
    // (never on the tensor cores unless pinned, and a call that short notices the search)
    if (simt_gemm_is_tiny(M, N, K) || ((long long)M * N * K < 2000000 && !getenv("ONNXB_FP32"))) return 0;
    const Choice c = choose(M, N, K, 1, false);
    return c.tc ? tc_fp32_gemm_workspace(M, N, K, c.plan) : 0;
}

// By the estimates: the small-image kernel's (the tiled ones run low where it applies), the FMA kernel's and the tensor-core
// kernel's, where a 1x1 convolution, which has no taps to share a staged pixel, goes by packed pixels (2011 -> 1280 channels
// 23x23, batch 3: 220 us staged, 58 packed, 134 by the im2col of 4-byte loads that both replace).  ONNXB_FP32 as above.
int simt_conv_on_tensor_cores(const ConvGeom &g, Fp32ConvPlan &plan, Fp32GemmPlan &gemm) {
    const char *pin = getenv("ONNXB_FP32");
    if (pin && pin[0] != 't') return 0;
    const long long pixels = (long long)g.N * g.P * g.Q, K = (long long)g.Cg * g.kH * g.kW;      // (each below 2^31)
    const bool flat = g.kH == 1 && g.kW == 1 && g.group == 1 && !(g.pt | g.pl | g.pb | g.pr);
    const double tc = flat ? kGemmScale * tc_fp32_gemm_plan(g.M, (int)pixels, g.C, gemm) : tc_fp32_conv_plan(g, plan);
    if (tc < 0 || (flat && tc_fp32_gemm_workspace(g.M, (int)pixels, g.C, gemm) >= (1ull << 33))) return 0;
    if (!pin) {
        const double small = g.small_cost;
        const Pick fma = search_shape(g.Mg, (int)pixels, (int)K, g.group, true);
        if (tc >= fma.cost || (small >= 0 && 0.85 * small < tc) || !tc_is_as_exact(g.Mg, (int)pixels, K, g.group, true, fma)) return 0;
    }
    return flat ? 2 : 1;
}

int launch_simt_conv(const ConvGeom &g, const float *X, const float *W, const float *B, const float *R, float *Y,
                     void *stream) {
    SgemmArgs a{};
    a.A = W; a.B = X; a.Y = Y; a.M = g.Mg; a.K = g.Cg * g.kH * g.kW;
    const long long cols = (long long)g.N * g.P * g.Q;        // below 2^31: Y has M times as many elements
    a.N = (int)cols;
    a.a_ld = a.K;
    a.bias = B; a.R = R; a.relu = g.relu;
    a.Cch = g.C; a.H = g.H; a.W = g.W; a.PQ = g.P * g.Q; a.Q = g.Q;
    a.sh = g.sh; a.sw = g.sw; a.dh = g.dh; a.dw = g.dw; a.pt = g.pt; a.pl = g.pl;
    a.taps = g.kH * g.kW; a.kW = g.kW; a.Mtot = g.M;
    a.dv_PQ = conv_divisor(a.PQ); a.dv_Q = conv_divisor(a.Q); a.dv_taps = conv_divisor(a.taps); a.dv_kW = conv_divisor(a.kW);
    const Choice ch = choose(a.M, a.N, a.K, g.group, true);
    const Pick pick = ch.pick;
    const double small = g.small_cost;
    const char *pin = getenv("ONNXB_FP32");              // "small" pins the small-image kernel
    if (small >= 0 && (pin ? pin[0] == 's' : 0.85 * small < ch.pick.cost))      // (the tiled estimate runs low here)
        return launch_small_conv(g, X, W, B, R, Y, stream);
    return launch_sgemm<kKContig, kPixels>(a, g.group, pick, (cudaStream_t)stream);
}

}  // namespace onnxb
