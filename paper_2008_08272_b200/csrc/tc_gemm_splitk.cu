// TF32 tensor-core GEMM for problems of few output tiles (small batches, small images, classifier heads):
//     Y[b] (M x N) = relu?( alpha * A' (M x K) * B'[b] (K x N) + beta * C + row bias + addend )
// The persistent kernel of tc_gemm.cu gives such a problem one serial K loop per tile on a fraction of the
// SMs.  Here a cluster of S CTAs shares one 128 x BN output tile: CTA r of the cluster reduces K-blocks
// [r * kb_per, (r + 1) * kb_per) into its own TMEM accumulator (TMA -> shared memory -> tcgen05.mma, as in
// tc_gemm.cu).  Every CTA finishes one slice of the tile's rows: the others write their partial sums of it straight
// from registers into a buffer of that CTA's shared memory (st.async, counted on an mbarrier there), and it adds them
// in rank order, so the result does not depend on timing, applies the epilogue and stores the slice.
// Bound: latency (launch, first fill, K loop, exchange); the split shortens the one part that grows with K.  Partial
// tiles parked in the own shared memory, a cluster barrier, reads of the peers' and a second cluster barrier took
// some 1.1 us longer (ResNet-50 at batch 1, with 37 such layers: 489 -> 447 us): a read waits for a trip to the peer
// and back, a write is sent and done with.
// ONNX Gemm's operands are rounded to TF32 (nearest) inside the kernel: while a stage waits for its MMAs, the
// eight epilogue warps, otherwise idle during the main loop, round it in place in shared memory, so callers
// pass A and B as they are and need no rounding pass in front (the tensor core would truncate them).  A
// convolution's operands arrive as the convolution families prepare them and are left alone.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstdlib>

#include "common.h"
#include "tc_common.cuh"
#include "tc_host.h"

namespace onnxb {

namespace {

using namespace tc;

constexpr int kBM = 128, kBK = 32, kMaxBN = 128;
constexpr int kWorkers = 8;                   // rounding, partial tile, reduction
constexpr int kThreads = (2 + kWorkers) * 32; // warp 0: TMA producer, warp 1: MMA issuer
constexpr int kRoundWarps = kWorkers / 2;     // warps that round one stage; the two halves take the stages in turn
constexpr int kMaxStages = 8;
constexpr int kABytes = kBM * kBK * 4;        // 16 KB
constexpr int kSmemLimit = 232448;

struct SkParams {
    int M, N, K;
    int a_mn, b_mn;            // operand is MN-major (else K-major)
    int a_kbox, b_kbox;        // K-major with K a multiple of 32: one copy brings all K blocks of a stage
    int b_big, b_nblk_full;    // MN-major B through a view of its full 32-column blocks: one copy as well
    int round;                 // round the operands in shared memory
    int BN, S, tiles_m, tiles_n, num_kb, kb_per, num_stages;
    int rows_per, pitch;       // rows of a slice; slots of 16 bytes between a slice's column groups (odd: see the exchange)
    uint32_t stage_bytes, a_bytes, recv_off, idesc;     // a_bytes: of one K block; recv_off: from the first stage to the partial sums
    float alpha, beta;
    const float *C, *row_bias, *R;
    long long c_si, c_sj;
    int relu, vec;             // vec: four columns per access (rows of Y, R and C are 16-byte aligned)
    int r_q, r_row, r_col;     // R sampled: see TcGemmProblem
    float *Yr;
    long long r_ld, r_bs;
    int r_split;
    ConvDivisor dv_rq, dv_rsplit;
    float *Y;
    long long y_ld, y_bs;
    int y_split;               // > 0: column j lies in group j / y_split, y_group elements further on
    long long y_group;
    ConvDivisor dv_split;
    unsigned int *err;
};

// kKS: K blocks per stage (two wherever a CTA has two: see tc_gemm.cu for what a stage costs its issuing threads)
// kExt: with a sampled addend or a second, rounded output; a form of its own (the code, not executed, cost Gemm 2048 x 224 x 144 3 %)
template <int kKS, bool kExt = false>
__global__ void __launch_bounds__(kThreads, 1)
tc_gemm_splitk_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                      const __grid_constant__ CUtensorMap tmBb, const __grid_constant__ SkParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem);
    uint8_t *stages = smem + 1024;
    uint8_t *recv = stages + p.recv_off;
    uint64_t *full = bars, *empty = bars + kMaxStages, *ready = bars + 2 * kMaxStages, *acc_full = bars + 3 * kMaxStages, *recv_full = acc_full + 1;
    uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(bars + 3 * kMaxStages + 2);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = p.S > 1 ? (int)cluster_ctarank() : 0;
    // row tiles fastest: the clusters running side by side share a B tile
    int tile = blockIdx.x / p.S;
    const int tm = tile % p.tiles_m;
    tile /= p.tiles_m;
    const int tn = tile % p.tiles_n, batch = tile / p.tiles_n;
    const int kb0 = rank * p.kb_per, kb1 = min(p.num_kb, kb0 + p.kb_per);
    const int nkb = max(kb1 - kb0, 0);                                // K-blocks this CTA reduces (0: a rank past the end)
    const int nsrc = min(p.S, (p.num_kb + p.kb_per - 1) / p.kb_per);  // ranks that have any
    const int row_lo = rank * p.rows_per;                             // the slice of rows this CTA finishes
    const int row_hi = min(min(kBM, row_lo + p.rows_per), p.M - tm * kBM);

    if (warp == 2) {
        // a barrier per lane: one thread would take a thousand cycles for them
        if (lane < p.num_stages) {
            mbar_init(&full[lane], 1);
            mbar_init(&empty[lane], 1);
            mbar_init(&ready[lane], kRoundWarps);
        }
        if (lane == 31) mbar_init(acc_full, 1);
        if (lane == 30 && p.S > 1) {
            mbar_init(recv_full, 1);
            mbar_arrive_expect_tx(recv_full, (uint32_t)(max(row_hi - row_lo, 0) * p.BN * 4 * nsrc));
        }
        mbar_fence_init();
    } else if (threadIdx.x == 0) {
        prefetch_tmap(&tmA);
        prefetch_tmap(&tmB);
        if (p.b_big) prefetch_tmap(&tmBb);
    }
    if (warp == 1) {
        tmem_alloc(tmem_holder, kMaxBN);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    if (p.S > 1) cluster_arrive();                                    // this CTA's barriers exist
    const uint32_t tmem_base = *tmem_holder;
    pdl_launch_dependents();

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer (lanes 0..na-1: A, then B)
        const bool big = p.b_mn && p.b_big && (tn + 1) * (p.BN / 32) <= p.b_nblk_full;
        const int na = p.a_mn ? kBM / 32 : p.a_kbox ? 1 : kKS;                        // copies per stage
        const int nb = p.b_mn ? (big ? 1 : p.BN / 32) : p.b_kbox ? 1 : kKS;
        const int ib = lane - na;
        const bool is_a = lane < na, active = lane < na + nb;
        const CUtensorMap *tmap = is_a ? &tmA : big ? &tmBb : &tmB;
        // this lane's copy: coordinates of the first stage, their step, and where it goes in a stage
        int c0 = 0, c1 = 0, c2 = 0, c3 = 0, d0 = 0, d1 = 0, d2 = 0;
        uint32_t off = 0;
        if (is_a) {
            if (p.a_mn) { off = (uint32_t)lane * (4096u * kKS); c0 = tm * kBM + lane * 32; c1 = kb0 * kBK; d1 = kKS * kBK; }
            else if (p.a_kbox) { c1 = tm * kBM; c2 = kb0; d2 = kKS; }
            else { off = (uint32_t)lane * p.a_bytes; c0 = (kb0 + lane) * kBK; c1 = tm * kBM; d0 = kKS * kBK; }
        } else {
            off = kKS * p.a_bytes;
            if (big) { c1 = kb0 * kBK; c2 = tn * (p.BN / 32); c3 = batch; d1 = kKS * kBK; }
            else if (p.b_mn) { off += (uint32_t)ib * (4096u * kKS); c0 = tn * p.BN + ib * 32; c1 = kb0 * kBK; c2 = batch; d1 = kKS * kBK; }
            else if (p.b_kbox) { c1 = tn * p.BN; c2 = kb0; c3 = batch; d2 = kKS; }
            else { off += (uint32_t)ib * ((uint32_t)p.BN * 128u); c0 = (kb0 + ib) * kBK; c1 = tn * p.BN; c2 = batch; d0 = kKS * kBK; }
        }
        int stage = 0;
        uint32_t phase = 0;
        pdl_wait();             // everything above overlapped the previous kernel's tail
        for (int kb = 0; kb < nkb; kb += kKS) {
            mbar_wait(&empty[stage], phase ^ 1, p.err, 40);
            if (lane == 0) mbar_arrive_expect_tx(&full[stage], p.stage_bytes);
            __syncwarp();
            if (active) tma_load_4d(stages + (size_t)stage * p.stage_bytes + off, tmap, &full[stage], c0, c1, c2, c3);
            c0 += d0;
            c1 += d1;
            c2 += d2;
            if (++stage == p.num_stages) { stage = 0; phase ^= 1; }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        if (elect_one() && nkb > 0) {
            const uint64_t mn_tmpl = make_smem_desc(0, 4096 * kKS, 512, kSwizzle128B32), k_tmpl = make_smem_desc(0, 16, 1024, kSwizzle128B);
            const uint64_t a_tmpl = p.a_mn ? mn_tmpl : k_tmpl, b_tmpl = p.b_mn ? mn_tmpl : k_tmpl;
            const uint32_t a_hi = (uint32_t)(a_tmpl >> 32), b_hi = (uint32_t)(b_tmpl >> 32);
            // (masked: within a cluster the CTA's rank stands in the upper bits of a shared-memory address)
            const uint32_t a_lo = (uint32_t)a_tmpl | ((smem_u32(stages) >> 4) & 0x3FFFu);
            const uint32_t b_lo = (uint32_t)b_tmpl | (((smem_u32(stages) + kKS * p.a_bytes) >> 4) & 0x3FFFu);
            const uint32_t a_k16 = (p.a_mn ? 1024u : 32u) >> 4, b_k16 = (p.b_mn ? 1024u : 32u) >> 4;
            const uint32_t a_sub16 = (p.a_mn ? 4096u : p.a_bytes) >> 4, b_sub16 = (p.b_mn ? 4096u : (uint32_t)p.BN * 128u) >> 4;
            const uint32_t stage16 = p.stage_bytes >> 4;
            uint64_t *landed = p.round ? ready : full;                // rounded as well, or as they arrive
            int stage = 0;
            uint32_t phase = 0, accumulate = 0;
            for (int kb = 0; kb < nkb; kb += kKS) {
                mbar_wait(&landed[stage], phase, p.err, 41);
                tc_fence_after_sync();
                const uint32_t al = a_lo + (uint32_t)stage * stage16, bl = b_lo + (uint32_t)stage * stage16;
                // (a share's last stage may hold a K block of the next rank's, or none: skipped)
#pragma unroll
                for (int sub = 0; sub < kKS; ++sub) {
                    if (sub == 0 || kb + sub < nkb) {
#pragma unroll
                        for (int k = 0; k < kBK / 8; ++k) {
                            mma_tf32_lohi(tmem_base, al + (uint32_t)sub * a_sub16 + (uint32_t)k * a_k16, a_hi,
                                          bl + (uint32_t)sub * b_sub16 + (uint32_t)k * b_k16, b_hi, p.idesc, accumulate);
                            accumulate = 1;
                        }
                    }
                }
                mma_commit(&empty[stage]);
                if (++stage == p.num_stages) { stage = 0; phase ^= 1; }
            }
            mma_commit(acc_full);
        }
    } else {
        if (p.round) {
            // round every landed stage to TF32 in place (elementwise, so the swizzle does not matter)
            const int rt = ((warp - 2) % kRoundWarps) * 32 + lane, mine = (warp - 2) / kRoundWarps;
            const int n4 = (int)(p.stage_bytes >> 4);
            int stage = 0;
            uint32_t phase = 0;
            for (int kb = 0, i = 0; kb < nkb; kb += kKS, ++i) {
                if ((i & 1) == mine) {
                    mbar_wait(&full[stage], phase, p.err, 43);
                    float4 *st4 = reinterpret_cast<float4 *>(stages + (size_t)stage * p.stage_bytes);
                    for (int j = rt; j < n4; j += 4 * kRoundWarps * 32) {
                        float4 v[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            if (j + u * kRoundWarps * 32 < n4) v[u] = st4[j + u * kRoundWarps * 32];
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            if (j + u * kRoundWarps * 32 < n4)
                                st4[j + u * kRoundWarps * 32] = make_float4(round_tf32_operand(v[u].x), round_tf32_operand(v[u].y), round_tf32_operand(v[u].z), round_tf32_operand(v[u].w));
                    }
                    fence_proxy_async_smem();          // generic-proxy writes, read next by the tensor core
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&ready[stage]);
                }
                if (++stage == p.num_stages) { stage = 0; phase ^= 1; }
            }
        }
        // ------------------------------------------------------------ hand every slice of the partial tile to the CTA that finishes it
        const int q = warp & 3, half = (warp - 2) >> 2;               // TMEM lane quarter; two warps share one
        const int row = q * 32 + lane;
        if (p.S > 1) cluster_wait();                                  // (the peers set up long ago)
        if (nkb > 0) {
            const int dst = min(row / p.rows_per, p.S - 1), n4 = p.BN / 4;
            const bool wanted = row < p.M - tm * kBM;
            uint32_t to = smem_u32(recv) + (uint32_t)((rank * n4 + half * 8) * p.pitch + row - dst * p.rows_per) * 16u, bar = smem_u32(recv_full);
            if (p.S > 1) {
                to = map_to_cta(to, (uint32_t)dst);
                bar = map_to_cta(bar, (uint32_t)dst);
            }
            mbar_wait(acc_full, 0, p.err, 42);
            tc_fence_after_sync();
            for (int c0 = half * 32; c0 < p.BN; c0 += 64, to += 256u * (uint32_t)p.pitch) {
                uint32_t v[32];
                tmem_ld_32x32(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)c0, v);
                tmem_ld_wait();
                if (wanted && p.S == 1) {
                    float4 *own = reinterpret_cast<float4 *>(recv) + (c0 / 4) * p.pitch + row;
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        own[j * p.pitch] = make_float4(__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1]),
                                                       __uint_as_float(v[4 * j + 2]), __uint_as_float(v[4 * j + 3]));
                } else if (wanted) {
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        st_async_v4(to + (uint32_t)(j * p.pitch) * 16u, v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3], bar);
                }
            }
        }
        tc_fence_before_sync();
        if (p.S == 1) asm volatile("bar.sync 1, %0;" ::"n"(kWorkers * 32) : "memory");
        else cluster_arrive();                                        // sent; waited for on the way out only

        // ------------------------------------------------------------ sum this CTA's slice of rows and store it
        pdl_wait();                                // long since satisfied: the producer passed its own before the first load
        const int t = (warp - 2) * 32 + lane;
        const int n4 = p.BN / 4;
        const int col4 = t % n4, gcol = tn * p.BN + col4 * 4;
        for (int rr = row_lo + t / n4; rr < row_hi; rr += kWorkers * 32 / n4) {
            if (gcol >= p.N) break;
            const int grow = tm * kBM + rr;
            long long yi[4];
            if (p.y_split) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int j = gcol + e, gr = conv_fdiv(j, p.y_split, p.dv_split);
                    yi[e] = (long long)gr * p.y_group + (long long)grow * p.y_ld + (j - gr * p.y_split);
                }
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) yi[e] = (long long)batch * p.y_bs + (long long)grow * p.y_ld + gcol + e;
            }
            // the addends are requested before the partial tiles are summed
            float add[4] = {0.f, 0.f, 0.f, 0.f};
            if (p.C) {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (gcol + e < p.N) add[e] = p.beta * __ldg(p.C + (long long)grow * p.c_si + (long long)(gcol + e) * p.c_sj);
            } else if (kExt && p.R && p.r_q) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int j = gcol + e, im = p.r_split ? conv_fdiv(j, p.r_split, p.dv_rsplit) : batch, pix = p.r_split ? j - im * p.r_split : j;
                    const int pr = conv_fdiv(pix, p.r_q, p.dv_rq);
                    if (j < p.N) add[e] = __ldg(p.R + im * p.r_bs + grow * p.r_ld + pr * p.r_row + (pix - pr * p.r_q) * p.r_col);
                }
            } else if (p.R) {
                if (p.vec) {
                    const float4 r = __ldg(reinterpret_cast<const float4 *>(p.R + yi[0]));
                    add[0] = r.x; add[1] = r.y; add[2] = r.z; add[3] = r.w;
                } else {
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (gcol + e < p.N) add[e] = __ldg(p.R + yi[e]);
                }
            }
            const float rb = p.row_bias ? __ldg(p.row_bias + grow) : 0.f;
            // lanes along columns: an odd pitch puts eight neighbours on different banks
            if (p.S > 1) mbar_wait_cluster(recv_full, 0, p.err, 44);
            const float4 *x = reinterpret_cast<const float4 *>(recv) + col4 * p.pitch + rr - row_lo;
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int s = 0; s < 8; ++s)
                if (s < nsrc) {
                    const float4 v = x[s * n4 * p.pitch];
                    a.x += v.x; a.y += v.y; a.z += v.z; a.w += v.w;
                }
            float o[4] = {fmaf(p.alpha, a.x, rb) + add[0], fmaf(p.alpha, a.y, rb) + add[1], fmaf(p.alpha, a.z, rb) + add[2],
                          fmaf(p.alpha, a.w, rb) + add[3]};
            if (p.relu) {
#pragma unroll
                for (int e = 0; e < 4; ++e) o[e] = fmaxf(o[e], 0.f);
            }
            if (kExt && p.Yr) {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (gcol + e < p.N) p.Yr[yi[e]] = round_tf32(o[e]);
            }
            if (p.vec) {
                *reinterpret_cast<float4 *>(p.Y + yi[0]) = make_float4(o[0], o[1], o[2], o[3]);
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (gcol + e < p.N) p.Y[yi[e]] = o[e];
            }
        }
    }

    // no CTA leaves before its peers have sent their shares (they have, unless a wait above gave up)
    if (p.S > 1) {
        if (warp < 2) {
            __syncwarp();
            cluster_wait();
            cluster_arrive();
        }
        cluster_wait();
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, kMaxBN);
    }
}

struct SkChoice {
    int BN, S;               // S = 0: the persistent kernel is the better one
};

// CTAs the device holds at once in clusters of S (clusters of 8 do not fill every GPC); queried once.
int resident_ctas(int S) {
    static std::atomic<int> cached[4] = {};
    const int i = S == 1 ? 0 : S == 2 ? 1 : S == 4 ? 2 : 3;
    int n = cached[i].load(std::memory_order_acquire);
    if (n > 0) return n;
    n = tc_host::num_sms();
    if (S > 1 && cudaFuncSetAttribute(tc_gemm_splitk_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit) == cudaSuccess) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(S * 148);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = kSmemLimit;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)S;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int clusters = 0;
        if (cudaOccupancyMaxActiveClusters(&clusters, tc_gemm_splitk_kernel<2>, &cfg) == cudaSuccess && clusters > 0) n = clusters * S;
        else cudaGetLastError();
    }
    cached[i].store(n, std::memory_order_release);
    return n;
}

// Shape with the shortest estimated time, against the persistent kernel's (both in ns, fitted to 95 problems: 1x1
// convolutions of ResNet-50 at batch 1 to 32 and Gemms from 1 x 1000 x 2048 to 1024 x 1024 x 4096; the choice is
// within 1 % of the best on average).  A wave of CTAs costs 1.4 us and more for its first fill and exchange, and a
// K block 160-420 ns (rounded in shared memory first: 130-620, with the rows of A there are).
// ONNX Gemm's operands may also be rounded by the pre-pass and then come here: half of a K block's time is the rounding, and where
// no operand is large the pre-pass is the shorter (1072 x 384 x 1696 17.4 -> 14.6 us, 416 x 736 x 4416 30.9 -> 24.1, 1024 x 80 x
// 5232 20.9 -> 15.8; but 128 x 4304 x 3136 27 -> 36, 32 x 4704 x 2432 14.8 -> 27).  The choice then is "not in this kernel", and
// falls again once they are rounded.
constexpr double kAhead = 0.85;      // of 0.75 to 1 the best against the estimate above on 104 problems (the pick is within 1.3 % of the better)
SkChoice search(const TcGemmProblem &g) {
    SkChoice c{0, 0};
    if ((g.a_batched && g.batch > 1) || (g.batch > 1 && g.b_batched && g.b_bs % 4)) return c;
    const int num_kb = (g.K + kBK - 1) / kBK;
    double best = 0.97 * tc_gemm_estimate_ns(g);
    const double pre = tc_gemm_prepass_ns(g);
    double ahead = 1e30;                                    // rounded by the pre-pass, then here
    for (int BN = 32; BN <= kMaxBN; BN *= 2)
        for (int S = 1; S <= 8 && S <= num_kb; S *= 2) {
            const long long tiles = (long long)((g.M + kBM - 1) / kBM) * ((g.N + BN - 1) / BN) * g.batch;
            const long long ctas = tiles * S;
            if (ctas > 4 * 148) break;
            const int units = resident_ctas(S);
            const double waves = (double)((ctas + units - 1) / units);
            const double rest = 1390.0 + 23.0 * BN, kb = (double)((num_kb + S - 1) / S);
            const double plain = waves * (kb * (72.0 + 2.71 * BN) + rest) + 1790.0;
            if (!g.round_operands) {
                if (plain < best) {
                    best = plain;
                    c = {BN, S};
                }
                continue;
            }
            const double t = waves * (kb * (64.0 + 1.94 * BN + 2.38 * std::min(g.M, kBM)) + rest) + 1790.0;
            if (t < best) {
                best = t;
                c = {BN, S};
            }
            ahead = std::min(ahead, kAhead * (pre + plain));
        }
    // (two launches keep the host busy for some 8 us where one takes 5: not for calls about as short as that)
    if (ahead < best && best > 10000.0) c = {0, 0};
    return c;
}

bool choose(const TcGemmProblem &g, SkChoice &c) {
    if (g.a_ld % 4 || g.b_ld % 4) return false;
    if (const char *e = getenv("ONNXB_GEMM_SPLITK")) {    // "BN,S": pin the shape for A/B measurements; "0": never
        int bn = 0, sp = 0;
        if (e[0] == '0') return false;
        if (sscanf(e, "%d,%d", &bn, &sp) == 2 && (bn == 32 || bn == 64 || bn == 128) &&
            (sp == 1 || sp == 2 || sp == 4 || sp == 8) && (g.K + kBK - 1) / kBK >= sp) {
            c = {bn, sp};
            return true;
        }
    }
    if (getenv("ONNXB_GEMM_PAIR") || getenv("ONNXB_GEMM_BN")) return false;      // the persistent kernel is being measured
    // each thread remembers the choices of its last few problems (the search costs a microsecond or so)
    struct Memo {
        int M, N, K, batch, flags;
        SkChoice c;
    };
    thread_local Memo memo[64] = {};
    const int flags = g.round_operands | (g.a_batched << 1) | (g.b_batched << 2) | 8;
    const unsigned h = ((unsigned)g.M * 2654435761u ^ (unsigned)g.N * 2246822519u ^ (unsigned)g.K * 3266489917u ^
                        (unsigned)g.batch * 668265263u ^ (unsigned)flags) >> 7;
    Memo &m = memo[h % 64];
    if (!(m.M == g.M && m.N == g.N && m.K == g.K && m.batch == g.batch && m.flags == flags))
        m = {g.M, g.N, g.K, g.batch, flags, search(g)};
    c = m.c;
    return c.S > 0;
}

}  // namespace

bool tc_gemm_splitk_fits(const TcGemmProblem &g) {
    SkChoice c;
    return choose(g, c);
}

int launch_tc_gemm_splitk(const TcGemmProblem &g, void *stream) {
    using namespace tc_host;
    SkChoice c;
    if (!choose(g, c)) return (int)cudaErrorInvalidValue;
    SkParams p{};
    p.M = g.M; p.N = g.N; p.K = g.K;
    p.a_mn = g.a_mn_major; p.b_mn = g.b_mn_major;
    p.round = g.round_operands;
    p.BN = c.BN; p.S = c.S;
    p.tiles_m = (g.M + kBM - 1) / kBM;
    p.tiles_n = (g.N + p.BN - 1) / p.BN;
    p.num_kb = (g.K + kBK - 1) / kBK;
    p.kb_per = (p.num_kb + p.S - 1) / p.S;
    // A K-major A of fewer than 128 rows is staged without the rows it has not (a classifier head at batch 1 has one):
    // the tensor core then reads whatever follows in shared memory for them, and no one reads those rows of the result.
    const int a_rows = p.a_mn ? kBM : std::min(kBM, (g.M + 7) / 8 * 8);
    p.a_bytes = (uint32_t)a_rows * kBK * 4;
    p.rows_per = (std::min(kBM, g.M) + p.S - 1) / p.S;
    p.pitch = p.rows_per | 1;
    const size_t recv_bytes = (size_t)p.S * (p.BN / 4) * p.pitch * 16;
    // two K blocks per stage, where that leaves two stages beside the partial sums
    const int ks = p.kb_per >= 2 ? 2 : 1;
    p.stage_bytes = (p.a_bytes + p.BN * 128) * ks;
    // (never more stages than the share has: a small footprint lets the next kernel's CTAs set up beside this one)
    p.num_stages = std::min({kMaxStages, std::max(2, (p.kb_per + ks - 1) / ks), (int)((kSmemLimit - 2048 - std::max(recv_bytes, (size_t)kABytes)) / p.stage_bytes)});
    p.idesc = tc::make_idesc_tf32(kBM, p.BN, p.a_mn, p.b_mn);
    p.alpha = g.alpha; p.beta = g.beta;
    p.C = g.C; p.c_si = g.c_si; p.c_sj = g.c_sj;
    p.row_bias = g.row_bias;
    p.R = g.C ? nullptr : g.residual;
    p.r_q = p.R ? g.r_q : 0; p.r_row = g.r_row; p.r_col = g.r_col; p.Yr = p.R ? g.Y_rounded : nullptr;
    p.r_split = g.r_split;
    p.dv_rsplit = conv_divisor(std::max(g.r_split, 1));
    p.r_ld = g.r_ld; p.r_bs = g.r_bs;
    p.dv_rq = conv_divisor(std::max(p.r_q, 1));
    p.relu = g.relu;
    p.Y = g.Y; p.y_ld = g.y_ld; p.y_bs = g.y_bs;
    p.y_split = g.y_split; p.y_group = g.y_group_stride;
    p.dv_split = conv_divisor(g.y_split > 0 ? g.y_split : 1);
    p.vec = g.y_split == 0 && g.N % 4 == 0 && g.y_ld % 4 == 0 && (g.batch == 1 || g.y_bs % 4 == 0) &&
            (reinterpret_cast<uintptr_t>(g.Y) & 15) == 0 && (reinterpret_cast<uintptr_t>(p.R) & 15) == 0;
    p.err = device_status_ptr();
    if (!p.err) return (int)cudaErrorUnknown;

    p.a_kbox = !p.a_mn && g.K % kBK == 0;
    p.b_kbox = !p.b_mn && g.K % kBK == 0;
    // K-major: (32 terms, row, K block, batch) or (term, row, batch, 1); MN-major: (row, term, batch, 1)
    auto operand = [&](CUtensorMap *tm, const float *base, int mn, int kbox, uint64_t n, long long ld, int batch, long long bs, uint32_t rows) {
        const uint64_t k = (uint64_t)g.K, nb = (uint64_t)batch, ldb = (uint64_t)ld * 4;
        const uint64_t bsb = batch > 1 ? (uint64_t)bs * 4 : ldb * (mn ? k : n);
        if (kbox) {
            const uint64_t dims[4] = {(uint64_t)kBK, n, k / kBK, nb}, str[3] = {ldb, kBK * 4, bsb};
            const uint32_t box[4] = {(uint32_t)kBK, rows, (uint32_t)ks, 1};
            return make_tmap(tm, base, 4, dims, str, box, kTmapSwizzle128);
        }
        const uint64_t dims[4] = {mn ? n : k, mn ? k : n, nb, 1}, str[3] = {ldb, bsb, bsb * nb};
        const uint32_t box[4] = {(uint32_t)(mn ? 32 : kBK), mn ? (uint32_t)(kBK * ks) : rows, 1, 1};
        return make_tmap(tm, base, 4, dims, str, box, mn ? kTmapSwizzle128Atom32 : kTmapSwizzle128);
    };
    CUtensorMap tmA, tmB;
    if (!operand(&tmA, g.A, p.a_mn, p.a_kbox, g.M, g.a_ld, 1, 0, a_rows) ||
        !operand(&tmB, g.B, p.b_mn, p.b_kbox, g.N, g.b_ld, g.b_batched ? g.batch : 1, g.b_bs, p.BN))
        return (int)cudaErrorInvalidValue;
    CUtensorMap tmBb = tmB;
    p.b_nblk_full = g.N / 32;
    if (p.b_mn && p.BN >= 64 && p.b_nblk_full * 32 >= p.BN) {
        const uint64_t nb = g.b_batched ? (uint64_t)g.batch : 1, ldb = (uint64_t)g.b_ld * 4;
        const uint64_t dims[4] = {32, (uint64_t)g.K, (uint64_t)p.b_nblk_full, nb};
        const uint64_t str[3] = {ldb, 128, nb > 1 ? (uint64_t)g.b_bs * 4 : ldb * g.K};
        const uint32_t box[4] = {32, (uint32_t)(kBK * ks), (uint32_t)(p.BN / 32), 1};
        p.b_big = make_tmap(&tmBb, g.B, 4, dims, str, box, kTmapSwizzle128Atom32) ? 1 : 0;
    }
    p.recv_off = (uint32_t)p.num_stages * p.stage_bytes;
    const size_t smem = smem_with_tmem(2048 + p.recv_off + std::max(recv_bytes, (size_t)kABytes), kMaxBN);      // (at least what an MMA of the last stage reads)
    auto kern = p.r_q || p.Yr ? (ks == 2 ? tc_gemm_splitk_kernel<2, true> : tc_gemm_splitk_kernel<1, true>)
                              : (ks == 2 ? tc_gemm_splitk_kernel<2> : tc_gemm_splitk_kernel<1>);
    const cudaError_t ae = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
    if (ae != cudaSuccess) return (int)ae;
    const dim3 grid((unsigned)((long long)p.tiles_m * p.tiles_n * g.batch * p.S)), block(kThreads);
    const cudaError_t le = p.S > 1 ? launch_pdl_cluster(kern, (unsigned)p.S, grid, block, smem, (cudaStream_t)stream, tmA, tmB, tmBb, p)
                                   : launch_pdl(kern, grid, block, smem, (cudaStream_t)stream, tmA, tmB, tmBb, p);
    count_launch();
    return (int)le;
}

}  // namespace onnxb
