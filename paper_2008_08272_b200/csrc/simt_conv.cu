// SIMT (fp32 FMA) convolution kernels: the path for contractions too thin for
// the tensor cores (few input channels per group, depthwise) and the general
// fallback that accepts every attribute combination of ONNX Conv (Sec. 4.1).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <type_traits>

#include "common.h"
#include "tc_common.cuh"
#include "tc_host.h"

namespace onnxb {

namespace {

// Convolution of small images (an MNIST-size layer): latency, not throughput.  A block owns 128 output pixels
// of one image and MB output channels of one group; it brings the group's padded input image and its
// filters into shared memory in one go (every load in flight at once, zeros for the padding, so the taps need
// no bounds checks) and each thread then sums its pixel's MB outputs.  Filters lie as [c][tap, padded to 4]
// (MB = 1: one 16-byte read serves four taps) or [c][tap][MB] (MB > 1: one read serves four channels).
// K > 0: a K x K filter with unrolled taps; K = 0: any.  One 14x14 image, 8 -> 16 channels, 5x5: 6.8 -> 4 us.
// The image is brought in position by position, no thread idle, stepping from one to the next without dividing; or (kRows) a warp a row,
// which takes a third of the instructions, but idle lanes mean more trips to memory one behind the other: 8 -> 16 5x5 on one 14x14 image
// 3.9 us by positions, 4.5 by rows (4.6 by positions with two divisions each), 3 -> 16 3x3 32x32 3.3, 4.2 (4.6), 1 -> 6 5x5 32x32 at batch
// 200 11.2, 14.5 (12.6); rows of 32 and 30: 1 -> 8 5x5 28x28 at batch 256 10.7, 10.1 (11.3), 1 -> 32 3x3 22.2, 21.1 (22.4).  So kRows where
// rows are all but whole warps and an SM has more than three blocks to issue.
// The arguments come to 224 bytes: a launch takes 0.3 us less of host time at 209 to 224 bytes of them (and 64 more) than at other sizes
// (empty kernels of 168 to 288 bytes, 2.0 and 2.3 us); MNIST at one image, five calls one by one, 20.8 us at 228 bytes, 19.9 at 224.
// Eight blocks per SM leave a thread 64 registers: with the 40 that the compiler takes by itself, for more blocks than shared memory has
// room for, a window's pixels come from there piece by piece: 8 -> 16 5x5 14x14 at batch 18 4.9 us, 4.5 so; 1 -> 8 28x28 at 256 10.9, 10.1.
constexpr int kSmallThreads = 128;
constexpr int kSmallSmem = 48 * 1024;

template <int MB, int K, bool kRows>
__global__ void __launch_bounds__(kSmallThreads, 8)
conv2d_small_kernel(const __grid_constant__ ConvGeom g, const float *__restrict__ X, const float *__restrict__ W,
                    const float *__restrict__ B, const float *__restrict__ R, float *__restrict__ Y, int Hp, int Wp,
                    const ConvDivisor dv_Wp, const ConvDivisor dv_Hp, const ConvDivisor dv_Q, const ConvDivisor dv_taps) {
    extern __shared__ __align__(16) float sm[];
    const int taps = K > 0 ? K * K : g.kH * g.kW, kW = K > 0 ? K : g.kW, taps4 = (taps + 3) / 4 * 4;
    const int ptiles = (g.P * g.Q + kSmallThreads - 1) / kSmallThreads, mtiles = (g.Mg + MB - 1) / MB;
    int b = blockIdx.x;
    const int pt = b % ptiles; b /= ptiles;
    const int mt = b % mtiles; b /= mtiles;
    const int grp = b % g.group, n = b / g.group;
    const int m0 = mt * MB, plane = Hp * Wp;
    float *ws = sm, *xs = sm + g.Cg * (MB == 1 ? taps4 : taps * MB);
    tc::pdl_launch_dependents();
    tc::pdl_wait();

    const int kred = g.Cg * taps;
    // eight loads in flight per thread
    for (int i0 = threadIdx.x; i0 < kred * MB; i0 += 8 * kSmallThreads) {
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int i = i0 + u * kSmallThreads, j = MB == 1 ? 0 : i & (MB - 1), k = i / MB;
            v[u] = i < kred * MB && m0 + j < g.Mg ? __ldg(W + (size_t)(grp * g.Mg + m0 + j) * kred + k) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int i = i0 + u * kSmallThreads, c = conv_fdiv(i, taps, dv_taps);
            if (i < kred * MB) ws[MB == 1 ? c * taps4 + (i - c * taps) : i] = v[u];
        }
    }
    const float *xg = X + ((size_t)n * g.C + (size_t)grp * g.Cg) * g.H * g.W;
    if (kRows) {
        // a warp a row: a thread keeps its column
        const int rows = g.Cg * Hp, step = kSmallThreads / 32;
#pragma unroll 1
        for (int wp = threadIdx.x & 31; wp < Wp; wp += 32) {
            const int w = wp - g.pl;
            const bool in = (unsigned)w < (unsigned)g.W;
#pragma unroll 1
            for (int r0 = threadIdx.x / 32; r0 < rows; r0 += 8 * step) {
                float v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int r = r0 + u * step, c = conv_fdiv(r, Hp, dv_Hp), h = r - c * Hp - g.pt;
                    v[u] = in && r < rows && (unsigned)h < (unsigned)g.H ? __ldg(xg + ((size_t)c * g.H + h) * g.W + w) : 0.f;
                }
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (r0 + u * step < rows) xs[(r0 + u * step) * Wp + wp] = v[u];
            }
        }
    } else {
        // no thread idle, from one position to the next without dividing
        const int total = g.Cg * plane, row = conv_fdiv(threadIdx.x, Wp, dv_Wp), dr = conv_fdiv(kSmallThreads, Wp, dv_Wp);
        int c = conv_fdiv(row, Hp, dv_Hp), h = row - c * Hp, w = threadIdx.x - row * Wp;
        const int dc = conv_fdiv(dr, Hp, dv_Hp), dh = dr - dc * Hp, dw = kSmallThreads - dr * Wp;
        for (int i0 = threadIdx.x; i0 < total; i0 += 8 * kSmallThreads) {
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const bool in = i0 + u * kSmallThreads < total && (unsigned)(h - g.pt) < (unsigned)g.H && (unsigned)(w - g.pl) < (unsigned)g.W;
                v[u] = in ? __ldg(xg + ((size_t)c * g.H + (h - g.pt)) * g.W + (w - g.pl)) : 0.f;
                w += dw; h += dh; c += dc;
                if (w >= Wp) { w -= Wp; ++h; }
                if (h >= Hp) { h -= Hp; ++c; }
            }
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (i0 + u * kSmallThreads < total) xs[i0 + u * kSmallThreads] = v[u];
        }
    }
    __syncthreads();

    const int pix = pt * kSmallThreads + threadIdx.x;
    if (pix >= g.P * g.Q) return;
    const int p = conv_fdiv(pix, g.Q, dv_Q), q = pix - p * g.Q;
    float acc[MB];
#pragma unroll
    for (int j = 0; j < MB; ++j) acc[j] = 0.f;
    const float *xc = xs + p * g.sh * Wp + q * g.sw;
    for (int c = 0; c < g.Cg; ++c, xc += plane) {
        if (K > 0) {
            float x[K > 0 ? K * K : 1];
#pragma unroll
            for (int r = 0; r < K; ++r)
#pragma unroll
                for (int s = 0; s < K; ++s) x[r * K + s] = xc[r * g.dh * Wp + s * g.dw];
            if (MB == 1) {
                const float4 *wc = reinterpret_cast<const float4 *>(ws + c * taps4);
#pragma unroll
                for (int t = 0; t < (K * K + 3) / 4; ++t) {
                    const float4 w = wc[t];
                    acc[0] = fmaf(x[4 * t], w.x, acc[0]);
                    if (4 * t + 1 < K * K) acc[0] = fmaf(x[4 * t + 1 < K * K ? 4 * t + 1 : 0], w.y, acc[0]);
                    if (4 * t + 2 < K * K) acc[0] = fmaf(x[4 * t + 2 < K * K ? 4 * t + 2 : 0], w.z, acc[0]);
                    if (4 * t + 3 < K * K) acc[0] = fmaf(x[4 * t + 3 < K * K ? 4 * t + 3 : 0], w.w, acc[0]);
                }
            } else {
#pragma unroll
                for (int t = 0; t < K * K; ++t) {
#pragma unroll
                    for (int j = 0; j + 3 < MB; j += 4) {
                        const float4 w = *reinterpret_cast<const float4 *>(ws + (c * taps + t) * MB + j);
                        acc[j] = fmaf(x[t], w.x, acc[j]);
                        acc[j + 1] = fmaf(x[t], w.y, acc[j + 1]);
                        acc[j + 2] = fmaf(x[t], w.z, acc[j + 2]);
                        acc[j + 3] = fmaf(x[t], w.w, acc[j + 3]);
                    }
                }
            }
        } else {
            int r = 0, s = 0;
            for (int t = 0; t < taps; ++t) {
                const float x = xc[r * g.dh * Wp + s * g.dw];
#pragma unroll
                for (int j = 0; j < MB; ++j) acc[j] = fmaf(x, ws[MB == 1 ? c * taps4 + t : (c * taps + t) * MB + j], acc[j]);
                if (++s == kW) { s = 0; ++r; }
            }
        }
    }
#pragma unroll
    for (int j = 0; j < MB; ++j) {
        if (m0 + j < g.Mg) {
            const int m = grp * g.Mg + m0 + j;
            const size_t yi = ((size_t)n * g.M + m) * g.P * g.Q + pix;
            float v = acc[j] + (B ? __ldg(B + m) : 0.f);
            if (R) v += __ldg(R + yi);
            if (g.relu) v = v > 0.f ? v : 0.f;
            Y[yi] = v;
        }
    }
}

// Depthwise convolution (group == C == M): purely HBM-bound, 2*kH*kW flops per
// output.  A block stages the input window of a 32 x 32 output tile of one
// (image, channel) plane in shared memory with coalesced row loads (zeros
// outside the image); each of its 256 threads then produces a column strip of
// four vertically adjacent outputs, so the rows of the window shared by the
// four outputs are read from shared memory once per tap column.
constexpr int kDwTP = 32, kDwTQ = 32, kDwRows = 4, kDwThreads = kDwTQ * (kDwTP / kDwRows);

__global__ void __launch_bounds__(kDwThreads)
conv2d_depthwise_kernel(const ConvGeom g, const float *__restrict__ X, const float *__restrict__ W,
                        const float *__restrict__ B, const float *__restrict__ R, float *__restrict__ Y, int q_tiles,
                        int p_tiles,
                        int in_rows, int in_cols, int pitch) {
    extern __shared__ float tile[];           // [in_rows][pitch] then weights [kH*kW]
    float *wsm = tile + in_rows * pitch;

    int bid = blockIdx.x;
    const int qt = bid % q_tiles; bid /= q_tiles;
    const int pt_ = bid % p_tiles; bid /= p_tiles;
    const int plane = bid;                    // n * C + c
    const int c = plane % g.C;
    const int p0 = pt_ * kDwTP, q0 = qt * kDwTQ;
    const int ih0 = p0 * g.sh - g.pt, iw0 = q0 * g.sw - g.pl;
    const float *xp = X + (size_t)plane * g.H * g.W;

    const int taps = g.kH * g.kW;
    for (int i = threadIdx.x; i < taps; i += kDwThreads) wsm[i] = W[(size_t)c * taps + i];
    // window rows actually needed by this tile (fewer at the bottom edge of the image)
    const int rows_out = min(kDwTP, g.P - p0);
    const int rows_in = min(in_rows, (rows_out - 1) * g.sh + (g.kH - 1) * g.dh + 1);
    for (int i = threadIdx.x; i < rows_in * in_cols; i += kDwThreads) {
        const int rr = i / in_cols, cc = i - rr * in_cols;
        const int ih = ih0 + rr, iw = iw0 + cc;
        float v = 0.f;
        if ((unsigned)ih < (unsigned)g.H && (unsigned)iw < (unsigned)g.W) v = __ldg(xp + (size_t)ih * g.W + iw);
        tile[rr * pitch + cc] = v;
    }
    __syncthreads();

    const int tq = threadIdx.x % kDwTQ, tp = (threadIdx.x / kDwTQ) * kDwRows;
    const int q = q0 + tq;
    if (q >= g.Q || p0 + tp >= g.P) return;
    float acc[kDwRows];
#pragma unroll
    for (int k = 0; k < kDwRows; ++k) acc[k] = 0.f;
    for (int s = 0; s < g.kW; ++s) {
        const float *col = tile + tq * g.sw + s * g.dw;
        for (int r = 0; r < g.kH; ++r) {
            const float w = wsm[r * g.kW + s];
#pragma unroll
            for (int k = 0; k < kDwRows; ++k)
                if (tp + k < rows_out) acc[k] = fmaf(col[((tp + k) * g.sh + r * g.dh) * pitch], w, acc[k]);
        }
    }
    const float bias = B ? __ldg(B + c) : 0.f;
#pragma unroll
    for (int k = 0; k < kDwRows; ++k) {
        const int p = p0 + tp + k;
        if (p < g.P) {
            float v = acc[k] + bias;
            const size_t yi = ((size_t)plane * g.P + p) * g.Q + q;
            if (R) v += __ldg(R + yi);
            if (g.relu) v = v > 0.f ? v : 0.f;
            Y[yi] = v;
        }
    }
}

// Gather for strided / oddly sized 1x1 convolutions, values rounded to TF32 (nearest, ties away):
//   merged:    Xg[c][n*P*Q + p*Q + q] = X[n][c][p*sh][q*sw], rows padded with zeros to the pitch;
//   per image: Xg[n][c][p*Q + q]      (pitch = P*Q).
// Both kernels below are bound by HBM (the pixels read once, the copy written once): one wave of eight blocks per SM, indices
// by multiplication (256 channels 56x56 -> 28x28 at batch 32: some 20 -> 15 us).

// Weights of the call, rounded to TF32 ahead of the pixels: a launch of its own for them in front cost up to 2 us (256 -> 512
// channels 56x56/2 at batch 32 41.2 -> 39.9 us in all, at batch 4 12.3 -> 10.3; with few pixels and many weights see launch_gather1x1).
struct RoundedCopy {
    const float4 *in;
    float4 *out;
    unsigned n4;
};
__device__ __forceinline__ void round_copy(const RoundedCopy &w) {
    for (unsigned i = blockIdx.x * 256u + threadIdx.x; i < w.n4; i += gridDim.x * 256u) {
        const float4 v = __ldg(w.in + i);
        w.out[i] = make_float4(tc::round_tf32(v.x), tc::round_tf32(v.y), tc::round_tf32(v.z), tc::round_tf32(v.w));
    }
}

// Any layout whose pitch is a multiple of four (both layouts have one): four consecutive outputs per
// thread, indices divided once and then stepped, four independent scalar loads, one 16-byte store.
__global__ void __launch_bounds__(256)
gather1x1_quad_kernel(const float *__restrict__ X, float4 *__restrict__ Xg4, unsigned total4, unsigned pitch,
                      unsigned NPQ, unsigned PQ, unsigned Q, unsigned C, unsigned HW, unsigned rowstep, unsigned sw,
                      int merged, const ConvDivisor dv_pitch, const ConvDivisor dv_PQ, const ConvDivisor dv_Q, const RoundedCopy w) {
    tc::pdl_launch_dependents();
    tc::pdl_wait();
    round_copy(w);
    for (unsigned i4 = blockIdx.x * 256u + threadIdx.x; i4 < total4; i4 += gridDim.x * 256u) {
        const unsigned i = i4 * 4u;
        const unsigned row = (unsigned)conv_fdiv((int)i, (int)pitch, dv_pitch);   // merged: channel; per image: n*C + c
        const unsigned j = i - row * pitch;                                        // a multiple of four
        unsigned n = 0, r = j;
        if (merged) {
            n = (unsigned)conv_fdiv((int)j, (int)PQ, dv_PQ);
            r = j - n * PQ;
        }
        unsigned pp = (unsigned)conv_fdiv((int)r, (int)Q, dv_Q), q = r - pp * Q;
        float v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const unsigned plane = merged ? n * C + row : row;
            v[e] = j + e < NPQ ? tc::round_tf32(__ldg(X + (size_t)plane * HW + pp * rowstep + q * sw)) : 0.f;
            // step to the next output pixel: along the row, then to the next row, then to the next image
            ++r;
            if (++q == Q) { q = 0; ++pp; }
            if (r == PQ) { r = 0; pp = 0; q = 0; ++n; }
        }
        Xg4[i4] = make_float4(v[0], v[1], v[2], v[3]);
    }
}

// Per-image layout, Q a multiple of 4, W a multiple of 4, column stride 1 or 2: four outputs per
// thread from one or two aligned 16-byte loads, one 16-byte store.
template <int SW>
__global__ void __launch_bounds__(256)
gather1x1_vec_kernel(const float4 *__restrict__ X4, float4 *__restrict__ Xg4, unsigned total4, unsigned PQ4,
                     unsigned Q4, unsigned HW4, unsigned rowstep4, const ConvDivisor dv_PQ4, const ConvDivisor dv_Q4, const RoundedCopy w) {
    tc::pdl_launch_dependents();
    tc::pdl_wait();
    round_copy(w);
    for (unsigned i = blockIdx.x * 256u + threadIdx.x; i < total4; i += gridDim.x * 256u) {
        const unsigned plane = (unsigned)conv_fdiv((int)i, (int)PQ4, dv_PQ4), r = i - plane * PQ4;
        const unsigned p = (unsigned)conv_fdiv((int)r, (int)Q4, dv_Q4), q4 = r - p * Q4;
        const float4 *src = X4 + (size_t)plane * HW4 + p * rowstep4 + q4 * SW;
        float4 o;
        if (SW == 1) {
            o = __ldg(src);
        } else {
            const float4 a = __ldg(src), b = __ldg(src + 1);
            o = make_float4(a.x, a.z, b.x, b.z);
        }
        Xg4[i] = make_float4(tc::round_tf32(o.x), tc::round_tf32(o.y), tc::round_tf32(o.z), tc::round_tf32(o.w));
    }
}

// Depthwise convolution with unit stride and dilation (group = C = M), the HBM-bound case: 2.25
// flop per byte, so the only thing that matters is to move each plane once with few instructions.
// A thread owns a strip of 4 output columns by ROWS output rows of one (image, channel) plane, reads
// the KH + ROWS - 1 input rows it needs straight from global memory (neighbouring threads' overlapping
// reads are served by L1) and keeps the window in registers: with ROWS = 4 and a 3x3 filter, 6 row loads
// and 144 FMAs for 16 outputs, every input row fetched 1.5 times instead of twice with ROWS = 2.  VEC: rows are whole
// 16-byte pieces and as wide as the output, so a row costs one aligned 16-byte load; the columns to its left and
// right come from the neighbouring lanes, which hold them (the first and last lane of a warp load theirs), and
// beyond the row's ends lies padding.  Otherwise every column is loaded on its own.
// The window of a strip whose rows are whole 16-byte pieces (plane: in global or in shared memory).  Every input row is
// requested before the first use; all lanes of the warp take part.
template <int KH, int KW, int ROWS, bool SHARED>
__device__ __forceinline__ void depthwise_window_vec(const float *plane, int H, int W, int h0, int q0, float (&v)[KH + ROWS - 1][KW + 3]) {
    constexpr int L = (KW - 1) / 2, RT = KW - 1 - L;       // columns to the left (= the pad) and right of the quad
    const int lane = threadIdx.x & 31;
    const bool left_in = q0 > 0, right_in = q0 + 4 < W;
    float e[KH + ROWS - 1][L > RT ? L : RT];               // what the warp's first and last lane load themselves
    auto get = [](const float *q) { return SHARED ? *q : __ldg(q); };
#pragma unroll
    for (int rr = 0; rr < KH + ROWS - 1; ++rr) {
        const int ih = h0 + rr;
        const bool row_in = (unsigned)ih < (unsigned)H;
        const float *row = plane + (ptrdiff_t)ih * W + q0;
        float4 m = make_float4(0.f, 0.f, 0.f, 0.f);
        if (row_in) m = SHARED ? *reinterpret_cast<const float4 *>(row) : __ldg(reinterpret_cast<const float4 *>(row));
        v[rr][L] = m.x; v[rr][L + 1] = m.y; v[rr][L + 2] = m.z; v[rr][L + 3] = m.w;
#pragma unroll
        for (int k = 0; k < (L > RT ? L : RT); ++k) {
            e[rr][k] = 0.f;
            if (lane == 0 && k < L && row_in && left_in) e[rr][k] = get(row - L + k);
            if (lane == 31 && k < RT && row_in && right_in) e[rr][k] = get(row + 4 + k);
        }
    }
#pragma unroll
    for (int rr = 0; rr < KH + ROWS - 1; ++rr) {
#pragma unroll
        for (int k = 0; k < L; ++k) {
            const float x = __shfl_up_sync(0xffffffffu, v[rr][L + 4 - L + k], 1);
            v[rr][k] = !left_in ? 0.f : lane == 0 ? e[rr][k] : x;
        }
#pragma unroll
        for (int k = 0; k < RT; ++k) {
            const float x = __shfl_down_sync(0xffffffffu, v[rr][L + k], 1);
            v[rr][L + 4 + k] = !right_in ? 0.f : lane == 31 ? e[rr][k] : x;
        }
    }
}

// Filter, addend, Relu and store of a strip: 4 output columns from q0, ROWS output rows from p0 of one plane.
template <int KH, int KW, int ROWS, bool VEC>
__device__ __forceinline__ void depthwise_strip(const ConvGeom &g, const float (&v)[KH + ROWS - 1][KW + 3], const float (&w)[KH * KW],
                                                float bias, const float *__restrict__ R, float *__restrict__ Y, size_t plane, int p0, int q0) {
    float acc[ROWS][4];
#pragma unroll
    for (int k = 0; k < ROWS; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[k][j] = bias;
#pragma unroll
    for (int rr = 0; rr < KH + ROWS - 1; ++rr) {
        // input row rr is filter row rr - k of output row p0 + k
#pragma unroll
        for (int k = 0; k < ROWS; ++k) {
            if (rr - k >= 0 && rr - k < KH) {
#pragma unroll
                for (int s = 0; s < KW; ++s)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[k][j] = fmaf(v[rr][j + s], w[(rr - k) * KW + s], acc[k][j]);
            }
        }
    }
    float *yp = Y + (plane * g.P + p0) * g.Q + q0;
#pragma unroll
    for (int k = 0; k < ROWS; ++k) {
        float *a = acc[k];
        if (p0 + k >= g.P) break;
        if (R) {
            const float *rr = R + (yp - Y) + (size_t)k * g.Q;
#pragma unroll
            for (int j = 0; j < 4; ++j) if (q0 + j < g.Q) a[j] += __ldg(rr + j);
        }
        if (g.relu) {
#pragma unroll
            for (int j = 0; j < 4; ++j) a[j] = a[j] > 0.f ? a[j] : 0.f;
        }
        float *yr = yp + (size_t)k * g.Q;
        if (VEC && q0 + 3 < g.Q) {
            *reinterpret_cast<float4 *>(yr) = make_float4(a[0], a[1], a[2], a[3]);
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) if (q0 + j < g.Q) yr[j] = a[j];
        }
    }
}

template <int KH, int KW, bool VEC, int ROWS>
__global__ void __launch_bounds__(256)
conv2d_depthwise_unit_kernel(const ConvGeom g, const float *__restrict__ X, const float *__restrict__ W,
                             const float *__restrict__ B, const float *__restrict__ R, float *__restrict__ Y,
                             unsigned items, unsigned Q4, unsigned P2, double inv_Q4, double inv_P2) {
    constexpr int WIN = KW + 3;                // input columns a strip of 4 outputs touches
    tc::pdl_launch_dependents();
    const unsigned i_own = blockIdx.x * 256u + threadIdx.x;
    if (!VEC && i_own >= items) return;
    const unsigned i = VEC && i_own >= items ? items - 1 : i_own;      // (the neighbours of a live lane must stay)
    // i = (plane * P2 + row group) * Q4 + column quad (P2 = row groups per plane); quotients by reciprocal multiplication in
    // double (right for 31-bit operands up to one unit, which the two comparisons repair)
    unsigned t = __double2uint_rd((double)i * inv_Q4);
    if (t * Q4 > i) --t;
    if ((t + 1) * Q4 <= i) ++t;
    const unsigned q4 = i - t * Q4;
    unsigned plane = __double2uint_rd((double)t * inv_P2);
    if (plane * P2 > t) --plane;
    if ((plane + 1) * P2 <= t) ++plane;
    const int p0 = (int)(t - plane * P2) * ROWS, q0 = (int)q4 * 4;
    const int c = (int)(plane % (unsigned)g.C);

    const float *xp = X + (size_t)plane * g.H * g.W;
    tc::pdl_wait();
    // Every input row of the window is requested before the first FMA: the kernel is bound by the
    // latency of these loads, so each thread keeps all of them in flight at once.
    float v[KH + ROWS - 1][WIN];
    if (VEC) {
        depthwise_window_vec<KH, KW, ROWS, false>(xp, g.H, g.W, p0 - g.pt, q0, v);
        if (i_own >= items) return;
    } else {
        const int iw0 = q0 - g.pl;
#pragma unroll
        for (int rr = 0; rr < KH + ROWS - 1; ++rr) {
            const int ih = p0 - g.pt + rr;
            const float *row = xp + (size_t)ih * g.W;
#pragma unroll
            for (int k = 0; k < WIN; ++k) {
                v[rr][k] = 0.f;
                if ((unsigned)ih < (unsigned)g.H && (unsigned)(iw0 + k) < (unsigned)g.W) v[rr][k] = __ldg(row + iw0 + k);
            }
        }
    }
    float w[KH * KW];
#pragma unroll
    for (int k = 0; k < KH * KW; ++k) w[k] = __ldg(W + (size_t)c * (KH * KW) + k);
    depthwise_strip<KH, KW, ROWS, VEC>(g, v, w, B ? __ldg(B + c) : 0.f, R, Y, plane, p0, q0);
}

// The same strips, the input streamed through shared memory: planes are contiguous, so a bulk copy brings a block's next
// `per` of them while it works on the last ones, and the loads that the kernel above waits for on every strip are
// never out of flight.  One wave of CTAs (as many as fit an SM), each with its own ring of kRingStages copies; more
// or larger ones were slower (256 channels 28x28, batch 64: 22.4 us by the kernel above, 20.3 with two stages and four
// CTAs per SM, 20.9 with three and three, 22.4 with five and two).  Bound by HBM, at 5.1 TB/s there.
constexpr int kRingStages = 2, kRingCtas = 4, kRingStageMax = 24576;

__global__ void __launch_bounds__(256, kRingCtas)
conv2d_depthwise_ring_kernel(const ConvGeom g, const float *__restrict__ X, const float *__restrict__ W, const float *__restrict__ B,
                             const float *__restrict__ R, float *__restrict__ Y, unsigned planes, unsigned per, unsigned Q4, unsigned P2,
                             const ConvDivisor dv_Q4, const ConvDivisor dv_P2, const ConvDivisor dv_C, unsigned int *err) {
    constexpr int KH = 3, KW = 3, ROWS = 4;                    // the one filter and strip that the launch gives it
    extern __shared__ __align__(128) float ring[];
    __shared__ uint64_t full[kRingStages];
    const unsigned units = (planes + per - 1) / per, plane_floats = (unsigned)(g.H * g.W);
    if (threadIdx.x == 0) {
        for (int k = 0; k < kRingStages; ++k) tc::mbar_init(&full[k], 1);
        tc::mbar_fence_init();
    }
    __syncthreads();
    tc::pdl_launch_dependents();
    tc::pdl_wait();
    auto fetch = [&](unsigned u, int stage) {
        const unsigned cnt = min(per, planes - u * per);
        tc::mbar_arrive_expect_tx(&full[stage], cnt * plane_floats * 4u);
        tc::bulk_load_1d(ring + (size_t)stage * per * plane_floats, X + (size_t)u * per * plane_floats, cnt * plane_floats * 4u, &full[stage]);
    };
    if (threadIdx.x == 0)
        for (int k = 0; k < kRingStages; ++k)
            if (blockIdx.x + k * gridDim.x < units) fetch(blockIdx.x + k * gridDim.x, k);
    int stage = 0;
    uint32_t phase = 0;
    for (unsigned u = blockIdx.x; u < units; u += gridDim.x) {
        const unsigned items = min(per, planes - u * per) * P2 * Q4, i = min(threadIdx.x, items - 1);     // (at most 256; the neighbours of a live lane must stay)
        const unsigned t = (unsigned)conv_fdiv((int)i, (int)Q4, dv_Q4), pl = (unsigned)conv_fdiv((int)t, (int)P2, dv_P2);
        const int q0 = (int)(i - t * Q4) * 4, p0 = (int)(t - pl * P2) * ROWS;
        const unsigned plane = u * per + pl;
        const unsigned c = plane - (unsigned)conv_fdiv((int)plane, g.C, dv_C) * (unsigned)g.C;
        float w[KH * KW];
#pragma unroll
        for (int k = 0; k < KH * KW; ++k) w[k] = __ldg(W + (size_t)c * (KH * KW) + k);
        const float bias = B ? __ldg(B + c) : 0.f;
        tc::mbar_wait(&full[stage], phase, err, 60);
        float v[KH + ROWS - 1][KW + 3];
        depthwise_window_vec<KH, KW, ROWS, true>(ring + ((size_t)stage * per + pl) * plane_floats, g.H, g.W, p0 - g.pt, q0, v);
        if (threadIdx.x < items) depthwise_strip<KH, KW, ROWS, true>(g, v, w, bias, R, Y, plane, p0, q0);
        __syncthreads();                                       // every thread has read the stage
        if (threadIdx.x == 0 && u + kRingStages * gridDim.x < units) fetch(u + kRingStages * gridDim.x, stage);
        if (++stage == kRingStages) { stage = 0; phase ^= 1; }
    }
}

// Depthwise convolution whose rows are no whole 16-byte pieces, or whose stride or dilation is not one: a thread owns
// ROWS outputs of one column of a plane, lanes run along the output columns, so that a load touches one line (two at
// column stride 2) where the strips above, four columns to a lane, touch four and more.  Bound by these loads' issue and by
// HBM, so the rows of the window that the thread's outputs share are loaded once: at row stride 1 its outputs lie a dilation
// apart, at row stride 2 (dilation 1) next to each other.  Column stride and dilation cost nothing and are any.  Against the
// tiles of conv2d_depthwise_kernel: 160 channels 70x70 3x3/2 with an addend, batch 26: 165 -> 25 us (floor 19); 176 channels
// 37x37 5x5/2, batch 38: 78 -> 26; 32 channels 179x114 dilation 2, batch 17: 105 -> 37.
template <int KH, int KW, int SH, int ROWS>
__global__ void __launch_bounds__(256)
conv2d_depthwise_column_kernel(const ConvGeom g, const float *__restrict__ X, const float *__restrict__ W, const float *__restrict__ B,
                               const float *__restrict__ R, float *__restrict__ Y, unsigned items, unsigned PG,
                               const ConvDivisor dv_Q, const ConvDivisor dv_PG, const ConvDivisor dv_C, const ConvDivisor dv_dh) {
    constexpr int NR = (ROWS - 1) * SH + KH;
    tc::pdl_launch_dependents();
    const unsigned i = blockIdx.x * 256u + threadIdx.x;
    if (i >= items) return;
    // i = (plane * PG + row group) * Q + column; a group's first row: a block of ROWS * dh rows, then one of its first dh
    const unsigned t = (unsigned)conv_fdiv((int)i, g.Q, dv_Q), q = i - t * (unsigned)g.Q;
    const unsigned plane = (unsigned)conv_fdiv((int)t, (int)PG, dv_PG), pg = t - plane * PG;
    const unsigned dh = SH == 1 ? (unsigned)g.dh : 1u;
    const unsigned blk = SH == 1 ? (unsigned)conv_fdiv((int)pg, g.dh, dv_dh) : pg;
    const unsigned p0 = SH == 1 ? blk * (ROWS * dh) + (pg - blk * dh) : pg * ROWS;
    const unsigned c = plane - (unsigned)conv_fdiv((int)plane, g.C, dv_C) * (unsigned)g.C;
    const float *xp = X + (size_t)plane * g.H * g.W, *wp = W + (size_t)c * (KH * KW);
    // (modulo 2^32: a row or column outside the image, however far, is no row or column of it)
    const unsigned h0 = p0 * SH - (unsigned)g.pt, w0 = q * (unsigned)g.sw - (unsigned)g.pl;
    tc::pdl_wait();
    float v[NR][KW], w[KH * KW];
#pragma unroll
    for (int rr = 0; rr < NR; ++rr) {
        const unsigned ih = h0 + rr * dh;
        const float *row = xp + (size_t)ih * g.W;
#pragma unroll
        for (int s = 0; s < KW; ++s) {
            const unsigned iw = w0 + s * (unsigned)g.dw;
            v[rr][s] = ih < (unsigned)g.H && iw < (unsigned)g.W ? __ldg(row + iw) : 0.f;
        }
    }
#pragma unroll
    for (int k = 0; k < KH * KW; ++k) w[k] = __ldg(wp + k);
    const float bias = B ? __ldg(B + c) : 0.f;
    const size_t y0 = ((size_t)plane * g.P + p0) * g.Q + q, ystep = (size_t)dh * g.Q;
    float r[ROWS];
#pragma unroll
    for (int k = 0; k < ROWS; ++k) r[k] = R && p0 + k * dh < (unsigned)g.P ? __ldg(R + y0 + k * ystep) : 0.f;
#pragma unroll
    for (int k = 0; k < ROWS; ++k) {
        float a = bias;
#pragma unroll
        for (int rr = 0; rr < KH; ++rr)
#pragma unroll
            for (int s = 0; s < KW; ++s) a = fmaf(v[k * SH + rr][s], w[rr * KW + s], a);
        if (R) a += r[k];
        if (g.relu) a = a > 0.f ? a : 0.f;
        if (p0 + k * dh < (unsigned)g.P) Y[y0 + k * ystep] = a;
    }
}

// Rows per thread: the fewest loads per column of a plane (rows past the last one are loaded too) that leave every SM
// 512 threads.
struct ColumnPick {
    int rows;
    long long PG, items;
};
ColumnPick depthwise_column_pick(const ConvGeom &g) {
    ColumnPick best{0, 0, 0};
    long long best_loads = 0;
    for (int rows : {8, 4, 2}) {
        if (rows == 8 && (g.kH == 5 || g.sh == 2)) continue;      // windows of that many registers are slower
        const long long dh = g.sh == 1 ? g.dh : 1, whole = g.P / (rows * dh), PG = whole * dh + std::min(dh, g.P - whole * rows * dh);
        const long long items = (long long)g.N * g.C * PG * g.Q, loads = PG * ((rows - 1) * g.sh + g.kH);
        if (best.rows && best.items >= 148LL * 512 && loads >= best_loads) continue;
        best = {rows, PG, items};
        best_loads = loads;
    }
    return best;
}

bool depthwise_column_fits(const ConvGeom &g) {
    if (!(g.Cg == 1 && g.Mg == 1 && (g.sh == 1 || (g.sh == 2 && g.dh == 1)))) return false;
    if (!((g.kH == 3 && g.kW == 3) || (g.kH == 5 && g.kW == 5))) return false;
    return depthwise_column_pick(g).items < (1LL << 31) - 256;
}

template <int K>
int launch_depthwise_column(const ConvGeom &g, const float *X, const float *W, const float *B, const float *R, float *Y, cudaStream_t st) {
    const ColumnPick p = depthwise_column_pick(g);
    auto kern = g.sh == 1 ? (p.rows == 8   ? conv2d_depthwise_column_kernel<K, K, 1, K == 3 ? 8 : 4>
                             : p.rows == 4 ? conv2d_depthwise_column_kernel<K, K, 1, 4>
                                           : conv2d_depthwise_column_kernel<K, K, 1, 2>)
                          : (p.rows == 4 ? conv2d_depthwise_column_kernel<K, K, 2, 4> : conv2d_depthwise_column_kernel<K, K, 2, 2>);
    const cudaError_t e = tc_host::launch_pdl(kern, dim3((unsigned)((p.items + 255) / 256)), dim3(256), 0, st, g, X, W, B, R, Y,
                                              (unsigned)p.items, (unsigned)p.PG, conv_divisor(g.Q), conv_divisor((int)p.PG),
                                              conv_divisor(g.C), conv_divisor(g.dh));
    count_launch();
    return (int)e;
}

// Every input and output row starts on a 16-byte boundary, as far as the sizes tell.
bool depthwise_rows_vectorised(const ConvGeom &g) { return g.pl == (g.kW - 1) / 2 && g.W % 4 == 0 && g.Q == g.W; }

// Where both kernels serve rows that are not: the strips' loads per output are fewer (2.25 against 3.75 at 3x3), the
// columns' threads more and their lines per load a quarter.  3x3: 64 planes of 74x74 6.3 -> 2.8 us, 33 of 177x226 7.2 ->
// 5.8, but 1170 of 59x59 12.5 -> 14.5; 5x5: 192 planes of 17x17 4.2 -> 2.8, but 800 of 51x39 10.4 -> 11.9.
bool depthwise_columns_first(const ConvGeom &g) { return (long long)g.N * g.C * g.P * g.Q < (g.kH == 3 ? 2000000 : 500000); }

template <int KH, int KW>
int launch_depthwise_unit(const ConvGeom &g, const float *X, const float *W, const float *B, const float *R, float *Y,
                          cudaStream_t st) {
    // four output rows per thread where that still gives every SM a few thousand threads, else two
    const bool rows4 = (long long)g.N * g.C * ((g.P + 3) / 4) * ((g.Q + 3) / 4) >= 148LL * 2048 * 2;
    const int rows = rows4 ? 4 : 2;
    const unsigned Q4 = (unsigned)((g.Q + 3) / 4), P2 = (unsigned)((g.P + rows - 1) / rows);
    const long long items = (long long)g.N * g.C * P2 * Q4;
    const unsigned blocks = (unsigned)((items + 255) / 256);
    // aligned 16-byte accesses: every input and output row starts on a 16-byte boundary
    const bool vec = depthwise_rows_vectorised(g) &&
                     (reinterpret_cast<uintptr_t>(X) & 15) == 0 && (reinterpret_cast<uintptr_t>(Y) & 15) == 0;
    // Planes per copy: a strip for every thread, and not many threads without one (56x56 has 196: 38.7 -> 39.4 us); several
    // units for every CTA, or the ring has nothing to run ahead of.  A 5x5 window does not leave room for four CTAs.
    const long long planes = (long long)g.N * g.C, plane_bytes = (long long)g.H * g.W * 4;
    const long long per = std::max(1LL, std::min(256LL / (P2 * Q4), kRingStageMax / plane_bytes)), strips = per * P2 * Q4;
    if (KH == 3 && KW == 3 && vec && rows4 && plane_bytes <= kRingStageMax && strips >= 224 && strips <= 256 &&
        planes >= per * 148 * kRingCtas * 2) {
        unsigned int *err = device_status_ptr();
        if (!err) return (int)cudaErrorUnknown;
        auto ring = conv2d_depthwise_ring_kernel;
        const cudaError_t ae = cudaFuncSetAttribute(ring, cudaFuncAttributeMaxDynamicSharedMemorySize, kRingStages * kRingStageMax);
        if (ae != cudaSuccess) return (int)ae;
        const unsigned units = (unsigned)((planes + per - 1) / per);
        const cudaError_t e = tc_host::launch_pdl(ring, dim3(std::min(units, 148u * kRingCtas)), dim3(256), (size_t)(kRingStages * per * plane_bytes), st,
                                                  g, X, W, B, R, Y, (unsigned)planes, (unsigned)per, Q4, P2, conv_divisor((int)Q4),
                                                  conv_divisor((int)P2), conv_divisor(g.C), err);
        count_launch();
        return (int)e;
    }
    auto kern = vec ? (rows4 ? conv2d_depthwise_unit_kernel<KH, KW, true, 4> : conv2d_depthwise_unit_kernel<KH, KW, true, 2>)
                    : (rows4 ? conv2d_depthwise_unit_kernel<KH, KW, false, 4> : conv2d_depthwise_unit_kernel<KH, KW, false, 2>);
    // early launch gains 0.5 us behind another kernel where the rows are vectorised, and loses as much where not
    if (vec) {
        const cudaError_t e = tc_host::launch_pdl(kern, dim3(blocks), dim3(256), 0, st, g, X, W, B, R, Y, (unsigned)items, Q4, P2,
                                                  1.0 / (double)Q4, 1.0 / (double)P2);
        count_launch();
        return (int)e;
    }
    kern<<<blocks, 256, 0, st>>>(g, X, W, B, R, Y, (unsigned)items, Q4, P2, 1.0 / (double)Q4, 1.0 / (double)P2);
    count_launch();
    return (int)cudaGetLastError();
}

bool depthwise_unit_fits(const ConvGeom &g) {
    if (!(g.Cg == 1 && g.Mg == 1 && g.sh == 1 && g.sw == 1 && g.dh == 1 && g.dw == 1)) return false;
    if (!((g.kH == 3 && g.kW == 3) || (g.kH == 5 && g.kW == 5))) return false;
    const long long items = (long long)g.N * g.C * ((g.P + 1) / 2) * ((g.Q + 3) / 4);
    return items < (1LL << 31) - 256;
}

void depthwise_window(const ConvGeom &g, int &rows, int &cols, int &pitch) {
    rows = (kDwTP - 1) * g.sh + (g.kH - 1) * g.dh + 1;
    cols = (kDwTQ - 1) * g.sw + (g.kW - 1) * g.dw + 1;
    pitch = cols | 1;                          // odd pitch: strided column reads stay conflict-free
}

}  // namespace

static size_t small_smem(const ConvGeom &g, int mb) {
    const long long Hp = (long long)(g.P - 1) * g.sh + (long long)(g.kH - 1) * g.dh + 1, Wp = (long long)(g.Q - 1) * g.sw + (long long)(g.kW - 1) * g.dw + 1;
    const long long taps = (long long)g.kH * g.kW;
    if (Hp * Wp > 16384 || taps > 4096 || g.Cg > 16384) return (size_t)-1;
    return (size_t)g.Cg * 4 * (Hp * Wp + (mb == 1 ? (taps + 3) / 4 * 4 : taps * mb));
}
// Blocks of a problem with mb channels each, or a negative number where the kernel does not apply.
static long long small_blocks(const ConvGeom &g, int mb) {
    if (small_smem(g, mb) > (size_t)kSmallSmem || (long long)g.P * g.Q > 4096) return -1;
    const long long ptiles = ((long long)g.P * g.Q + kSmallThreads - 1) / kSmallThreads;
    const long long blocks = (long long)g.N * g.group * ((g.Mg + mb - 1) / mb) * ptiles;
    return blocks > 1000000 ? -1 : blocks;
}
// Estimated SM cycles against the other kernels', or a negative number where the kernel does not apply: with as many channels per
// block as still leave every SM two blocks.
double small_conv_cost(const ConvGeom &g) {
    const long long ptiles = ((long long)g.P * g.Q + kSmallThreads - 1) / kSmallThreads;
    int mb = 16;
    for (; mb >= 4; mb /= 2)
        if (g.Mg > mb / 2 && (long long)g.N * g.group * ((g.Mg + mb - 1) / mb) * ptiles >= 148 * 2) break;
    if (mb < 4) mb = 1;
    const long long blocks = small_blocks(g, mb);
    if (blocks < 0) return -1;
    // One wave of resident blocks: the loads come in batches of eight per thread, each a trip to L2, then the sum;
    // and no less than what an SM's blocks need in turn (measured: 100 cycles per element a thread brings in).
    const size_t smem = small_smem(g, mb);
    const double kred = (double)g.Cg * g.kH * g.kW, per_sm = (double)((blocks + 147) / 148);
    const double unrolled = g.kH == g.kW && (g.kH == 3 || g.kH == 5) ? 1.0 : 2.5;
    const double fill = (double)smem / 4 / kSmallThreads;
    const double resident = std::min(16.0, 200e3 / (double)(smem + 1024)), waves = std::max(1.0, per_sm / resident);
    const double latency = waves * (fill / 8 * 700.0 + kred * 9.0 * unrolled);
    const double issue = per_sm * (fill * 100.0 + kred * unrolled * (mb == 1 ? 3.0 : 1.5 + 2.2 * mb));
    return 5500.0 + std::max(latency, issue);
}
// Channels per block of a problem that comes here, fitted to MNIST's layers at batch 1 to 200: what a block takes by itself, and half of
// that for every other block on its SM (0.4 with eight channels and more).  (By the rule above the second layer at batch 18, 576 blocks of
// one channel, brings every image in sixteen times: 7.5 us, 4.5 with four channels, 6.3 with eight.)  Of 93 layers of other shapes (1 to
// 12 channels, 3x3 to 7x7, images of 8x8 to 48x48, batch 1 to 256) it picks within 8 % of the best in 84 and 23 % off at most
// (16 -> 32 channels 3x3 8x8 in two groups at batch 100: 5.0 us with four, 4.1 with eight).
int small_conv_channels(const ConvGeom &g) {
    int best = 1, pinned = 0;                                // ONNXB_FP32 = "small,channels" pins them, too
    double cost = -1;
    if (const char *pin = getenv("ONNXB_FP32")) sscanf(pin, "small,%d", &pinned);
    const double kred = (double)g.Cg * g.kH * g.kW * (g.kH == g.kW && (g.kH == 3 || g.kH == 5) ? 1.0 : 2.5);
    for (int mb : {1, 4, 8, 16}) {
        const long long blocks = (pinned ? mb == pinned : mb == 1 || g.Mg > mb / 2) ? small_blocks(g, mb) : -1;
        if (blocks < 0) continue;
        const double one = (double)small_smem(g, mb) / 4 / kSmallThreads / 8 * 900.0 + kred * (mb <= 4 ? 18.0 : 60.0);
        const double c = one * (1.0 + (mb <= 4 ? 0.5 : 0.4) * (double)((blocks + 147) / 148 - 1));
        if (cost < 0 || c < cost) {
            cost = c;
            best = mb;
        }
    }
    return best;
}

int launch_small_conv(const ConvGeom &g, const float *X, const float *W, const float *B, const float *R, float *Y, void *stream) {
    const int mb = g.small_mb, taps = g.kH * g.kW;
    const int Hp = (g.P - 1) * g.sh + (g.kH - 1) * g.dh + 1, Wp = (g.Q - 1) * g.sw + (g.kW - 1) * g.dw + 1;
    const long long ptiles = ((long long)g.P * g.Q + kSmallThreads - 1) / kSmallThreads;
    const long long blocks = (long long)g.N * g.group * ((g.Mg + mb - 1) / mb) * ptiles;
    const int k = g.kH == g.kW && (g.kH == 3 || g.kH == 5) ? g.kH : 0;
    const bool rows = (Wp + 3) % 32 < 4 && blocks > 3LL * tc_host::num_sms();
    auto pick = [&](auto channels) {
        constexpr int MB = decltype(channels)::value;
        if (rows) return k == 3 ? conv2d_small_kernel<MB, 3, true> : k == 5 ? conv2d_small_kernel<MB, 5, true> : conv2d_small_kernel<MB, 0, true>;
        return k == 3 ? conv2d_small_kernel<MB, 3, false> : k == 5 ? conv2d_small_kernel<MB, 5, false> : conv2d_small_kernel<MB, 0, false>;
    };
    auto kern = mb == 1   ? pick(std::integral_constant<int, 1>())
                : mb == 4 ? pick(std::integral_constant<int, 4>())
                : mb == 8 ? pick(std::integral_constant<int, 8>())
                          : pick(std::integral_constant<int, 16>());
    // Blocks placed while the previous kernel still holds its SMs crowd on those that happen to have room: so much shared memory is
    // asked for that no SM takes more than its share.  MNIST from a graph at batch 18 33.0 -> 11.4 us, at batch 39 43.1 -> 16.1 (with the
    // channels per block above).  From 148 blocks on in place of 100, the second layer of four images and a 1x1 layer behind it took 12.4
    // us for 8.1; from the first on nothing is gained, and two streams lose (5.6 -> 5.9 for a layer each); to 16 per SM: no difference.
    size_t smem = small_smem(g, mb);
    const long long sms = tc_host::num_sms(), share = (blocks + sms - 1) / sms;
    if (blocks > 100 && share <= 8) {
        smem = std::max(smem, smem_for_share(share));
        const cudaError_t ae = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (ae != cudaSuccess) return (int)ae;
    }
    const cudaError_t e = tc_host::launch_pdl(kern, dim3((unsigned)blocks), dim3(kSmallThreads), smem, (cudaStream_t)stream, g, X, W, B, R, Y, Hp, Wp,
                                              conv_divisor(Wp), conv_divisor(Hp), conv_divisor(g.Q), conv_divisor(taps));
    count_launch();
    return (int)e;
}

bool simt_depthwise_supports(const ConvGeom &g) {
    if (!(g.Cg == 1 && g.Mg == 1)) return false;
    int rows, cols, pitch;
    depthwise_window(g, rows, cols, pitch);
    const long long floats = (long long)rows * pitch + (long long)g.kH * g.kW;
    if (floats * 4 > 96 * 1024) return false;
    const long long q_tiles = (g.Q + kDwTQ - 1) / kDwTQ, p_tiles = (g.P + kDwTP - 1) / kDwTP;
    return q_tiles * p_tiles * (long long)g.N * g.C <= 2147483647LL;
}

int launch_gather1x1(const ConvGeom &g, const float *X, float *Xg, long long pitch, bool merged, const float *W, float *Wr, long long w_count, void *stream) {
    const RoundedCopy w{reinterpret_cast<const float4 *>(W), reinterpret_cast<float4 *>(Wr), W ? (unsigned)(w_count / 4) : 0u};
    const long long total = merged ? (long long)g.C * pitch : (long long)g.N * g.C * pitch;
    cudaStream_t st = (cudaStream_t)stream;
    const long long total4 = total / 4;                       // every pitch is a multiple of four
    // (for the weights of the call, too, which outnumber the pixels in wide layers on few of them: 52 blocks for the pixels of one image
    // of 14x14 took 40 turns for 1024 -> 2048 channels' weights, 18.4 us in all; 9.3 by a turn's worth of blocks, 11.5 with a launch
    // of its own for the weights; 512 -> 2048 on 7x7 15.8, 7.8, 8.6; 2048 -> 2048 7x7/2 35, 10.8, 12.1)
    const long long for_pixels = (total4 + 255) / 256;
    const unsigned blocks = (unsigned)std::min<long long>(std::max<long long>(for_pixels, (w.n4 + 255) / 256), 148LL * 8);
    // A small copy is set up beside the previous kernel's tail (one image, 7x7 to 28x28: 1.0-1.3 us less).  The blocks of a
    // large one, placed while that kernel still holds its SMs, would crowd on some of them (batch 32: 15 -> 22 us); those of the
    // weights, a turn or a few each, may (plainly launched 1024 -> 2048 14x14/2 at one to four images 10.3 to 14.4 us, early 9.3 to 12.6).
    auto launch = [&](auto kernel, auto... args) {
        if (for_pixels <= 2 * 148) return tc_host::launch_pdl(kernel, dim3(blocks), dim3(256), 0, st, args...);
        kernel<<<blocks, 256, 0, st>>>(args...);
        return cudaGetLastError();
    };
    cudaError_t e;
    if (!merged && g.Q % 4 == 0 && g.W % 4 == 0 && (g.sw == 1 || g.sw == 2) && g.Q * g.sw <= g.W) {
        const unsigned PQ4 = g.P * g.Q / 4, Q4 = g.Q / 4, HW4 = g.H * g.W / 4, rowstep4 = g.sh * g.W / 4;
        e = launch(g.sw == 1 ? gather1x1_vec_kernel<1> : gather1x1_vec_kernel<2>, reinterpret_cast<const float4 *>(X),
                   reinterpret_cast<float4 *>(Xg), (unsigned)total4, PQ4, Q4, HW4, rowstep4, conv_divisor((int)PQ4), conv_divisor((int)Q4), w);
    } else {
        e = launch(gather1x1_quad_kernel, X, reinterpret_cast<float4 *>(Xg), (unsigned)total4, (unsigned)pitch,
                   (unsigned)(merged ? g.N * g.P * g.Q : g.P * g.Q), (unsigned)(g.P * g.Q), (unsigned)g.Q, (unsigned)g.C,
                   (unsigned)(g.H * g.W), (unsigned)(g.sh * g.W), (unsigned)g.sw, merged ? 1 : 0, conv_divisor((int)pitch),
                   conv_divisor(g.P * g.Q), conv_divisor(g.Q), w);
    }
    count_launch();
    return (int)e;
}

int launch_simt_depthwise(const ConvGeom &g, const float *X, const float *W, const float *B, const float *R, float *Y,
                          void *stream) {
    const bool unit = depthwise_unit_fits(g);
    if (depthwise_column_fits(g) && (!unit || (!depthwise_rows_vectorised(g) && depthwise_columns_first(g))))
        return g.kH == 3 ? launch_depthwise_column<3>(g, X, W, B, R, Y, (cudaStream_t)stream)
                         : launch_depthwise_column<5>(g, X, W, B, R, Y, (cudaStream_t)stream);
    if (unit) {
        if (g.kH == 3) return launch_depthwise_unit<3, 3>(g, X, W, B, R, Y, (cudaStream_t)stream);
        return launch_depthwise_unit<5, 5>(g, X, W, B, R, Y, (cudaStream_t)stream);
    }
    int rows, cols, pitch;
    depthwise_window(g, rows, cols, pitch);
    const int q_tiles = (g.Q + kDwTQ - 1) / kDwTQ, p_tiles = (g.P + kDwTP - 1) / kDwTP;
    const size_t smem = ((size_t)rows * pitch + (size_t)g.kH * g.kW) * sizeof(float);
    if (smem > 48 * 1024) {
        const cudaError_t e =
            cudaFuncSetAttribute(conv2d_depthwise_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
        if (e != cudaSuccess) return (int)e;
    }
    const unsigned blocks = (unsigned)((long long)q_tiles * p_tiles * g.N * g.C);
    conv2d_depthwise_kernel<<<blocks, kDwThreads, smem, (cudaStream_t)stream>>>(g, X, W, B, R, Y, q_tiles, p_tiles, rows,
                                                                              cols, pitch);
    count_launch();
    return (int)cudaGetLastError();
}

}  // namespace onnxb
