// Geometry of the implicit-GEMM convolution kernel, shared by host planning and
// device code (plain integer arithmetic, no CUDA types).
//
// "Slot space".  For every image the kernel lays the (zero-padded, stride-decimated)
// input out as a grid of Hs x Ws slots per parity plane; slot (hq, wq) of plane (a, b)
// holds the padded input pixel (hq*sh + a, wq*sw + b).  Output pixel (p, q) is anchored
// at slot u = p*Ws + q, and filter tap (r, s) reads plane ((r*dh) % sh, (s*dw) % sw) at
// slot u + ((r*dh)/sh)*Ws + (s*dw)/sw: a fixed shift per tap.  Images follow each other
// every L = Hs*Ws slots, so a GEMM row tile is simply 128 consecutive global slots, and
// the im2col operand of a tap is the same shared-memory tile read from a shifted start
// address.  Hs and Ws are chosen as small as possible: the trailing zero padding of one
// row (image) is allowed to alias the leading zero padding of the next.
#pragma once
#include <algorithm>
#include <cstdint>

#if defined(__CUDACC__)
#define ONNXB_HD __host__ __device__
#else
#define ONNXB_HD
#endif

namespace onnxb {

constexpr int kConvMaxPlanes = 4;
constexpr int kConvMaxTaps = 64;
constexpr int kConvMaxSteps = 128;     // MMA K-steps (8 reduction terms each) per channel block
constexpr int kConvMaxSeg = 8;

struct ConvDivisor {
    uint32_t d, m, s1, s2;
};

struct TcConvPlan {
    // problem
    int N, C, H, W, M, Cg, Mg, kH, kW, P, Q, pt, pl, sh, sw, dh, dw, group, relu;
    // slot space
    int Hs, Ws, L;
    long long total_slots;           // N * L
    int planes, pa[kConvMaxPlanes], pb[kConvMaxPlanes];
    int a_min, a_max;                // smallest / largest used row parity
    int taps;
    // Reduction blocking.  A channel block holds KB input channels as KB/4 chunks of 4 (one 16-byte
    // operand row per slot and chunk).  One MMA K-step consumes two chunks:
    //   KB = 16 ("channel pairs"): chunks 2j, 2j+1 of the same tap, two steps per tap;
    //   KB = 4  ("tap pairs", for C/group < 16): the single chunk read at two taps of the same plane.
    int KB, nchunks, n_steps;
    int chunk_groups, chunks_per_unit;   // how the re-lay splits a slot's chunks over threads: nchunks = groups x per unit
    uint32_t step_a[kConvMaxSteps];      // A descriptor low word relative to the stage: offset/16 | (LBO/16) << 16
    short src_tap[kConvMaxSteps][2];     // which filter tap feeds chunk 0 / 1 of the step's weights (-1: zeros)
    short src_c0[kConvMaxSteps][2];      // and from which channel offset inside the block
    // tiling
    int ctas;                        // CTAs working on one tile: 1, or 2 (a cluster pair issuing M = 256 MMAs)
    int MT;                          // 128-row accumulator tiles per CTA (1 or 2)
    int BN, ctiles;                  // output channels per tile, tiles per group
    int BNH;                         // weight rows each CTA stages per K-step = BN / ctas
    int SLOTS;                       // slots per plane held in one A stage = MT*128 + largest tap shift
    int ncb;                         // channel blocks = ceil(Cg / KB)
    int pix_tiles;                   // ceil(total_slots / (ctas*MT*128))
    long long total_tiles;
    // raw staging
    int raw_mode;                    // 0: tensor-map boxes [KB][BOXP] over X seen as (H*W, N*C); 1: whole-image slabs;
                                     // 2: one copy of rows per channel, [channel][BOXP]
    // X is channel-major: raw_mode 0 over X seen as (images x H*W, C).  The images that a tile touches follow one another there,
    // so its pixels are one range, and a few boxes bring several small images that slabs or boxes of each took a copy for.
    int x_cm;
    uint32_t y_image4, y_chan4;      // bytes from one image of Y (and R) to the next, and from one channel
    int BOXP;
    int KBR;                         // channels staged per block: KB, or all of a group's if it has fewer
    // shared memory carve-up (bytes)
    int a_stage_bytes, raw_stage_bytes, b_stage_bytes, nb_stages, nr_stages, na_stages;
    int spb, b_step_bytes, b_steps;  // K-steps per weight stage, bytes of one step's weights, weight stages per block
    int chunk_pitch, plane_pitch;    // bytes between 4-channel chunks / parity planes inside an A stage
    uint32_t idesc;
    long long packed_floats;         // size of the packed weight buffer
    // divisors device code needs per slot, as multiply-and-shift constants (see conv_fdiv)
    ConvDivisor dv_L, dv_Ws, dv_Hs, dv_BOXP, dv_SLOTS, dv_pss;
    int boxp_shift;                  // log2(BOXP) when BOXP is a power of two, else -1
    int split, cb_per;               // CTAs (a cluster) sharing a tile's channel blocks, blocks of each; split = 1: none
    int cols_per;                    // split: output channels of the tile that each CTA finishes, a multiple of 4
    int b_resident;                  // all tiles use the same few weights: fetched once per CTA
    int relay;                       // pairs: the odd CTA's "operand stage written" goes through its relay warp
};

// floor(n / d) for any 32-bit unsigned n.  On the device: the round-up multiply-and-shift method
// (Granlund and Montgomery, "Division by invariant integers using multiplication"): with
// l = ceil(log2 d) and m = floor(2^32 (2^l - d) / d) + 1, t = high32(m * n) and
// q = (t + ((n - t) >> min(l, 1))) >> max(l - 1, 0).  On the host: plain division.
// (The host passes the divisor itself: while a plan is being filled its constants are not yet set.)
ONNXB_HD inline int conv_fdiv(int n, int d, const ConvDivisor &dv) {
#if defined(__CUDA_ARCH__)
    (void)d;
    const uint32_t un = (uint32_t)n, t = __umulhi(dv.m, un);
    return (int)((t + ((un - t) >> dv.s1)) >> dv.s2);
#else
    (void)dv;
    return (int)((uint32_t)n / (uint32_t)d);
#endif
}
inline ConvDivisor conv_divisor(int d) {
    ConvDivisor dv;
    dv.d = (uint32_t)d;
    int l = 0;
    while ((1ull << l) < (unsigned long long)d) ++l;
    dv.m = (uint32_t)(((1ull << 32) * ((1ull << l) - (unsigned long long)d)) / (unsigned long long)d + 1);
    dv.s1 = l < 1 ? (uint32_t)l : 1u;
    dv.s2 = l > 1 ? (uint32_t)(l - 1) : 0u;
    return dv;
}

struct ConvAxis {
    int E, Amax, npar, par[kConvMaxPlanes];
};

// Slot extent along one axis: input size I, output size O, leading pad, stride s, dilation d, kernel k.
inline bool conv_plan_axis(int I, int O, int pad, int s, int d, int k, ConvAxis &ax) {
    int offmax[64];
    bool used[64];
    if (s > 64) return false;
    for (int a = 0; a < s; ++a) { used[a] = false; offmax[a] = 0; }
    ax.Amax = 0;
    for (int t = 0; t < k; ++t) {
        const int a = (t * d) % s, o = (t * d) / s;
        used[a] = true;
        offmax[a] = std::max(offmax[a], o);
        ax.Amax = std::max(ax.Amax, o);
    }
    ax.npar = 0;
    int a_min = -1;
    long long e = O;
    for (int a = 0; a < s; ++a) {
        if (!used[a]) continue;
        if (ax.npar == kConvMaxPlanes) return false;
        ax.par[ax.npar++] = a;
        if (a_min < 0) a_min = a;
        const int z = pad > a ? (pad - a + s - 1) / s : 0;         // leading zero slots of this parity
        e = std::max<long long>(e, (long long)O + offmax[a] - z);
    }
    e = std::max<long long>(e, ((long long)I + pad - a_min + s - 1) / s);
    e = std::min<long long>(e, (long long)O + ax.Amax);
    ax.E = (int)e;
    return true;
}

// Plan of the fp32 kernel (tc_fp32.cu): the same slot space, a tile is 128 consecutive slots and their halo.
constexpr int kFp32MaxPlanes = 16, kFp32MaxSteps = 128, kFp32MaxSeg = 8;
struct Fp32ConvPlan {
    int N, C, H, W, M, Cg, Mg, kW, P, Q, pt, pl, sh, sw, dh, dw, group, taps;
    int Hs, Ws, L, planes, SLOTS;        // slots per image; parity planes; slots of a plane in a stage
    int a_min, a_max;                    // smallest / largest used row parity
    int tiles_r, per_image;              // pixel tiles; of each image, or 0 where a tile may hold parts of several
    int pitch;                           // floats from one channel's staged rows to the next's, congruent to H*W modulo 4
    short pa[kFp32MaxPlanes], pb[kFp32MaxPlanes];
    int nch, ncb;                        // four-channel chunks per block, blocks
    int n_steps, n_groups, spg;          // K-steps of a block, and the partial sums they form
    int BN, tiles_c, split;
    uint32_t step_a[kFp32MaxSteps];      // slot of the step's first chunk in the stage | distance of its second << 16
    short src_tap[kFp32MaxSteps][2], src_c0[kFp32MaxSteps][2];
    ConvDivisor dv_L, dv_Ws, dv_slots, dv_SLOTS, dv_per_image;
};
// First slot of a pixel tile.
ONNXB_HD inline int fp32_conv_first_slot(const Fp32ConvPlan &g, int rt) {
    if (!g.per_image) return rt * 128;
    const int n = conv_fdiv(rt, g.per_image, g.dv_per_image);
    return n * g.L + (rt - n * g.per_image) * 128;
}
// The rows of the images that a tile's slots lie in: where each image's begin in X's plane and in a channel's staged rows.
struct Fp32ConvSegs {
    int n_first, nseg;
    int f0[kFp32MaxSeg], len[kFp32MaxSeg], at[kFp32MaxSeg];
};
ONNXB_HD inline void fp32_conv_segments(const Fp32ConvPlan &g, int rt, int grp, Fp32ConvSegs &t) {
    const long long G0 = fp32_conv_first_slot(g, rt), all = (long long)g.N * g.L, end = G0 + g.SLOTS < all ? G0 + g.SLOTS : all;
    t.n_first = conv_fdiv((int)G0, g.L, g.dv_L);
    t.nseg = conv_fdiv((int)(end - 1), g.L, g.dv_L) - t.n_first + 1;
    int at = 4;                          // (a later channel's first copy may start up to three elements before its row)
    for (int i = 0; i < t.nseg; ++i) {
        const long long base = (long long)(t.n_first + i) * g.L;
        const int lo = (int)(G0 > base ? G0 - base : 0), hi = (int)(end < base + g.L ? end - base : g.L);      // [lo, hi)
        int h0 = conv_fdiv(lo, g.Ws, g.dv_Ws) * g.sh + g.a_min - g.pt, h1 = conv_fdiv(hi - 1, g.Ws, g.dv_Ws) * g.sh + g.a_max - g.pt;
        if (h0 < 0) h0 = 0;
        if (h1 > g.H - 1) h1 = g.H - 1;
        t.f0[i] = h0 * g.W;
        t.len[i] = h0 <= h1 ? (h1 - h0 + 1) * g.W : 0;
        // as far from a 16-byte boundary as in X (the pitch keeps that for every channel), and clear of what the copy before,
        // in whole 16-byte pieces, may write
        const int e = ((t.n_first + i) * g.C + grp * g.Cg) * g.H * g.W + t.f0[i];
        t.at[i] = (at + 3) / 4 * 4 + (e & 3);
        at = t.at[i] + t.len[i] + 3;
    }
}
// Where a copy of X that has to reach element `last` (exclusive) ends: a whole number of 16-byte pieces, none past the x_whole
// elements of X that are such pieces.  (The smaller of the two is rounded up: last + 3 may not fit an int.)
ONNXB_HD inline int fp32_conv_copy_end(int last, int x_whole) { return ((last < x_whole ? last : x_whole) + 3) & ~3; }

struct TcConvSegs {
    int n_first, nseg;
    int hq0, wq0;                    // slot row / column of the tile's first slot within image n_first
    int f0[kConvMaxSeg];             // first flat pixel (h*W + w) staged for the image
    int base[kConvMaxSeg];           // float offset of the image's data inside the raw stage
    int nbox[kConvMaxSeg];           // boxes (mode 0) / 1 (mode 1) / pixels (mode 2) / 0 when nothing of the image is needed
    int total_floats;                // of the stage (mode 2: of a channel)
    int one_image;                   // every slot of the tile lies in image n_first
};

// Which part of which images the A stage of the tile starting at global slot G0 needs.
ONNXB_HD inline void tc_conv_segments(const TcConvPlan &g, long long G0, TcConvSegs &t) {
    long long Gend = G0 + g.SLOTS;
    if (Gend > g.total_slots) Gend = g.total_slots;
    if (G0 >= g.total_slots) {       // the second CTA of a pair on the last, half-empty tile
        t.n_first = g.N;
        t.nseg = 0;
        t.hq0 = t.wq0 = 0;
        t.total_floats = 0;
        t.one_image = 0;
        return;
    }
    t.n_first = conv_fdiv((int)G0, g.L, g.dv_L);
    {
        const int u0 = (int)(G0 - (long long)t.n_first * g.L);
        t.hq0 = conv_fdiv(u0, g.Ws, g.dv_Ws);
        t.wq0 = u0 - t.hq0 * g.Ws;
    }
    const int n_last = conv_fdiv((int)(Gend - 1), g.L, g.dv_L);
    t.nseg = n_last - t.n_first + 1;
    if (t.nseg > kConvMaxSeg) t.nseg = kConvMaxSeg;   // excluded by the planner
    t.one_image = t.nseg == 1 && Gend == G0 + g.SLOTS;
    int base = 0;
    int first = -1, end = 0;         // channel-major: the tile's range of pixels, from image n_first's first
    const int HW = g.H * g.W;
    for (int i = 0; i < t.nseg; ++i) {
        const long long n = t.n_first + i;
        const long long lo = G0 > n * g.L ? G0 : n * g.L;
        const long long hi = Gend < (n + 1) * g.L ? Gend : (n + 1) * g.L;
        const int u_lo = (int)(lo - n * g.L), u_hi = (int)(hi - n * g.L);   // [u_lo, u_hi)
        const int hq_lo = conv_fdiv(u_lo, g.Ws, g.dv_Ws), hq_hi = conv_fdiv(u_hi - 1, g.Ws, g.dv_Ws);
        int h_min = hq_lo * g.sh + g.a_min - g.pt;
        int h_max = hq_hi * g.sh + g.a_max - g.pt;
        if (h_min < 0) h_min = 0;
        if (h_max > g.H - 1) h_max = g.H - 1;
        t.base[i] = base;
        if (g.x_cm) {
            t.nbox[i] = 0;
            if (h_min <= h_max) {
                if (first < 0) first = i * HW + h_min * g.W;
                end = i * HW + (h_max + 1) * g.W;
            }
        } else if (h_min > h_max) {
            t.f0[i] = 0;
            t.nbox[i] = 0;
        } else if (g.raw_mode == 1) {
            t.f0[i] = 0;
            t.nbox[i] = 1;
            base += g.KBR * g.H * g.W;
        } else {
            const int f0 = (h_min * g.W) & ~3;
            const int len = (h_max + 1) * g.W - f0;
            t.f0[i] = f0;
            if (g.raw_mode == 2) {
                t.nbox[i] = (len + 3) & ~3;          // (within the plane: H * W is a multiple of 4)
                base += t.nbox[i];
                continue;
            }
            t.nbox[i] = conv_fdiv(len + g.BOXP - 1, g.BOXP, g.dv_BOXP);
            base += t.nbox[i] * g.BOXP * g.KBR;
        }
    }
    if (g.x_cm && first >= 0) {
        // (a copy starts on a 16-byte boundary: up to three pixels of what lies before)
        const int start = (int)(((long long)t.n_first * HW + first) & ~3LL) - t.n_first * HW;
        for (int i = 0; i < t.nseg; ++i) t.f0[i] = start - i * HW;
        t.nbox[0] = conv_fdiv(end - start + g.BOXP - 1, g.BOXP, g.dv_BOXP);
        base = t.nbox[0] * g.BOXP * g.KBR;
    }
    t.total_floats = base;
}

}  // namespace onnxb
