// Laying out a convolution's weights for the tensor core: [group][channel tile][channel block][K-step][half] of 4 reduction terms
// (channels of the block, at one tap) for every output channel of the tile.
//
// A block takes eight output channels and one channel block: W's rows are read as they lie (a warp a channel), parked in shared
// memory, and written eight channels' 16-byte pieces at a time.  Bound: both tensors' bytes, and for most layers a launch's latency.
// (A thread per piece, lanes along the output channels, read every 4 bytes from another 32-byte sector, and the sectors again for
// every tap: it added 15 us to a convolution of 512 -> 512 channels 3x3, now 6, and 47 to one of 5x5, now 10.)
#pragma once
#include <algorithm>
#include <cstdint>

#include "tc_common.cuh"

namespace onnxb {

constexpr int kPackRows = 8, kPackThreads = kPackRows * 32;
constexpr int kPackFloats = 1024;                 // of an output channel in a channel block: 128 K-steps of 8 terms

// Blocks (x), and blocks that share one's K-steps (y) where the x are fewer than the SMs: each reads the same rows, and 16 steps are
// what its threads write at once (32 -> 48 channels 7x7, 12 blocks and 98 steps: 18.4 -> 17.1 us with its convolution of 62x66).
template <class Plan>
inline dim3 pack_weights_grid(const Plan &g, int tiles, int tile_rows) {
    const long long x = (long long)g.group * tiles * (tile_rows / kPackRows) * g.ncb;
    const long long y = std::min<long long>((g.n_steps + 15) / 16, std::max<long long>(1, 148 / x));
    return dim3((unsigned)x, (unsigned)y);
}

// `tiles` channel tiles of tile_rows (a multiple of 8) channels in a group, `kb` input channels in a block.
// put(index of the tile over all groups, channel block, K-step, half, channel of the tile, its four terms)
template <class Plan, class Put>
__device__ __forceinline__ void pack_weights(const Plan &g, const float *__restrict__ W, int tiles, int tile_rows, int kb, const Put &put) {
    __shared__ float rows[kPackRows][kPackFloats + 4];
    const unsigned octets = (unsigned)(tile_rows / kPackRows);
    unsigned t = blockIdx.x;
    const int cb = (int)(t % (unsigned)g.ncb); t /= (unsigned)g.ncb;
    const int r0 = (int)(t % octets) * kPackRows; t /= octets;
    const int ct = (int)(t % (unsigned)tiles), grp = (int)(t / (unsigned)tiles);
    const int chans = min(kb, g.Cg - cb * kb), warp = (int)threadIdx.x / 32, lane = (int)threadIdx.x % 32;
    tc::pdl_wait();
    {
        const int mg = ct * tile_rows + r0 + warp, len = mg < g.Mg ? chans * g.taps : 0;
        const float *src = W + ((size_t)(grp * g.Mg + mg) * g.Cg + (size_t)cb * kb) * g.taps;
        for (int i0 = lane; i0 < len; i0 += 16 * 32) {
            float v[16];                          // in flight together
#pragma unroll
            for (int k = 0; k < 16; ++k) v[k] = i0 + k * 32 < len ? __ldg(src + i0 + k * 32) : 0.f;
#pragma unroll
            for (int k = 0; k < 16; ++k)
                if (i0 + k * 32 < len) rows[warp][i0 + k * 32] = v[k];
        }
    }
    __syncthreads();
    for (int i = (int)(blockIdx.y * kPackThreads + threadIdx.x); i < g.n_steps * 2 * kPackRows; i += (int)gridDim.y * kPackThreads) {
        const int row = i % kPackRows, half = i / kPackRows & 1, step = i / (2 * kPackRows);
        const int tap = g.src_tap[step][half], c0 = g.src_c0[step][half], mg = ct * tile_rows + r0 + row;
        float v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = mg < g.Mg && tap >= 0 && c0 + e < chans ? rows[row][(c0 + e) * g.taps + tap] : 0.f;
        put((size_t)(grp * tiles + ct), cb, step, half, r0 + row, v);
    }
}

}  // namespace onnxb
