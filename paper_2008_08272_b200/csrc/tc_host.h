// Host-side interface of the tensor-core family.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <algorithm>
#include <cstdint>

#include "common.h"

namespace onnxb {

// D[b] (M x N) = A'[b] (M x K) * B'[b] (K x N); Y = relu?(alpha*D + beta*C + row_bias).
// An operand is "MN-major" when its row (A') / column (B') index is the contiguous one.
// ld = element stride of the non-contiguous axis, bs = element stride between batches.
struct TcGemmProblem {
    int M, N, K, batch;
    const float *A, *B;
    int a_mn_major, b_mn_major;
    long long a_ld, b_ld, a_bs, b_bs;
    int a_batched, b_batched;
    float alpha, beta;
    const float *C;
    long long c_si, c_sj;
    const float *row_bias;
    const float *residual;   // optional addend with Y's own layout, added before Relu (ignored when C is given)
    // A residual read at every r_col-th place of every so-many-th row of its own images instead (r_q > 0: pixels in a row of the
    // output): planes r_ld elements apart, images r_bs, the rows that are read r_row, the places r_col.
    int r_q;
    int r_split;             // columns are the pixels of images of so many (0: of one image, the batch's)
    long long r_ld, r_bs;
    int r_row, r_col;
    float *Y_rounded;        // a second output of a layer with a residual, laid out like Y: Y rounded to TF32; may be NULL
    int relu;
    int round_operands;      // A and B are raw fp32: the split-K form rounds them itself, the other form is given copies
    float *Y;
    long long y_ld, y_bs;
    // When y_split > 0 the N columns are `y_split`-wide groups laid y_group_stride elements apart in Y
    // (column j lives at (j / y_split) * y_group_stride + j % y_split of its row): the pixels of several
    // NCHW images contracted as one wide GEMM.
    int y_split;
    long long y_group_stride;
};

bool tc_gemm_supports(const TcGemmProblem &g);
int launch_tc_gemm(const TcGemmProblem &g, void *stream);
// Split-K form for few output tiles (tc_gemm_splitk.cu); launch_tc_gemm uses it where it fits.
double tc_gemm_estimate_ns(const TcGemmProblem &g);       // the persistent kernel's estimated time
double tc_gemm_prepass_ns(const TcGemmProblem &g);        // and that of the launch that rounds ONNX Gemm's operands in front of it
bool tc_gemm_splitk_fits(const TcGemmProblem &g);
int launch_tc_gemm_splitk(const TcGemmProblem &g, void *stream);

// Shared memory to launch a CTA with that uses `smem` bytes of it and allocates `columns` of TMEM (128, 256 or 512).
// tcgen05.alloc waits for columns without limit, and the CTAs of a cluster wait for one another with theirs held: two
// clusters of different streams could each hold on one SM what the other waits for on another.  So no CTA is to find too
// little, or what there is in pieces: one that allocates a quarter of TMEM reserves so much shared memory that five do not
// fit an SM, one that allocates more so much that it does not fit beside another of either kind.  (At present their
// registers rule both out as well, and nearly every launch uses more anyway.)
constexpr size_t kSmemPerSm = 228 * 1024, kSmemPerCta = 1024;        // (the second: what the system adds for each CTA)
constexpr size_t kSmemQuarterTmem = 46 * 1024, kSmemMoreTmem = 184 * 1024;
static_assert(5 * (kSmemQuarterTmem + kSmemPerCta) > kSmemPerSm, "five quarters of TMEM on one SM");
static_assert(kSmemMoreTmem + kSmemQuarterTmem + 2 * kSmemPerCta > kSmemPerSm, "more than TMEM on one SM");
inline size_t smem_with_tmem(size_t smem, uint32_t columns) { return std::max(smem, columns <= 128 ? kSmemQuarterTmem : kSmemMoreTmem); }

// The least shared memory of a block of which no more than `share` fit an SM: what is left is for other kernels' blocks, of the next
// launch or of another stream (with all that lets `share` fit, a fp32 Gemm beside a small-image convolution took 15.0 us for the two,
// 13.9 so).
inline size_t smem_for_share(long long share) { return (size_t)(kSmemPerSm / (share + 1) - kSmemPerCta) / 128 * 128 + 128; }

// Address of the device error word of the current device (NULL on failure).
unsigned int *device_status_ptr();

namespace tc_host {
// Launch `kernel` so that it may begin (up to its pdl_wait()) before the previous kernel of the stream
// has finished.  Returns the cudaError_t of the launch.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                              Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// The same for a kernel launched as clusters of `cluster_x` CTAs along x (grid.x a multiple of it).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl_cluster(void (*kernel)(KArgs...), unsigned cluster_x, dim3 grid, dim3 block, size_t smem,
                                      cudaStream_t st, Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster_x;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

constexpr int kTmapSwizzleNone = 0, kTmapSwizzle128 = 1, kTmapSwizzle128Atom32 = 2;
bool make_tmap(CUtensorMap *out, const void *base, int rank, const uint64_t *dims, const uint64_t *strides_bytes,
               const uint32_t *box, int swizzle);
int num_sms();
}  // namespace tc_host

}  // namespace onnxb
