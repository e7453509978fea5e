// Internal declarations shared by the translation units of libonnx_b200.
#pragma once
#include <atomic>
#include <cstddef>
#include <cstdint>

#include "onnx_b200.h"
#include "tc_conv_plan.h"

namespace onnxb {

// Floats from one channel to the next in a channel-major tensor ([channel][image][row][column]), padded to whole 128-byte lines.
inline long long channel_pitch(long long images, long long h, long long w) { return (images * h * w + 31) / 32 * 32; }

// A convolution problem with every ONNX default and auto_pad already resolved.
struct ConvGeom {
    int x_cm, y_cm;          // X, Y (and R) are channel-major
    int N, C, H, W;          // input
    int M, Cg, kH, kW;       // weights: M output channels, Cg = C/group input channels each
    int P, Q;                // output spatial size
    int pt, pl, pb, pr;      // resolved pads (h_begin, w_begin, h_end, w_end)
    int sh, sw, dh, dw;
    int group, Mg;           // Mg = M/group
    int has_bias, relu;
    int small_mb;            // output channels per block of the small-image kernel,
    double small_cost;       // and its estimate (small_conv_cost)
};

struct Fp32GemmPlan {        // tile width, and CTAs that share a tile's reduction (tc_fp32.cu)
    int BN, split;
};

}  // namespace onnxb

struct onnxb_conv2d_desc_s {
    onnxb::ConvGeom g;
    int family;              // onnxb_kernel_family
    onnxb::TcConvPlan plan;  // valid when family == ONNXB_KERNEL_MMA_IMPLICIT
    // ONNXB_KERNEL_SIMT_DIRECT on the tensor cores where it is given workspace: 1 by the convolution plan below, 2 as a Gemm of
    // packed pixels
    int fp32_tc;
    onnxb::Fp32ConvPlan fp32;
    onnxb::Fp32GemmPlan fp32_gemm;
    size_t workspace_bytes;
    int64_t y_dims[4];
    int64_t pads[4];
};

namespace onnxb {

extern std::atomic<uint64_t> g_launches;
inline void count_launch(int n = 1) { g_launches.fetch_add((uint64_t)n, std::memory_order_relaxed); }

int kernel_override();   // -1 = automatic

// SIMT family (simt_conv.cu / simt_gemm.cu).  All return a cudaError_t as int.
// R (everywhere below): optional addend with Y's shape, added before Relu (a residual connection); may be NULL.
int launch_simt_conv(const ConvGeom &g, const float *X, const float *W, const float *B, const float *R, float *Y,
                     void *stream);
// Whether the convolution belongs on the tensor cores (fp32 by split operands, tc_fp32.cu), and its plan there: the
// descriptor's fp32_tc.
int simt_conv_on_tensor_cores(const ConvGeom &g, Fp32ConvPlan &plan, Fp32GemmPlan &gemm);
int launch_simt_depthwise(const ConvGeom &g, const float *X, const float *W, const float *B, const float *R, float *Y,
                          void *stream);
double small_conv_cost(const ConvGeom &g);           // estimated SM cycles; negative: not for this problem
int small_conv_channels(const ConvGeom &g);          // output channels per block, the descriptor's small_mb
int launch_small_conv(const ConvGeom &g, const float *X, const float *W, const float *B, const float *R, float *Y,
                      void *stream);
bool simt_depthwise_supports(const ConvGeom &g);
bool conv_fits_mma_gemm(const ConvGeom &g);
bool conv_fits_mma_gather_gemm(const ConvGeom &g);   // other unpadded 1x1: gather the pixels read, then the same GEMM
size_t conv_gather_workspace_bytes(const ConvGeom &g);
// (W: weights to round to TF32 into Wr in the same launch, or NULL; their count is a multiple of 4)
int launch_gather1x1(const ConvGeom &g, const float *X, float *Xg, long long pitch, bool merged, const float *W, float *Wr, long long w_count, void *stream);
// implicit-GEMM tensor-core convolution (tc_conv.cu)
bool tc_conv_plan(const ConvGeom &g, TcConvPlan &plan, bool forced = false);
size_t tc_conv_workspace_bytes(const TcConvPlan &plan);
// phase: both steps (pack the weights into the workspace, then convolve), or one of them alone
constexpr int kTcConvPackAndRun = 0, kTcConvPackOnly = 1, kTcConvRunOnly = 2;
int launch_tc_conv(const TcConvPlan &plan, const float *X, const float *W, const float *B, const float *R, float *Y,
                   void *workspace, void *stream, int phase = kTcConvPackAndRun, bool round_y = false);   // 1x1 stride-1 convolution expressible as a batched TMA GEMM

struct GemmProblem {
    int M, N, K;
    int transA, transB;
    float alpha, beta;
    long long c_stride_i, c_stride_j;   // element strides of C along i and j (0 = broadcast)
    int relu;
};
bool simt_gemm_is_tiny(long long M, long long N, long long K);   // small enough for the dot-product kernel
// Scratch with which a Gemm of the fp32 family runs on the tensor cores (0: it does not); without it runs on the FMA units.
size_t simt_gemm_workspace_bytes(int M, int N, int K);
int launch_simt_gemm(const GemmProblem &p, const float *A, const float *B, const float *C, float *Y, void *workspace,
                     size_t workspace_bytes, void *stream);
// fp32 through split TF32 operands on the tensor cores (tc_fp32.cu): the same problems, once they are large.  The
// plans return their estimated SM cycles, the packing launch included for Gemm (negative: no plan).
double tc_fp32_gemm_plan(int M, int N, int K, Fp32GemmPlan &plan);
size_t tc_fp32_gemm_workspace(int M, int N, int K, const Fp32GemmPlan &plan);
int launch_tc_fp32_gemm(const GemmProblem &p, const Fp32GemmPlan &plan, const float *A, const float *B, const float *C, float *Y,
                        void *workspace, void *stream);
int launch_tc_fp32_conv1x1(const ConvGeom &g, const Fp32GemmPlan &plan, const float *X, const float *W, const float *B, const float *R,
                           float *Y, void *workspace, void *stream);
double tc_fp32_conv_plan(const ConvGeom &g, Fp32ConvPlan &plan);
size_t tc_fp32_conv_workspace(const Fp32ConvPlan &plan);
int launch_tc_fp32_conv(const ConvGeom &g, const Fp32ConvPlan &plan, const float *X, const float *W, const float *B, const float *R,
                        float *Y, void *packed, void *stream, int phase);

}  // namespace onnxb
