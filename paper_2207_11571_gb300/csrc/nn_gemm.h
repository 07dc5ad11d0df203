// BF16 tensor-core GEMM for sm_103a (tcgen05 + TMA + TMEM), the dense contraction of
// the forcing network (Sec. 2.2, Fig. 2).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace dgnn {

// Epilogue applied to the FP32 accumulator tile C = A B^T:
enum GemmKind {
  kGemmBiasReluBf16 = 0,  // out bf16 = relu(C + bias)              (hidden layer)
  kGemmAffineF32 = 1,     // out f32  = (C + bias) * scale + shift   (output layer; scale/shift may be null)
  kGemmF32 = 2,           // out f32  = C (+ bias if given)
  kGemmLossBf16 = 3,      // output layer of a training step: y = C + bias against the scaled targets,
                          // out bf16 = dL/dy of the MSE, its column sums, the squared errors' sum
  kGemmMaskBf16 = 4       // out bf16 = C * (mask > 0)  (gradient through ReLU), its column sums
};

struct GemmEpilogue {
  int kind = kGemmF32;
  const float* bias = nullptr;
  const float* scale = nullptr;
  const float* shift = nullptr;
  const __nv_bfloat16* mask = nullptr;
  int ldm = 0;
  void* out = nullptr;
  int ldo = 0;
  int relu = 0;  // f32 kinds: apply max(., 0) after the bias
  // gradient kinds: FP32 sums of the unrounded output over each 32 rows, [ceil(M / 32)][N]
  float* colsum = nullptr;
  // kGemmLossBf16: targets Y[idx ? idx[r] : r][N], their scaling, dy = grad_scale (y - t), and
  // partial sums of (y - t)^2, one per epilogue warp and tile (gemm_loss_partials of them)
  const float* Y = nullptr;
  const int64_t* idx = nullptr;
  const float* mean = nullptr;
  const float* sd = nullptr;
  float grad_scale = 0.f;
  double* loss_part = nullptr;
};

// C[M x N] = A[M x K] B[N x K]^T with the given epilogue.  A and B are row-major bf16 with
// leading dimensions lda, ldb (elements, multiples of 8, base 16-byte aligned);
// K is the reduction length: TMA reads columns at or beyond K, and rows beyond M (N),
// as zeros.  err_flag (device int) is set non-zero if a bounded wait inside the kernel
// ran out.  Returns a dg_status.
int gemm_bf16(const __nv_bfloat16* A, int lda, const __nv_bfloat16* B, int ldb, int M, int N, int K,
              const GemmEpilogue& ep, int* err_flag, cudaStream_t st);

// Number of loss partials of a kGemmLossBf16 product.
int gemm_loss_partials(int M, int N);

// Gradient of a layer's input: dx [rows][lda] = bf16(dy W * (act > 0)), with its FP32 column
// sums over each 32 rows, colsum [ceil(rows / 32)][in].  dy [rows][ldy] (o columns), W [o][ldw]
// (in columns), act [rows][lda] (the layer's input): row-major bf16, read as they lie.
int input_gradient(const __nv_bfloat16* dy, int ldy, const __nv_bfloat16* W, int ldw, int rows, int in, int o,
                   const __nv_bfloat16* act, int lda, __nv_bfloat16* dx, float* colsum, int* err_flag,
                   cudaStream_t st);

// Weight gradients of all layers in one launch: dW_l [M_l x N_l] = G_l^T A_l over `rows` rows,
// G_l row-major [rows][ldg] (M_l columns), A_l row-major [rows][lda] (N_l columns), both read
// as they lie.  The rows are cut into grad_splits(M_l, N_l, rows) runs; split z of layer l
// writes its partial product to out + z * split_stride + offset_l.
struct GradLayer {
  const __nv_bfloat16* G;
  const __nv_bfloat16* A;
  int ldg, lda, M, N;
  long long offset;
};
constexpr int kMaxGradLayers = 9;
int weight_gradients(const GradLayer* layers, int L, int rows, float* out, long long split_stride, int* err_flag,
                     cudaStream_t st);
constexpr int kMaxSplits = 8;
int grad_splits(int M, int N, int rows);

// 2D tensor map of a row-major bf16 matrix [rows][cols] (leading dimension ld elements),
// box of 64 columns x box_rows rows with the 128-byte swizzle; cached.  Returns a dg_status.
int make_map(CUtensorMap* map, const __nv_bfloat16* ptr, long long rows, long long cols, long long ld, int box_rows);

}  // namespace dgnn
