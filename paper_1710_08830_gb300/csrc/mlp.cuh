// Interface of the network's tensor-core GEMMs (k_mlp_tc.cu) to its passes (k_mlp.cu).
#pragma once

#include <cuda_runtime.h>

namespace tufrg {

// Element-wise sources of a GEMM operand: element (r, c) at r ld + c of row-major buffers.
enum { MLP_F32 = 0,      // S (FP32)
       MLP_GELU = 1,     // GELU(S)
       MLP_BF16 = 2,     // S (BF16)
       MLP_DGELU = 3,    // S GELU'(S2): the upstream gradient S through the activation at S2
       MLP_MSE = 4 };    // 2 (S - S2) scale: the gradient of scale * sum (S - S2)^2
struct MlpSrc {
    const void *S;
    const float *S2;
    int ld, trans;       // trans: the operand is the transpose of the buffer
    int mode;
    float scale;
};

// C[M][N] = A B (+ bias): A as M rows (element (m, k); trans: buffer [K][M]), B as N rows (element (n, k); trans: buffer
// [K][N]).  BF16 kind: both operands rounded to BF16; FP32 kind: A in FP32, B exact in BF16.
struct MlpGemm {
    MlpSrc A, B;
    float *C;
    int M, N, K;
    const float *bias;
};

// Partial column sums of a source (and, for MLP_MSE, partial sums of (S - S2)^2) formed beside the packing.
struct MlpSums {
    MlpSrc src;
    int rows, cols;
    float *part;         // [mlp_sum_parts(rows)][cols]
    double *loss_part;   // [mlp_loss_parts(rows, cols)] (MLP_MSE)
};

size_t mlp_tc_scratch_bytes(int M, int N, int K);
int mlp_sum_parts(int rows);
int mlp_loss_parts(int rows, int cols);
// one or two GEMMs whose operands share one packing launch and one GEMM launch; every kernel returns at once while
// *skip != 0
cudaError_t mlp_gemms(cudaStream_t s, bool fp32, const MlpGemm *g, int n, const MlpSums *sums, const int *skip, void *ws,
                      size_t ws_bytes, int *err);
// bias gradients of all layers and the loss (times inv_n) from the partial sums
cudaError_t mlp_finish(cudaStream_t s, int n_layers, const int *dout, float *const *part, float *const *db, int n_part,
                       const double *loss_part, int n_loss, double inv_n, float *loss);

}  // namespace tufrg
