// gemm_grad.cu -- instantiations of the tensor-core GEMM whose epilogue
// multiplies by GELU'(z) (backward pass of the Sec. 3.2 network). The weights are
// read as they lie, [out][in], as the N-major operand of dZ W.
#include "gemm_launch.cuh"

namespace chemgb {
int gemm_gelu_grad(const void *X, int64_t ldx, const void *W, int64_t ldw, int M, int N, int K, const float *z,
                   int64_t ldz, void *out, int64_t ldo, int *err, cudaStream_t st) {
    if (M <= 0 || N <= 0 || K <= 0) return CHEM_OK;
    EpiGeluGrad e{M, N, z, ldz, static_cast<__nv_bfloat16 *>(out), ldo};
    return launch_gemm_grouped_bn<128, 6>(GemmOperand{X, ldx, kMap2D, 0}, GemmOperand{W, ldw, kMap2D, 0}, 1, kMap2D, 0, M,
                                          N, K, e, err, st, 0);
}
int gemm_gelu_grad_grouped(const GemmOperand &X, const GemmOperand &W, int G, int M, int N, int K, const float *z,
                           int64_t ldz, int64_t g_z, void *out, int64_t ldo, int64_t g_out, int *err, cudaStream_t st) {
    if (M <= 0 || N <= 0 || K <= 0 || G <= 0) return CHEM_OK;
    EpiGeluGrad e{M, N, z, ldz, static_cast<__nv_bfloat16 *>(out), ldo, g_z, g_out};
    return launch_gemm_grouped_bn<128, 6>(X, W, G, kMapColGrp, g_out, M, N, K, e, err, st, 0);
}
}  // namespace chemgb
