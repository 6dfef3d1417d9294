// tcgen05 GEMM, operand layout "wgrad" (see des_tc_gemm.cuh).
#include "des_tc_gemm.cuh"
DES_DEFINE_TC_GEMM(TcGemm_wgrad, cutlass::layout::ColumnMajor, cutlass::layout::RowMajor, 128, 64)
DES_DEFINE_TC_GEMM(TcGemm_wgrad_wide, cutlass::layout::ColumnMajor, cutlass::layout::RowMajor, 256, 256)
int des_tc_gemm_wgrad(bool wide, int M, int N, int K, int L, const void* A, const void* B, const float* C, float* D, float beta,
                      void* ws, size_t ws_bytes, cudaStream_t stream) {
  if (wide) { DES_TC_GEMM_BODY(TcGemm_wgrad_wide) }
  DES_TC_GEMM_BODY(TcGemm_wgrad)
}
