// The register form of AAb_Solver for clusters of 16 (see aab_reg.cuh).
#include "aab_reg.cuh"

namespace mihs {
namespace aabk {

RegKernel reg_kernel_16(int m, int dp) { return reg_kernel_cl<16>(m, dp); }

int reg_error_16(int* code) {
  int v = 0, zero = 0;
  MIHS_CUDA_TRY(cudaMemcpyFromSymbol(&v, g_aab_reg_error, sizeof(int)));
  if (v != 0) MIHS_CUDA_TRY(cudaMemcpyToSymbol(g_aab_reg_error, &zero, sizeof(int)));
  *code = v;
  return MIHS_OK;
}

}  // namespace aabk
}  // namespace mihs
