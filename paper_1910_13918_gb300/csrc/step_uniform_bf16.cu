// The fused uniform step with BF16 storage (step_uniform.cuh).
#include "step_uniform.cuh"

namespace sllbm {

cudaError_t launch_step_uniform_bf16(const StepArgs& a, const UniformTables& t, cudaStream_t s) {
  return launch_step_uniform_store<__nv_bfloat16>(a, t, s);
}

}  // namespace sllbm
