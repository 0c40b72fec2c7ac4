// Kernel instantiations for the ProbHumanoid36 problem class: the FP32 path
// runs the one-lane-per-configuration tree kernel (the cyclic form: the warp kernel), the plain FP64 path and the collision
// check the thread-per-configuration kernels.
#include "mcp_tree.cuh"

namespace mcp {

template <>
cudaError_t launch_project<ProbHumanoid36>(const HostModel &hm, const ProjCall &c, int *launches) {
  if (c.precision == 1) {
    if (c.total <= 0) return cudaSuccess;
    if (c.segments) return cudaErrorNotSupported;
    cudaError_t e =
        launch_plain64_any<ProbHumanoid36>(hm, c, BatchSrc<double>{static_cast<const double *>(c.q_in), c.ld_in});
    *launches += 1;
    if (e == cudaSuccess && c.fused_check) e = check_outputs<ProbHumanoid36>(hm, c, launches);
    return e;
  }
  // stacked form: one lane per configuration; the cyclic form's masked
  // sub-steps run on the warp-per-configuration kernel
  cudaError_t e = c.cyclic ? launch_project_warp<ProbHumanoid36>(hm, c, launches)
                           : launch_project_tree<ProbHumanoid36>(hm, c, launches);
  if (e == cudaSuccess && c.fused_check) e = check_outputs<ProbHumanoid36>(hm, c, launches);
  return e;
}

template <>
cudaError_t launch_check<ProbHumanoid36>(const HostModel &hm, const CheckCall &c, int *launches) {
  return launch_check_impl<ProbHumanoid36>(hm, c, launches);
}

template <>
cudaError_t launch_vjp<ProbHumanoid36>(const HostModel &, const VjpCall &, int *) {
  return cudaErrorNotSupported;
}

MCP_NO_EXTEND(ProbHumanoid36)

}  // namespace mcp
