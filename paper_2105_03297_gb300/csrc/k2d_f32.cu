// 2D pass kernels, FP32 instances (inner solve of the mixed-precision path).
#include "nodal.cuh"
#include "pass_force.cuh"
namespace rve {
template cudaError_t launch_pass_a_2d<float>(const PassArgs<float>&, cudaStream_t);
template cudaError_t launch_pass_c_2d<float>(const PassArgs<float>&, cudaStream_t);
template cudaError_t launch_pass_e_2d<float>(const PassArgs<float>&, cudaStream_t);
template cudaError_t launch_cg_finish_x<float>(const PassArgs<float>&, cudaStream_t);
template cudaError_t launch_force_2d<float>(const PassArgs<float>&, cudaStream_t);
template cudaError_t launch_nodal_finish<float>(const PassArgs<float>&, const float*, const float*, const float*, cudaStream_t);
}  // namespace rve
