// gf_flow_fp32_3d_w16.cu -- the 3D, width 16 instantiations of the fused FP32 kernel.
#include "gf_flow_fp32_kernel.cuh"

namespace gf {
namespace f32k {

template <>
FlowKernel kernel_of<3, 16>(int tile, bool gw, int mode) { return pick_kernel<3, 16>(tile, gw, mode); }

}  // namespace f32k
}  // namespace gf
