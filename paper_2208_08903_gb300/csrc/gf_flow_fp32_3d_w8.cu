// gf_flow_fp32_3d_w8.cu -- the 3D, width 8 instantiations of the fused FP32 kernel.
#include "gf_flow_fp32_kernel.cuh"

namespace gf {
namespace f32k {

template <>
FlowKernel kernel_of<3, 8>(int tile, bool gw, int mode) { return pick_kernel<3, 8>(tile, gw, mode); }

}  // namespace f32k
}  // namespace gf
