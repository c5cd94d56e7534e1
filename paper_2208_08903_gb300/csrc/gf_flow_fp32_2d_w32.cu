// gf_flow_fp32_2d_w32.cu -- the 2D, width 32 instantiations of the fused FP32 kernel.
#include "gf_flow_fp32_kernel.cuh"

namespace gf {
namespace f32k {

template <>
FlowKernel kernel_of<2, 32>(int tile, bool gw, int mode) { return pick_kernel<2, 32>(tile, gw, mode); }

}  // namespace f32k
}  // namespace gf
