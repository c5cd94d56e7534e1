// gf_train_bwd_3d.cu -- the 3D instantiations of the reverse pass kernels.
#include <algorithm>

#include "gf_train_bwd.cuh"

namespace gf {
namespace bwd {

BwdOps ops_3d(int C) {
    switch (C) {
        case 8: return make_ops<3, 8>();
        case 16: return make_ops<3, 16>();
        case 24: return make_ops<3, 24>();
        default: return make_ops<3, 32>();
    }
}

}  // namespace bwd
}  // namespace gf
