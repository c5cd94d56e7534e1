// gf_train_bwd_2d.cu -- the 2D instantiations of the reverse pass kernels.
#include <algorithm>

#include "gf_train_bwd.cuh"

namespace gf {
namespace bwd {

BwdOps ops_2d(int C) {
    switch (C) {
        case 8: return make_ops<2, 8>();
        case 16: return make_ops<2, 16>();
        case 24: return make_ops<2, 24>();
        default: return make_ops<2, 32>();
    }
}

}  // namespace bwd
}  // namespace gf
