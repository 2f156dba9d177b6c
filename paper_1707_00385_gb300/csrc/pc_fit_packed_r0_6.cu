// Instantiations for ranges stored as 16-bit offsets from a per-tile base, with
// radius and stride read at run time (r = 0) and for dense windows of radius 1
// to 6, unrolled (plain sums, 32 x 8 tiles).  The arithmetic after loading a
// range is the float32 kernels' own.
#include "pc_fit.cuh"

namespace pcurv {

const KernelOps* ops_packed_r0_6(int r) {
    switch (r) {
        case 0: return make_ops8<0, PREC_PACKED>();
        case 1: return make_ops8<1, PREC_PACKED>();
        case 2: return make_ops8<2, PREC_PACKED>();
        case 3: return make_ops8<3, PREC_PACKED>();
        case 4: return make_ops8<4, PREC_PACKED>();
        case 5: return make_ops8<5, PREC_PACKED>();
        case 6: return make_ops8<6, PREC_PACKED>();
        default: return nullptr;
    }
}

}  // namespace pcurv
