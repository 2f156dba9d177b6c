// Instantiations for ranges stored as 16-bit offsets from a per-tile base, for
// dense windows of radius 7 to 12, unrolled (plain sums, 32 x 8 tiles).  The
// arithmetic after loading a range is the float32 kernels' own.
#include "pc_fit.cuh"

namespace pcurv {

const KernelOps* ops_packed_r7_12(int r) {
    switch (r) {
        case 7: return make_ops8<7, PREC_PACKED>();
        case 8: return make_ops8<8, PREC_PACKED>();
        case 9: return make_ops8<9, PREC_PACKED>();
        case 10: return make_ops8<10, PREC_PACKED>();
        case 11: return make_ops8<11, PREC_PACKED>();
        case 12: return make_ops8<12, PREC_PACKED>();
        default: return nullptr;
    }
}

}  // namespace pcurv
