// Instantiations of compensated sums (run-time radius and stride, 32 x 8 tiles,
// per-frame and persistent batch kernels).
#include "pc_fit.cuh"

namespace pcurv {

const KernelOps* ops_kahan(bool packed) {
    return packed ? make_ops8<0, PREC_KAHAN | PREC_PACKED>() : make_ops8<0, PREC_KAHAN>();
}

}  // namespace pcurv
