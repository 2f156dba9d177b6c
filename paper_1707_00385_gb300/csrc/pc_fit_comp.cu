// Instantiations of compensated sums whose J^T W J part is compensated block by
// block (run-time radius and stride, 32 x 8 tiles, per-frame and persistent
// batch kernels).
#include "pc_fit.cuh"

namespace pcurv {

const KernelOps* ops_compensated(bool packed) {
    return packed ? make_ops8<0, PREC_BLOCKS | PREC_PACKED>() : make_ops8<0, PREC_BLOCKS>();
}

}  // namespace pcurv
