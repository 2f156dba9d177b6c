// Instantiations of compensated sums whose J^T W J part is compensated block by
// block (run-time radius and stride, 32 x 8 tiles, per-frame and persistent
// batch kernels), for float32 ranges and 16-bit storage.
#include "pc_fit.cuh"

namespace pcurv {

const KernelOps* ops_compensated(int format) {
#define PC_COMP_OPS(P) {{launch_fit_rw<0, P, 8>, nullptr}, {launch_batch_rw<0, P, 8>, nullptr}, {occupancy_rw<0, P, 8>, nullptr}}
    static const KernelOps k[3] = {PC_COMP_OPS(PREC_BLOCKS | PREC_KAHAN), PC_COMP_OPS(PREC_BLOCKS | PREC_KAHAN | 2),
                                   PC_COMP_OPS(PREC_BLOCKS | PREC_KAHAN | 4)};
#undef PC_COMP_OPS
    return format < 0 || format > 2 ? nullptr : &k[format];
}

}  // namespace pcurv
