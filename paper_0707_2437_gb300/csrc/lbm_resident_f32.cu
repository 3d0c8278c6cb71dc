// Instances of the resident kernel for one storage kind.
#include "lbm_resident.cuh"

namespace vss {

ResidentKernel resident_kernel_f32(int rnd, bool field, int shape) {
    (void)rnd;
    return field ? resident_of<ST_F32, 0, 1>(shape) : resident_of<ST_F32, 0, 0>(shape);
}

}  // namespace vss
