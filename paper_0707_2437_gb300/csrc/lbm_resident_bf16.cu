// Instances of the resident kernel for one storage kind.
#include "lbm_resident.cuh"

namespace vss {

ResidentKernel resident_kernel_bf16(int rnd, bool field, int shape) {
    return field ? resident_of<ST_BF16, 0, 1>(shape)
                 : (rnd ? resident_of<ST_BF16, 1, 0>(shape) : resident_of<ST_BF16, 0, 0>(shape));
}

}  // namespace vss
