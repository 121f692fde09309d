// Resident kernel instantiations: iterate float, weights __nv_bfloat16, 2 to 6 classes.
#include "fw_resident.cuh"

namespace fw {
ResKern* make_res_bf16_lo(int K) {
    switch (K) {
        case 2: return new ResKernImpl<float, __nv_bfloat16, 2, true>();
        case 3: return new ResKernImpl<float, __nv_bfloat16, 3, true>();
        case 4: return new ResKernImpl<float, __nv_bfloat16, 4, true>();
        case 5: return new ResKernImpl<float, __nv_bfloat16, 5, true>();
        case 6: return new ResKernImpl<float, __nv_bfloat16, 6, true>();
        default: return nullptr;
    }
}
}  // namespace fw
