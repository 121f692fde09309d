// Resident kernel instantiations: iterate float, weights __nv_bfloat16, 7 to 10 classes.
#include "fw_resident.cuh"

namespace fw {
ResKern* make_res_bf16_hi(int K) {
    switch (K) {
        case 7: return new ResKernImpl<float, __nv_bfloat16, 7, true>();
        case 8: return new ResKernImpl<float, __nv_bfloat16, 8, true>();
        case 9: return new ResKernImpl<float, __nv_bfloat16, 9, true>();
        case 10: return new ResKernImpl<float, __nv_bfloat16, 10, true>();
        default: return nullptr;
    }
}
}  // namespace fw
