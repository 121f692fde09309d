// Resident kernel instantiations: iterate float, weights __nv_bfloat16, 11 to 16 classes.
#include "fw_resident.cuh"

namespace fw {
ResKern* make_res_bf16_top(int K) {
    switch (K) {
        case 11: return new ResKernImpl<float, __nv_bfloat16, 12, false>();
        case 12: return new ResKernImpl<float, __nv_bfloat16, 12, true>();
        case 13: case 14: case 15: return new ResKernImpl<float, __nv_bfloat16, 16, false>();
        case 16: return new ResKernImpl<float, __nv_bfloat16, 16, true>();
        default: return nullptr;
    }
}
}  // namespace fw
