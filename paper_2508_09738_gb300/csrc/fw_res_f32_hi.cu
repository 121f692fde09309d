// Resident kernel instantiations: iterate float, weights float, 7 to 10 classes.
#include "fw_resident.cuh"

namespace fw {
ResKern* make_res_f32_hi(int K) {
    switch (K) {
        case 7: return new ResKernImpl<float, float, 7, true>();
        case 8: return new ResKernImpl<float, float, 8, true>();
        case 9: return new ResKernImpl<float, float, 9, true>();
        case 10: return new ResKernImpl<float, float, 10, true>();
        default: return nullptr;
    }
}
}  // namespace fw
