// Resident kernel instantiations: iterate float, weights float, 11 to 16 classes.
#include "fw_resident.cuh"

namespace fw {
ResKern* make_res_f32_top(int K) {
    switch (K) {
        case 11: return new ResKernImpl<float, float, 12, false>();
        case 12: return new ResKernImpl<float, float, 12, true>();
        case 13: case 14: case 15: return new ResKernImpl<float, float, 16, false>();
        case 16: return new ResKernImpl<float, float, 16, true>();
        default: return nullptr;
    }
}
}  // namespace fw
