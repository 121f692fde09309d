// Resident kernel instantiations: iterate float, weights float, 2 to 6 classes.
#include "fw_resident.cuh"

namespace fw {
ResKern* make_res_f32_lo(int K) {
    switch (K) {
        case 2: return new ResKernImpl<float, float, 2, true>();
        case 3: return new ResKernImpl<float, float, 3, true>();
        case 4: return new ResKernImpl<float, float, 4, true>();
        case 5: return new ResKernImpl<float, float, 5, true>();
        case 6: return new ResKernImpl<float, float, 6, true>();
        default: return nullptr;
    }
}
}  // namespace fw
