// Resident kernel instantiations: iterate double, weights double, 2 to 16 classes.
#include "fw_resident.cuh"

namespace fw {
ResKern* make_res_f64(int K) {
    switch (K) {
        case 2: case 3: case 4: return new ResKernImpl<double, double, 4, false>();
        case 5: case 6: case 7: case 8: return new ResKernImpl<double, double, 8, false>();
        case 9: case 10: return new ResKernImpl<double, double, 10, false>();
        case 11: case 12: return new ResKernImpl<double, double, 12, false>();
        case 13: case 14: case 15: case 16: return new ResKernImpl<double, double, 16, false>();
        default: return nullptr;
    }
}
}  // namespace fw
