// kernels_f64_bwd.cu -- instantiations of the sweep kernel for double, mode 1, sample
// groups of at least one warp (full-warp reductions), stages in rounds
// or with the op switch.
#include "kernels.h"
#include "resident.cuh"

namespace vqc {

const void* sweep_ptr_f64_bwd(int K, bool rounds) {
    if (!rounds) {
        switch (K) {
        case 1: return reinterpret_cast<const void*>(&sweep_kernel<double, 1, 1, true, false, true, false>);
        case 2: return reinterpret_cast<const void*>(&sweep_kernel<double, 2, 1, true, false, true, false>);
        case 3: return reinterpret_cast<const void*>(&sweep_kernel<double, 3, 1, true, false, true, false>);
        default: return nullptr;
        }
    }
    switch (K) {
    case 1: return reinterpret_cast<const void*>(&sweep_kernel<double, 1, 1, true, false>);
    case 2: return reinterpret_cast<const void*>(&sweep_kernel<double, 2, 1, true, false>);
    case 3: return reinterpret_cast<const void*>(&sweep_kernel<double, 3, 1, true, false>);
    default: return nullptr;
    }
}

}  // namespace vqc
