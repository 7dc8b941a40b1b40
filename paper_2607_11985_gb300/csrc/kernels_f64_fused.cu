// kernels_f64_fused.cu -- instantiations of the sweep kernel for double, mode 1
// with FUSED: the backward that sweeps forward itself and writes E
// (vqc_forward_backward), for full-warp sample groups with
// stages in rounds or the op switch, and sub-warp ones.
#include "kernels.h"
#include "resident.cuh"

namespace vqc {

const void* sweep_ptr_f64_fused(int K, bool full, bool rounds) {
    if (full && !rounds) {
        switch (K) {
        case 1: return reinterpret_cast<const void*>(&sweep_kernel<double, 1, 1, true, true, true, false>);
        case 2: return reinterpret_cast<const void*>(&sweep_kernel<double, 2, 1, true, true, true, false>);
        case 3: return reinterpret_cast<const void*>(&sweep_kernel<double, 3, 1, true, true, true, false>);
        default: return nullptr;
        }
    }
    if (full) {
        switch (K) {
        case 1: return reinterpret_cast<const void*>(&sweep_kernel<double, 1, 1, true, true>);
        case 2: return reinterpret_cast<const void*>(&sweep_kernel<double, 2, 1, true, true>);
        case 3: return reinterpret_cast<const void*>(&sweep_kernel<double, 3, 1, true, true>);
        case 4: return reinterpret_cast<const void*>(&sweep_kernel<double, 4, 1, true, true>);
        default: return nullptr;
        }
    }
    if (!full) {
        switch (K) {
        case 1: return reinterpret_cast<const void*>(&sweep_kernel<double, 1, 1, false, true>);
        case 2: return reinterpret_cast<const void*>(&sweep_kernel<double, 2, 1, false, true>);
        case 3: return reinterpret_cast<const void*>(&sweep_kernel<double, 3, 1, false, true>);
        case 4: return reinterpret_cast<const void*>(&sweep_kernel<double, 4, 1, false, true>);
        default: return nullptr;
        }
    }
    return nullptr;
}

}  // namespace vqc
