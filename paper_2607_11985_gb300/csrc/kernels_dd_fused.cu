// kernels_dd_fused.cu -- instantiations of the FUSED backward (it sweeps
// forward itself and writes E; vqc_forward_backward) with double-float
// arithmetic (complex128 storage), full-warp sample groups with factored stages or
// without, sub-warp ones.
#include "kernels.h"
#include "resident.cuh"

namespace vqc {

const void* sweep_ptr_dd_fused(int K, bool full, bool factored) {
    if (full && factored) {
        switch (K) {
        case 1: return reinterpret_cast<const void*>(&sweep_kernel<dd, 1, 1, true, true, false>);
        case 2: return reinterpret_cast<const void*>(&sweep_kernel<dd, 2, 1, true, true, false>);
        case 3: return reinterpret_cast<const void*>(&sweep_kernel<dd, 3, 1, true, true, false>);
        default: return nullptr;
        }
    }
    if (full) {
        switch (K) {
        case 1: return reinterpret_cast<const void*>(&sweep_kernel<dd, 1, 1, true, true>);
        case 2: return reinterpret_cast<const void*>(&sweep_kernel<dd, 2, 1, true, true>);
        case 3: return reinterpret_cast<const void*>(&sweep_kernel<dd, 3, 1, true, true>);
        default: return nullptr;
        }
    }
    switch (K) {
    case 1: return reinterpret_cast<const void*>(&sweep_kernel<dd, 1, 1, false, true>);
    case 2: return reinterpret_cast<const void*>(&sweep_kernel<dd, 2, 1, false, true>);
    case 3: return reinterpret_cast<const void*>(&sweep_kernel<dd, 3, 1, false, true>);
    default: return nullptr;
    }
}

}  // namespace vqc
