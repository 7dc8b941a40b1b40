// kernels_hbm_nph.cu -- the float pass kernels for plans without diagonal
// two-qubit phase ops (CRZ, RZZ): no phase cases in the switch (see apply_op).
#include "kernels.h"
#include "pass.cuh"

namespace vqc {

const void* pass_ptr_f32_nph(int mode, int K, bool full) {
    if (mode == 0 && K == 5)
        return full ? reinterpret_cast<const void*>(&pass_kernel<float, 5, 0, true, false>)
                    : reinterpret_cast<const void*>(&pass_kernel<float, 5, 0, false, false>);
    if (mode == 1 && K == 4)
        return full ? reinterpret_cast<const void*>(&pass_kernel<float, 4, 1, true, false>)
                    : reinterpret_cast<const void*>(&pass_kernel<float, 4, 1, false, false>);
    return nullptr;
}

}  // namespace vqc
