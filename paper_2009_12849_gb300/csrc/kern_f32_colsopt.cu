// FP32 opt-in column kernels: persistent cp.async and TMA-staged variants.
#include "persist.cuh"
#include "pickers.h"
#include "tma.cuh"

namespace mp {
template <> KernelFn pick_fwd_cols_persist<float>(int n) { MP_PICK_F32(k_cols_persist, nullptr, , false) }
template <> KernelFn pick_inv_cols_persist<float>(int n) { MP_PICK_F32(k_cols_persist, nullptr, , true) }
template <> ColsTmaFn pick_cols_tma<float>(int n, bool inv) {
    if (inv) { MP_PICK_F32(k_cols_tma, nullptr, , true) }
    MP_PICK_F32(k_cols_tma, nullptr, , false)
}
}  // namespace mp
