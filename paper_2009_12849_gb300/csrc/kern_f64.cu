// FP64 kernels with FP64 butterflies: the run-time plan of the lengths that have no
// fixed-point kernels (kern_fx.cu), the vertical solve, and, for plans made with the
// persistent or fused variants switched on, the compile-time lengths.
#include "fused.cuh"
#include "pickers.h"
#include "tri64.cuh"

namespace mp {
template <> KernelFn pick_k_fwd_rows<double>(int n) { MP_PICK_F64(k_fwd_rows, (k_fwd_rows<double, 0>)) }
template <> KernelFn pick_k_inv_rows<double>(int n) { MP_PICK_F64(k_inv_rows, (k_inv_rows<double, 0>)) }
template <> KernelFn pick_k_fwd_cols<double>(int n) { MP_PICK_F64(k_fwd_cols, (k_fwd_cols<double, 0>)) }
template <> KernelFn pick_k_inv_cols<double>(int n) { MP_PICK_F64(k_inv_cols, (k_inv_cols<double, 0>)) }
template <> KernelFn pick_fwd_cols_persist<double>(int n) { MP_PICK_F64(k_cols_persist, nullptr, , false) }
template <> KernelFn pick_inv_cols_persist<double>(int n) { MP_PICK_F64(k_cols_persist, nullptr, , true) }
template <> KernelFn pick_fwd_fused<double>(int n) { MP_PICK_F64(k_fwd_fused, nullptr) }
template <> KernelFn pick_inv_fused<double>(int n) { MP_PICK_F64(k_inv_fused, nullptr) }
KernelFn pick_tri64(bool pair, bool unit) {
    if (unit) return pair ? k_tri64<true, true> : k_tri64<false, true>;
    return pair ? k_tri64<true, false> : k_tri64<false, false>;
}
template <> ColsTmaFn pick_cols_tma<double>(int, bool) { return nullptr; }
}  // namespace mp
