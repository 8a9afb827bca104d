// FP32 row-transform kernels (forward divergence + x-transform, inverse
// x-transform + correction) and the register-resident vertical solve.
#include "pickers.h"
#include "tri.cuh"

namespace mp {
template <> KernelFn pick_k_fwd_rows<float>(int n) {
    if (KernelFn f = pick_f32_ext(kFwdRows, n)) return f;
    MP_PICK_F32(k_fwd_rows, (k_fwd_rows<float, 0>))
}
KernelFn pick_tri_cols(int levels) { return levels == 16 ? k_tri_cols<16> : k_tri_cols<kTriMaxL>; }
template <> KernelFn pick_k_inv_rows<float>(int n) {
    if (KernelFn f = pick_f32_ext(kInvRows, n)) return f;
    MP_PICK_F32(k_inv_rows, (k_inv_rows<float, 0>))
}
}  // namespace mp
