// Transform kernels of FP64 plans in 64-bit block fixed point (fx.cuh) for one
// group of compile-time lengths.  Compiled once per group:
//   -DMP_FX_GROUP=0..8
#include "fx.cuh"
#include "pickers.h"

#if !defined(MP_FX_GROUP)
#error "compile with -DMP_FX_GROUP=<0..8>"
#endif

#define MP_FX_LIST2(G) MP_FX_CT##G
#define MP_FX_LIST1(G) MP_FX_LIST2(G)
#define MP_FX_LIST MP_FX_LIST1(MP_FX_GROUP)
#define MP_FX_NAME2(G) pick_fx_##G
#define MP_FX_NAME(G) MP_FX_NAME2(G)

namespace mp {
KernelFn MP_FX_NAME(MP_FX_GROUP)(KernelKind kind, int n) {
#define MP_CASE(N)                                 \
    case N:                                        \
        switch (kind) {                            \
            case kFwdRows: return k_fwd_rows_fx<N>; \
            case kInvRows: return k_inv_rows_fx<N>; \
            case kFwdCols: return k_fwd_cols_fx<N>; \
            default: return k_inv_cols_fx<N>;      \
        }
    switch (n) {
        MP_FX_LIST(MP_CASE)
        default: return nullptr;
    }
#undef MP_CASE
}
}  // namespace mp
