// Kernel selection across translation units.  The host code picks kernels
// through these functions; each precision's kernels are instantiated (and
// compiled in parallel) in their own translation unit (kern_*.cu).
//
// Lengths with a compile-time FFT plan get their own instantiation: FP32 every
// 2^a 3^b 5^c length from 36 to 2048 (MP_F32_CT_CORE and MP_F32_CT_EXT*), FP64 every one from
// 36 to 1024 in fixed point (MP_FX_CT*) and 64, 128, 256 and 1024 in FP64 butterflies
// (MP_PICK_F64: the opt-in variants' plans).  Other lengths run the run-time
// plan (template argument 0).
#pragma once
#include "tma.cuh"

namespace mp {

using KernelFn = void (*)(ProjParams);
using ColsTmaFn = void (*)(ProjParams, ColMaps);

template <typename R> KernelFn pick_k_fwd_rows(int n);
template <typename R> KernelFn pick_k_inv_rows(int n);
template <typename R> KernelFn pick_k_fwd_cols(int n);
template <typename R> KernelFn pick_k_inv_cols(int n);
template <typename R> KernelFn pick_fwd_cols_persist(int n);   // nullptr if no compile-time plan
template <typename R> KernelFn pick_inv_cols_persist(int n);
template <typename R> KernelFn pick_fwd_fused(int n);
template <typename R> KernelFn pick_inv_fused(int n);
template <typename R> KernelFn pick_tridiag();
KernelFn pick_tri64(bool pair, bool unit); // tri64.cuh: FP64 spectra, 64 threads a block
KernelFn pick_tri_cols(int levels);      // tri.cuh: FP32 spectra, levels per warp 16 or 32
// FP32 column kernels with the spectral pitch, tile width and radix schedule
// (e: elements per thread, 32 or 16) fixed at compile time (nx = ny = 64, 96,
// 128, 192, 256, 512, 1024 with the default tiles; E = 16 for 256, 512, 1024
// with 256-thread tiles); nullptr otherwise
KernelFn pick_cols_square_f32(int ny, int nxp, int tw, int bs, bool inv, int e);
// grouped-launch kernels of batched FP32 projections (group.cuh): phase 0..4
// = forward rows, forward columns, vertical solve, inverse columns, inverse
// rows, for length n (the rows' nx or the columns' ny; any n for phase 2);
// nullptr when n has no compile-time plan
struct GroupArgs;
using GroupFn = void (*)(const GroupArgs);
// (square: nx = ny; with nxp and tw the group's spectral pitch and tile width,
// which select the column kernels that have them compiled in when they match)
GroupFn pick_group_f32(int phase, int n, bool square = false, int nxp = 0, int tw = 0);
GroupFn pick_group_tri_cols(int levels);
// FP32 persistent pipelines of the forward and inverse transforms (pipe.cuh);
// nullptr for grids without them
// (ef: the variants streaming u, v, w with evict-first L2 priority)
KernelFn pick_fwd_pipe(int nx, int ny, bool ef = false);
KernelFn pick_inv_pipe(int nx, int ny, bool ef = false);
// tensor-core split-precision forward column transforms (tcdft.cuh), format
// 1 (TF32 x 3) or 2 (BF16 x 6): nullptr unless ny = 1024; and their dynamic
// shared memory
KernelFn pick_fwd_cols_tc(int ny, int fmt);
unsigned fwd_cols_tc_smem(int fmt);
// refinement passes: FP32 transforms on FP64 fields (row kernels with F = double)
KernelFn pick_refined_fwd_rows(int n);
KernelFn pick_refined_inv_rows(int n);
KernelFn pick_refined_inv_cols(int n);   // the potential alone
template <typename R> ColsTmaFn pick_cols_tma(int n, bool inv);  // nullptr if none

}  // namespace mp

// Body of a picker: the compile-time lengths of the precision, else DEFAULT.
#define MP_PICK_F32(KERNEL, DEFAULT, ...)                              \
    switch (n) {                                                       \
        case 64: return KERNEL<float, 64 __VA_ARGS__>;                 \
        case 96: return KERNEL<float, 96 __VA_ARGS__>;                 \
        case 128: return KERNEL<float, 128 __VA_ARGS__>;               \
        case 192: return KERNEL<float, 192 __VA_ARGS__>;               \
        case 256: return KERNEL<float, 256 __VA_ARGS__>;               \
        case 512: return KERNEL<float, 512 __VA_ARGS__>;               \
        case 1024: return KERNEL<float, 1024 __VA_ARGS__>;             \
        default: return DEFAULT;                                       \
    }
// Extended FP32 compile-time lengths: every other 2^a 3^b 5^c length from 36
// to 2048.  They get the default kernels only, compiled in groups of up to 9
// lengths, rows and columns apart, so that the translation units build in
// parallel (kern_f32_ext.cu, compiled once per group and part).  (The run-time
// plans, which take one stage at a time through two shared buffers with every
// index computed, need 2.5 to 3 times as long: 768x640x72 2.41 -> 0.80 ms,
// 1536x1280x20 2.65 -> 1.09, 900x625x60 2.46 -> 1.00, 2048^2 x 8 2.32 -> 0.86)
#define MP_F32_CT_EXT1(F) F(135) F(144) F(150) F(160) F(162) F(180) F(200) F(216)
#define MP_F32_CT_EXT2(F) F(225) F(240) F(243) F(250) F(270) F(288) F(300) F(320)
#define MP_F32_CT_EXT3(F) F(324) F(360) F(375) F(384) F(400) F(405) F(432) F(450)
#define MP_F32_CT_EXT4(F) F(480) F(486) F(500)
#define MP_F32_CT_EXT5(F) F(540) F(576) F(600) F(625) F(640) F(648) F(675) F(720)
#define MP_F32_CT_EXT6(F) F(729) F(750) F(768) F(800) F(810) F(864) F(900) F(960)
#define MP_F32_CT_EXT7(F) F(972) F(1000) F(1080) F(1125) F(1152) F(1200) F(1215) F(1250)
#define MP_F32_CT_EXT8(F) F(1280) F(1296) F(1350) F(1440) F(1458) F(1500) F(1536) F(1600)
#define MP_F32_CT_EXT9(F) F(1620) F(1728) F(1800) F(1875) F(1920) F(1944) F(2000) F(2025)
#define MP_F32_CT_EXT10(F) F(2048) F(36) F(40) F(45) F(48) F(50) F(54) F(60)
#define MP_F32_CT_EXT11(F) F(72) F(75) F(80) F(81) F(90) F(100) F(108) F(120) F(125)
// every group
#define MP_F32_CT_EXT_GROUPS(G) G(1) G(2) G(3) G(4) G(5) G(6) G(7) G(8) G(9) G(10) G(11)
// FP32 lengths that also have the opt-in variants (persistent, TMA, fused)
#define MP_F32_CT_CORE(F) F(64) F(96) F(128) F(192) F(256) F(512) F(1024)

namespace mp {
enum KernelKind { kFwdRows = 0, kInvRows = 1, kFwdCols = 2, kInvCols = 3 };
// group g, part 0 (rows: kFwdRows, kInvRows) or 1 (columns); nullptr when n is
// not in the group or kind not in the part
#define MP_EXT_DECL(G) KernelFn pick_f32_ext_##G##_0(KernelKind kind, int n); KernelFn pick_f32_ext_##G##_1(KernelKind kind, int n);
MP_F32_CT_EXT_GROUPS(MP_EXT_DECL)
#undef MP_EXT_DECL
inline KernelFn pick_f32_ext(KernelKind kind, int n) {
#define MP_EXT_FNS(G) pick_f32_ext_##G##_0, pick_f32_ext_##G##_1,
    KernelFn (*const fns[])(KernelKind, int) = {MP_F32_CT_EXT_GROUPS(MP_EXT_FNS)};
#undef MP_EXT_FNS
    for (auto f : fns)
        if (KernelFn k = f(kind, n)) return k;
    return nullptr;
}
// FP32 lengths with a compile-time plan (core or extended)
inline bool ct_length_f32(int n) {
#define MP_CT_CASE(N) case N:
    switch (n) {
        MP_F32_CT_CORE(MP_CT_CASE)
#define MP_CT_GROUP(G) MP_F32_CT_EXT##G(MP_CT_CASE)
        MP_F32_CT_EXT_GROUPS(MP_CT_GROUP)
#undef MP_CT_GROUP
            return true;
        default:
            return false;
    }
#undef MP_CT_CASE
}
// Lengths whose FP64 transforms run in fixed point (fx.cuh), in groups that
// compile in parallel (kern_fx.cu).
#define MP_FX_CT0(F) MP_F32_CT_CORE(F)
#define MP_FX_CT1(F) MP_F32_CT_EXT1(F)
#define MP_FX_CT2(F) MP_F32_CT_EXT2(F)
#define MP_FX_CT3(F) MP_F32_CT_EXT3(F)
#define MP_FX_CT4(F) MP_F32_CT_EXT4(F) F(36) F(40) F(45) F(48) F(50)
#define MP_FX_CT5(F) MP_F32_CT_EXT5(F)
#define MP_FX_CT6(F) MP_F32_CT_EXT6(F)
#define MP_FX_CT7(F) F(972) F(1000) F(54) F(60) F(72) F(75) F(80)
#define MP_FX_CT8(F) F(81) F(90) F(100) F(108) F(120) F(125)
#define MP_FX_CT_GROUPS(G) G(0) G(1) G(2) G(3) G(4) G(5) G(6) G(7) G(8)
#define MP_FX_DECL(G) KernelFn pick_fx_##G(KernelKind kind, int n);
MP_FX_CT_GROUPS(MP_FX_DECL)
#undef MP_FX_DECL
inline KernelFn pick_fx(KernelKind kind, int n) {
#define MP_FX_TRY(G) \
    if (KernelFn k = pick_fx_##G(kind, n)) return k;
    MP_FX_CT_GROUPS(MP_FX_TRY)
#undef MP_FX_TRY
    return nullptr;
}
inline bool ct_length_fx(int n) {
#define MP_CT_CASE(N) case N:
#define MP_CT_GROUP(G) MP_FX_CT##G(MP_CT_CASE)
    switch (n) {
        MP_FX_CT_GROUPS(MP_CT_GROUP)
            return true;
        default:
            return false;
    }
#undef MP_CT_GROUP
#undef MP_CT_CASE
}
inline bool ct_core_f32(int n) {
#define MP_CT_CASE(N) case N:
    switch (n) {
        MP_F32_CT_CORE(MP_CT_CASE)
            return true;
        default:
            return false;
    }
#undef MP_CT_CASE
}
}  // namespace mp

#define MP_PICK_F64(KERNEL, DEFAULT, ...)                              \
    switch (n) {                                                       \
        case 64: return KERNEL<double, 64 __VA_ARGS__>;                \
        case 128: return KERNEL<double, 128 __VA_ARGS__>;              \
        case 256: return KERNEL<double, 256 __VA_ARGS__>;              \
        case 1024: return KERNEL<double, 1024 __VA_ARGS__>;            \
        default: return DEFAULT;                                       \
    }
