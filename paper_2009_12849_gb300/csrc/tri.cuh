// Vertical solve (step a3) of FP32 spectra with a column's levels held in
// registers, a warp per L levels (16, or 32 for tall grids) of 32 columns.
//
// Each warp of a group loads its levels of the group's 32 columns at once (a
// lane per column), so D' is read once and 32 columns x 256 levels (64 KB) are
// in flight per group.  The elimination runs from both ends: the lower warps
// eliminate upwards, the upper ones downwards, each warp taking the running
// value from its outer neighbour through shared memory; the two fronts meet
// between two warps, which solve for the two levels there, and the
// substitution runs outwards again.  A warp stores its levels while the next
// one works.  The order of a column's arithmetic depends on nz alone.
//
// Bound by: the 12 bytes per point that the levels take, for large grids; by
// the serial chain for small ones, which is why the chain has no division:
// with E_k = -e_k = A[k+1] + delta_k, delta_k = |lambda| s_k + A[k] delta_{k-1} / E_{k-1}
// (every term positive: no cancellation however small lambda is; the
// elimination of Grassmann, Taksar and Heyman, 1985, for M-matrices) and E_k =
// P_k / P_{k-1}, delta_k = Q_k / P_{k-1}, the pivots come from
//   Q_k = |lambda| s_k P_{k-1} + A[k] Q_{k-1}
//   P_k = (A[k+1] + |lambda| s_k) P_{k-1} + A[k] Q_{k-1},
// two fused multiply-adds per level in the chain.  Rows are scaled by powers
// of two (sigma_k, nearest A[k] + A[k+1]) and (P, Q) divided by P every
// kTriRenorm levels, so that they stay in range; the reciprocals P_{k-1} / P_k
// (one approximate reciprocal and one Newton correction of the quotient) hang
// off the chain.  The pivots do not depend on D' and are formed while it is in
// flight.  Measured (GB300, event to event): 64^3 26.5 -> 15 us, 256^2 x 128 83 ->
// 30 us, 405^2 x 93 75 -> 45 us, 1024^2 x 256 813 -> 650 us (4.95 TB/s of the 3.2 GB
// it must move), against thread-per-column sweeps with 8 levels in flight, the
// reciprocal in the chain and D' read twice.  One turn per warp from bottom to
// top with 32 levels a warp took 34 us and 915 us.
//
// The near-zero wavenumbers of a mixed or refined plan (pivots from the plan's
// table, FP32-pair arithmetic) go through the warps in turn, a few levels at a
// time, each warp loading its next levels while others work.  Pairs hold 48 bits where
// FP64 elimination, which refined plans ran before, holds 53; their right-hand sides
// and results are stored in FP32.  Refined solves of one, two and three passes on eleven
// grids (noise and smooth fields, six of each) came out as with FP64 elimination:
// geometric means 1.00, 0.99 and 1.00 of its errors in the velocities.
#pragma once
#include "kernels.cuh"

namespace mp {

constexpr int kTriWarps = 8;                 // most warps of a block
constexpr int kTriMaxL = 32;                 // most levels of a warp; nz <= kTriMaxL * kTriWarps
constexpr int kTriRenorm = 8;                // levels between restarts of the pivot recurrence
// the scaled pivots lie between 0.02 (columns that run in FP32 have |lambda| >=
// 0.02 v_max, see kFp64Fraction) and 2 + 1.5 |lambda| s_k / sigma_k; kTriRenorm of
// them multiply up in FP32's range below this bound on |lambda| s_k / sigma_k
constexpr double kTriMaxRatio = 1e4;
// levels per turn of the FP32-pair columns (their operands fit the registers
// that L levels of an FP32 column take)
MP_HD constexpr int tri_pair_chunk(int L) { return L / 4; }

// Groups of a launch: full 32-column chunks of every spectral row first (rows
// in the order 0, ny-1, 1, ny-2, ...: the near-zero wavenumbers, whose chain is
// the longest, start first), then the rows' remaining nxh % 32 columns,
// gathered from several rows so that their lanes are not idle (nx a power of
// two leaves one column: a chunk of its own would double the groups at nx = 64).
MP_HD constexpr int tri_tail_width(int nxh) {
    const int rem = nxh & 31;
    return rem == 0 ? 0 : rem <= 4 ? 4 : rem <= 8 ? 8 : rem <= 16 ? 16 : 32;
}
MP_HD constexpr long long tri_groups(int nxh, int ny) {
    const int tw = tri_tail_width(nxh);
    return (long long)ny * (nxh >> 5) + (tw ? (ny + 32 / tw - 1) / (32 / tw) : 0);
}
// Levels per warp: 16 keeps three blocks of 8 warps on an SM (32: two) and
// leaves less of the last warp empty.
MP_HD constexpr int tri_levels(int nz) { return nz <= 16 * kTriWarps ? 16 : kTriMaxL; }
MP_HD constexpr int tri_warps(int nz) { return (nz + tri_levels(nz) - 1) / tri_levels(nz); }

// Handovers between two warps of a group: the giver's writes are visible to
// the taker.  A warp takes pivots on one named barrier (id = its index in the
// block) and values on another (id + kTriWarps), since an outer neighbour may be
// a whole phase ahead; the warp that solves the middle takes the other front on
// the group's first warp's pivot barrier, which nothing else uses.
__device__ __forceinline__ void tri_give(int id) {
    __syncwarp();
    asm volatile("bar.arrive %0, 64;" ::"r"(id) : "memory");
}
__device__ __forceinline__ void tri_take(int id) {
    __syncwarp();
    asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory");
}

__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

struct TriSmem {
    float piv[kTriWarps][32];                // pivots' running Q / P taken by a warp
    float4 val[kTriWarps][32];               // values taken by a warp
    float4 mid[kTriWarps][32];               // the lower front at the middle
    float4 c0[kTriWarps][kTriMaxL];             // per-level constants of each warp, in its own order
    float2 c1[kTriWarps][kTriMaxL];
};

// Columns in FP32.  act: the lane's column takes part (the others compute on
// zeros).  w of nw: the warp's place in its group; wb: in its block.  r counts
// the warp's levels from its outer end (the bottom for the lower warps, the
// top for the upper ones): `next` is the neighbour towards the middle.
template <int kTriL>
__device__ __forceinline__ void tri_columns_f32(const ProjParams& p, TriSmem& sm, float2 (&d)[kTriL],
                                                size_t base, float lam, bool act, int w, int nw, int wb) {
    const int nz = p.nz, lane = threadIdx.x & 31;
    const size_t LS = (size_t)p.ny * p.nxp;
    const int nlo = nw > 1 ? nw / 2 : 1;     // lower warps
    const bool up = w >= nlo;                // upper side: levels counted downwards
    const int k0 = w * kTriL;
    const int n = min(kTriL, nz - k0);
    const int rb = up ? kTriL - n : 0, re = up ? kTriL : n;      // levels of the grid: rb <= r < re
    const bool outer = up ? w + 1 == nw : w == 0;
    const int wi = up ? -1 : 1;              // the neighbour towards the middle
    const bool meet_lo = nw > 1 && w + 1 == nlo, meet_up = up && w == nlo;
    const bool inner = nw == 1 || meet_lo || meet_up;
    {
        // levels past the top are identities: the sweeps below run without a
        // branch per level, so that the scheduler interleaves their chains
        float4 c0 = make_float4(0.f, 1.f, 0.f, 0.f);
        float2 c1 = make_float2(0.f, 0.f);
        if (lane < kTriL && lane >= rb && lane < re) {
            const int k = up ? k0 + kTriL - 1 - lane : k0 + lane;
            // s/sigma, A[k+1]/sigma, A[k]/sigma, -1/sigma; A[k+1], scale/dzn[k+1], A[k], -scale/dzn[k]
            c0 = __ldg(&p.tri32[2 * k]);
            const float4 t = __ldg(&p.tri32[2 * k + 1]);
            if (up) c0 = make_float4(c0.x, c0.z, c0.y, c0.w);
            c1 = up ? make_float2(t.z, t.w) : make_float2(t.x, t.y);
        }
        if (lane < kTriL) {
            sm.c0[wb][lane] = c0;            // s, A(next), A(previous) over sigma; -1/sigma
            sm.c1[wb][lane] = c1;            // A(next); scale/dzn of the face to it, signed
        }
        __syncwarp();
    }
    const float4* c0 = sm.c0[wb];
    const float2* c1 = sm.c1[wb];
    float g[kTriL];                          // 1/e_k = -1/E_k
#pragma unroll
    for (int r = 0; r < kTriL; ++r) g[r] = 0.f;
    float Q = 0.f;                           // delta / E of the previous level
    if (!outer) {
        tri_take(wb);
        Q = sm.piv[wb][lane];
    }
#pragma unroll
    for (int s = 0; s < kTriL; s += kTriRenorm) {
        if (s < re && s + kTriRenorm > rb) {
            float P = 1.f;
#pragma unroll
            for (int r = s; r < s + kTriRenorm; ++r) {
                const float4 c = c0[r];
                const float t = c.z * Q;
                const float P0 = fmaf(fmaf(lam, c.x, c.y), P, t);
                Q = fmaf(lam * c.x, P, t);
                const float rc = rcp_approx(P0);
                const float q = P * rc;
                g[r] = fmaf(fmaf(-P0, q, P), rc, q) * c.w;
                P = P0;
                if (r == s + kTriRenorm - 1) Q *= rc;
            }
        }
    }
    if (!inner) {
        sm.piv[wb + wi][lane] = Q;
        tri_give(wb + wi);
    }
    // y_r = D'_r - A/e y of the previous level
    float m = 0.f;
    float2 y = make_float2(0.f, 0.f);
    if (!outer) {
        tri_take(wb + kTriWarps);
        const float4 c = sm.val[wb][lane];
        m = c.x;
        y = make_float2(c.y, c.z);
    }
#pragma unroll
    for (int s = 0; s < kTriL; s += kTriRenorm) {
        if (s < re && s + kTriRenorm > rb) {
#pragma unroll
            for (int r = s; r < s + kTriRenorm; ++r) {
                y = make_float2(d[r].x - m * y.x, d[r].y - m * y.y);
                d[r] = y;
                m = c1[r].x * g[r];
            }
        }
    }
    float2 ph = make_float2(0.f, 0.f);
    if (!inner) {
        sm.val[wb + wi][lane] = make_float4(m, y.x, y.y, 0.f);
        tri_give(wb + wi + kTriWarps);
    } else if (meet_lo) {
        sm.mid[wb - w][lane] = make_float4(m, y.x, y.y, Q);
        tri_give(wb - w);
    } else if (meet_up) {
        // E = delta(up) + A delta(low) / E(low) at the lowest level of the upper side
        tri_take(wb - w);
        const float4 c = sm.mid[wb - w][lane];
        const float q = Q - c1[kTriL - 1].x * c.w * g[kTriL - 1];
        d[kTriL - 1] = make_float2(y.x - c.x * c.y, y.y - c.x * c.z);
        g[kTriL - 1] = __fdiv_rn(g[kTriL - 1], q);
        sm.val[wb - 1][lane] = make_float4(d[kTriL - 1].x * g[kTriL - 1], d[kTriL - 1].y * g[kTriL - 1], 0.f, 0.f);
        tri_give(wb - 1 + kTriWarps);
    }
    // substitution outwards: p_r = (y_r - A p(next)) / e_r
    if (nw > 1 && !meet_up) {
        tri_take(wb + kTriWarps);
        const float4 c = sm.val[wb][lane];
        ph = make_float2(c.x, c.y);
    }
    float2 nxt = ph;
#pragma unroll
    for (int s = kTriL - kTriRenorm; s >= 0; s -= kTriRenorm) {
        if (s < re && s + kTriRenorm > rb) {
#pragma unroll
            for (int r = s + kTriRenorm - 1; r >= s; --r) {
                const float a = c1[r].x;
                ph = make_float2((d[r].x - a * ph.x) * g[r], (d[r].y - a * ph.y) * g[r]);
                d[r] = ph;
            }
        }
    }
    if (!outer) {
        sm.val[wb - wi][lane] = make_float4(ph.x, ph.y, 0.f, 0.f);
        tri_give(wb - wi + kTriWarps);
    }
    if (!act) return;
    const float scale = (float)p.scale;
    const ptrdiff_t step = up ? (ptrdiff_t)LS : -(ptrdiff_t)LS;
    float2* sk = (float2*)p.S + (size_t)(up ? k0 : k0 + kTriL - 1) * LS + base;
    float2* gk = (float2*)p.G + (size_t)(up ? k0 : k0 + kTriL) * LS + base;
    // the face between the two sides is the lower one's; level nz - 1 of a
    // single warp has none above
    const int rf = (meet_up || nw == 1) ? re - 1 : re;
#pragma unroll
    for (int r = kTriL - 1; r >= 0; --r) {
        if (r >= rb && r < re) {
            const float iz = c1[r].y;
            if (r < rf) __stcs(gk, make_float2((nxt.x - d[r].x) * iz, (nxt.y - d[r].y) * iz));
            __stcs(sk, make_float2(d[r].x * scale, d[r].y * scale));
            nxt = d[r];
        }
        sk += step;
        gk += step;
    }
}

// a - b * c on FP32 pairs.
__device__ __forceinline__ F2P fp_msub(F2P a, F2P b, F2P c) {
    const float q = b.hi * c.hi;
    const float e = fmaf(b.hi, c.lo, fmaf(b.lo, c.hi, fmaf(b.hi, c.hi, -q)));
    const F2P s = fp_two_sum(a.hi, -q);
    return fp_fast_two_sum(s.hi, s.lo + (a.lo - e));
}

// Near-zero wavenumbers on FP32 pairs with the plan's pivots (the recurrences
// of tridiag_column_pair).  Chunk c of B levels belongs to warp c mod
// nw, which loads its next chunk's operands while other warps work; y waits in
// S and G (real, imaginary part) between the sweeps.
template <int B>
__device__ __forceinline__ void tri_columns_pair(const ProjParams& p, TriSmem& sm, size_t base, int slot, bool mean,
                                                 bool act, int w, int nw, int wb) {
    const int nz = p.nz, lane = threadIdx.x & 31, w0 = wb - w;
    const size_t LS = (size_t)p.ny * p.nxp, GS = (size_t)p.nslots;
    float2* S = (float2*)p.S;
    float2* G = (float2*)p.G;
    const float2* pm = p.pvm + slot;
    const float4* pg = p.pvgb + slot;
    const int nch = (nz + B - 1) / B;
    auto take = [&]() { if (nw > 1) tri_take(wb + kTriWarps); };
    auto give = [&](int c) { if (nw > 1) tri_give(w0 + c % nw + kTriWarps); };
    float2 dv[B], mv[B];
    auto load_fwd = [&](int c) {
#pragma unroll
        for (int i = 0; i < B; ++i) {
            const int k = c * B + i;
            const bool in = act && k < nz;
            dv[i] = in ? S[(size_t)k * LS + base] : make_float2(0.f, 0.f);
            mv[i] = in ? pm[(size_t)k * GS] : make_float2(0.f, 0.f);
        }
    };
    if (w < nch) load_fwd(w);
    for (int c = w; c < nch; c += nw) {
        F2P yr{0.f, 0.f}, yi{0.f, 0.f};
        if (c > 0) {
            take();
            const float4 t = sm.val[w0][lane];
            yr = F2P{t.x, t.y};
            yi = F2P{t.z, t.w};
        }
        float4 yy[B];
#pragma unroll
        for (int i = 0; i < B; ++i) {
            const F2P m{mv[i].x, mv[i].y};
            yr = fp_msub(F2P{dv[i].x, 0.f}, m, yr);
            yi = fp_msub(F2P{dv[i].y, 0.f}, m, yi);
            if (mean && c == 0 && i == 0) yr = yi = F2P{0.f, 0.f};
            yy[i] = make_float4(yr.hi, yr.lo, yi.hi, yi.lo);
        }
        if (c + 1 < nch) {
            sm.val[w0][lane] = make_float4(yr.hi, yr.lo, yi.hi, yi.lo);
            give(c + 1);
        }
        if (act) {
#pragma unroll
            for (int i = 0; i < B; ++i) {
                const int k = c * B + i;
                if (k < nz) {
                    S[(size_t)k * LS + base] = make_float2(yy[i].x, yy[i].y);
                    G[(size_t)k * LS + base] = make_float2(yy[i].z, yy[i].w);
                }
            }
        }
        if (c + nw < nch) load_fwd(c + nw);
    }
    // back substitution: p_k = y_k / e_k - (A[k+1] / e_k) p_{k+1}
    if (w >= nch) return;
    const float scale = (float)p.scale;
    float2 ys[B], yg[B];
    float4 gv[B];
    auto load_bwd = [&](int c) {
#pragma unroll
        for (int i = 0; i < B; ++i) {
            const int k = c * B + i;
            const bool in = act && k < nz;
            ys[i] = in ? S[(size_t)k * LS + base] : make_float2(0.f, 0.f);
            yg[i] = in ? G[(size_t)k * LS + base] : make_float2(0.f, 0.f);
            gv[i] = in ? pg[(size_t)k * GS] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    const int c_last = w + ((nch - 1 - w) / nw) * nw;
    load_bwd(c_last);
    for (int c = c_last; c >= 0; c -= nw) {
        // y / e does not wait for the level above
        F2P rr[B], ri[B];
#pragma unroll
        for (int i = 0; i < B; ++i) {
            const F2P g{gv[i].x, gv[i].y};
            rr[i] = fp_mul(F2P{ys[i].x, ys[i].y}, g);
            ri[i] = fp_mul(F2P{yg[i].x, yg[i].y}, g);
        }
        F2P pr{0.f, 0.f}, pi{0.f, 0.f};
        if (c + 1 < nch) {
            take();
            const float4 t = sm.val[w0][lane];
            pr = F2P{t.x, t.y};
            pi = F2P{t.z, t.w};
        }
        const F2P ar = pr, ai = pi;                  // the level above this chunk
#pragma unroll
        for (int i = B - 1; i >= 0; --i) {
            const F2P b{gv[i].z, gv[i].w};           // 0 at the top level and past it
            pr = fp_msub(rr[i], b, pr);
            pi = fp_msub(ri[i], b, pi);
            rr[i] = pr;
            ri[i] = pi;
        }
        if (c > 0) {
            sm.val[w0][lane] = make_float4(pr.hi, pr.lo, pi.hi, pi.lo);
            give(c - 1);
        }
        if (act) {
            F2P ur = ar, ui = ai;
#pragma unroll
            for (int i = B - 1; i >= 0; --i) {
                const int k = c * B + i;
                if (k < nz) {
                    if (k + 1 < nz) {
                        const float iz = p.idzn32[k + 1] * scale;
                        const F2P dr = fp_sub(ur, rr[i]), di = fp_sub(ui, ri[i]);
                        G[(size_t)(k + 1) * LS + base] = make_float2((dr.hi + dr.lo) * iz, (di.hi + di.lo) * iz);
                    }
                    S[(size_t)k * LS + base] = make_float2(rr[i].hi * scale, ri[i].hi * scale);
                    ur = rr[i];
                    ui = ri[i];
                }
            }
        }
        if (c - nw >= 0) load_bwd(c - nw);
    }
}

// Block blk of an instance's launch: p.tri_gpb groups of 32 columns with
// tri_warps(nz) warps each (a single group's FP32-pair columns use every warp
// of the block).
template <int kTriL>
__device__ __forceinline__ void tri_group(const ProjParams& p, TriSmem& sm, int blk) {
    const int wb = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nw = (p.nz + kTriL - 1) / kTriL;
    const bool solo = p.tri_gpb == 1;
    const int gi = solo ? 0 : wb / nw;
    const int w = wb - gi * nw;
    const int grp = blk * p.tri_gpb + gi;
    if (gi >= p.tri_gpb || grp >= tri_groups(p.nxh, p.ny)) return;
    const int nfull = p.nxh >> 5;
    const int nmain = p.ny * nfull;
    int ky, kx;
    if (grp < nmain) {
        const int r = grp / nfull;
        kx = ((grp - r * nfull) << 5) + lane;
        ky = (r & 1) ? p.ny - 1 - (r >> 1) : (r >> 1);
    } else {
        const int tw = tri_tail_width(p.nxh);
        ky = (grp - nmain) * (32 / tw) + lane / tw;
        kx = (nfull << 5) + lane % tw;
    }
    const bool in = ky < p.ny && kx < p.nxh;
    const int kyg = p.ky_base + ky;
    const size_t base = in ? (size_t)ky * p.nxp + kx : 0;
    // the levels are on their way before the columns' kind is known
    float2 d[kTriL];
    auto load = [&]() {                      // (lanes without a column read column 0)
        const size_t LS = (size_t)p.ny * p.nxp;
        const bool up = nw > 1 && w >= nw / 2;
        const int k0 = w * kTriL, n = min(kTriL, p.nz - k0);
        const int rb = up ? kTriL - n : 0, re = up ? kTriL : n;
        const ptrdiff_t step = up ? -(ptrdiff_t)LS : (ptrdiff_t)LS;
        const float2* src = (const float2*)p.S + (size_t)(up ? k0 + kTriL - 1 : k0) * LS + base;
#pragma unroll
        for (int r = 0; r < kTriL; ++r) {
            d[r] = make_float2(0.f, 0.f);
            if (r >= rb && r < re) d[r] = *src;
            src += step;
        }
    };
    load();
    const int ws = in ? p.wslot[kyg * p.nwr + (kx >> 5)] : -1;
    const float lam = in ? (float)-(p.lamx[kx] + p.lamy[kyg]) : 1.f;     // |lambda|
    const bool pair = in && ws >= 0, f32 = in && ws < 0;
    // every warp of the group sees the same lanes, so all take the same turns
    const bool any32 = __any_sync(0xffffffffu, f32);
    if (__any_sync(0xffffffffu, pair)) {
        const int np = solo ? (int)(blockDim.x >> 5) : nw;
        tri_columns_pair<tri_pair_chunk(kTriL)>(p, sm, base, pair ? ws + (kx & 31) : 0, pair && kx == 0 && kyg == 0, pair, w, np, wb);
        // both kinds in one group: the barriers are free again when all are here
        if (any32) {
            __syncwarp();
            asm volatile("bar.sync %0, %1;" ::"r"(wb - w), "r"(np * 32) : "memory");
            load();
        }
    }
    if (any32 && w < nw) tri_columns_f32<kTriL>(p, sm, d, base, lam, f32, w, nw, wb);
}

template <int L>
__global__ void __launch_bounds__(32 * kTriWarps, L == 16 ? 3 : 2) k_tri_cols(ProjParams p) {
    begin_after_previous();
    __shared__ TriSmem sm;
    tri_group<L>(p, sm, blockIdx.x);
}

}  // namespace mp
