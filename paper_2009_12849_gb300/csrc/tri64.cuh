// Vertical solve (step a3) of FP64 plans: two threads per column, or per pair of
// columns ky and ny - ky, which share lambda and so their pivots.  One thread
// eliminates the lower levels upwards, the other the upper ones downwards; they
// exchange the fronts through shared memory, and each substitutes back outwards.
//
// Bound by FP64 arithmetic (1.7 multiply-adds per clock and SM), so what counts
// is the FP64 operations per column and level: 28 with a column per thread, a
// library division per pivot and the pivot e = lambda s - (A + A') - A^2 / e; 19 here,
// 15 for a paired column.  The pivots are those of the positive form of tri.cuh
// (E = A[k+1] + delta, delta = |lambda| s + A[k] rho, rho = delta / E: no
// cancellation for small lambda), their reciprocals one approximate reciprocal
// and one step of Householder's third-order iteration r (1 + e + e^2), e = 1 - E r;
// the scaling by 1/(nx ny), where that is a power of two, is the forward columns'
// (UNIT: it goes into their exponents).  Columns are taken linearly over (ky, kx), so that no lane idles at the
// end of a row (nx = 64 left half of them idle).
// GB300, one launch: 64^3 74 -> 37 us, 256^2 x 128 304 -> 147 us, 360x300x75 190 -> 146 us.
#pragma once
#include "kernels.cuh"

namespace mp {

constexpr int kTri64Batch = 4;           // levels whose loads are in flight (one batch ahead)

__device__ __forceinline__ double rcp64(double x) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double e = fma(-x, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

struct Tri64Smem {
    double ig[32], rho[32];              // the lower front: 1/E, delta/E and y of its last level
    double2 y[32][2], p[32][2];          // p of the upper side's lowest level
};

template <int NC, bool UNIT>
__device__ __forceinline__ void tri64_columns(const ProjParams& p, Tri64Smem& sm, const size_t (&base)[NC],
                                              double lam, bool mean, bool act, bool up, int lane) {
    constexpr int B = kTri64Batch;
    const int nz = p.nz, nlo = (nz + 1) / 2;
    const int n = !act ? 0 : up ? nz - nlo : nlo;      // levels of this thread, from its outer end
    const size_t LS = (size_t)p.ny * p.nxp;
    double2* S = (double2*)p.S;
    double2* G = (double2*)p.G;
    const double* __restrict__ ap = p.acoef + (up ? 1 : 0);      // coupling to the level before (outwards)
    const double* __restrict__ an = p.acoef + (up ? 0 : 1);      // and to the next one
    const double* __restrict__ s = p.svol;
    auto lev = [&](int i) { return up ? nz - 1 - i : i; };
    double ig = 0.0, rho = 0.0, delta = 0.0;           // 1/E, delta/E and delta of the level before
    double2 y[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) y[c] = make_double2(0.0, 0.0);
    double2 cur[B][NC], nxt[B][NC];
    auto load = [&](double2 (&d)[B][NC], int ib) {
#pragma unroll
        for (int i = 0; i < B; ++i)
#pragma unroll
            for (int c = 0; c < NC; ++c)
                d[i][c] = (ib + i < n) ? S[(size_t)lev(ib + i) * LS + base[c]] : make_double2(0.0, 0.0);
    };
    load(cur, 0);
    for (int ib = 0; ib < n; ib += B) {
        load(nxt, ib + B);
#pragma unroll
        for (int i = 0; i < B; ++i) {
            if (ib + i < n) {
                const int k = lev(ib + i);
                const double ak = ap[k];
                const double m = ak * ig;
                delta = fma(ak, rho, lam * s[k]);
                ig = rcp64(an[k] + delta);
                rho = delta * ig;
                const bool pin = mean && k == 0;
                if (pin) {                   // p[0] = 0
                    ig = 0.0;
                    rho = 1.0;
                }
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    y[c] = make_double2(fma(m, y[c].x, cur[i][c].x), fma(m, y[c].y, cur[i][c].y));
                    if (pin) y[c] = make_double2(0.0, 0.0);
                    S[(size_t)k * LS + base[c]] = y[c];
                }
                G[(size_t)k * LS + base[0]].x = -ig;
            }
        }
#pragma unroll
        for (int i = 0; i < B; ++i)
#pragma unroll
            for (int c = 0; c < NC; ++c) cur[i][c] = nxt[i][c];
    }
    // the middle: E = delta(up) + A rho(low), p = -(y(up) + A / E(low) y(low)) / E
    if (!up) {
        sm.ig[lane] = ig;
        sm.rho[lane] = rho;
#pragma unroll
        for (int c = 0; c < NC; ++c) sm.y[lane][c] = y[c];
    }
    __syncthreads();
    const bool two = nz > 1;
    double2 ph[NC];
    if (up && two) {
        const double ah = an[nlo];
        const double e = rcp64(fma(ah, sm.rho[lane], delta));
        const double m = ah * sm.ig[lane];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const double2 yl = sm.y[lane][c];
            ph[c] = make_double2(-e * fma(m, yl.x, y[c].x), -e * fma(m, yl.y, y[c].y));
            sm.p[lane][c] = ph[c];
        }
    }
    __syncthreads();
    if (!up) {
#pragma unroll
        for (int c = 0; c < NC; ++c) ph[c] = two ? sm.p[lane][c] : make_double2(0.0, 0.0);
    }
    // substitution outwards: p_k = (y_k - A p(next)) / e_k
    const double* __restrict__ idzn = UNIT ? p.idzn : p.idzn_scaled;
    auto scaled = [&](double2 v) { return UNIT ? v : make_double2(v.x * p.scale, v.y * p.scale); };
    int first = n - 1;
    if (up && n > 0) {                       // the middle's level is solved
#pragma unroll
        for (int c = 0; c < NC; ++c) S[(size_t)nlo * LS + base[c]] = scaled(ph[c]);
        first = n - 2;
    }
    double cg[B], ng[B];
    auto load_back = [&](double2 (&d)[B][NC], double (&g)[B], int ib) {
#pragma unroll
        for (int i = 0; i < B; ++i) {
            const size_t o = (size_t)(ib - i >= 0 ? lev(ib - i) : 0) * LS;
            g[i] = ib - i >= 0 ? G[o + base[0]].x : 0.0;
#pragma unroll
            for (int c = 0; c < NC; ++c) d[i][c] = ib - i >= 0 ? S[o + base[c]] : make_double2(0.0, 0.0);
        }
    };
    load_back(cur, cg, first);
    for (int ib = first; ib >= 0; ib -= B) {
        load_back(nxt, ng, ib - B);
#pragma unroll
        for (int i = 0; i < B; ++i) {
            if (ib - i >= 0) {
                const int k = lev(ib - i);
                const int kf = up ? k : k + 1;           // the face towards the middle
                const double a1 = an[k];
                const double iz = up ? -idzn[kf] : idzn[kf];
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const double2 pn = make_double2(fma(-a1, ph[c].x, cur[i][c].x) * cg[i],
                                                    fma(-a1, ph[c].y, cur[i][c].y) * cg[i]);
                    if (kf < nz)
                        G[(size_t)kf * LS + base[c]] = make_double2((ph[c].x - pn.x) * iz, (ph[c].y - pn.y) * iz);
                    S[(size_t)k * LS + base[c]] = scaled(pn);
                    ph[c] = pn;
                }
            }
        }
#pragma unroll
        for (int i = 0; i < B; ++i) {
            cg[i] = ng[i];
#pragma unroll
            for (int c = 0; c < NC; ++c) cur[i][c] = nxt[i][c];
        }
    }
}

// Blocks of two warps: the lower and the upper halves of 32 columns or pairs.
// PAIR: over (ky <= ny/2, kx), the columns ky and ny - ky of a whole spectrum;
// otherwise a column of the launch's rows each.  UNIT: D^ is scaled already.
template <bool PAIR, bool UNIT>
__global__ void __launch_bounds__(64) k_tri64(ProjParams p) {
    __shared__ Tri64Smem sm;
    const int lane = threadIdx.x & 31;
    const bool up = threadIdx.x >= 32;
    const int nky = PAIR ? p.ny / 2 + 1 : p.ny;
    const int t = min(blockIdx.x * 32 + lane, nky * p.nxh - 1);
    const bool act = blockIdx.x * 32 + lane < nky * p.nxh;
    const int ky = t / p.nxh, kx = t - ky * p.nxh;
    const int kyg = p.ky_base + ky;
    const double lam = -(p.lamx[kx] + p.lamy[kyg]);
    const bool mean = kx == 0 && kyg == 0;
    const size_t b0 = (size_t)ky * p.nxp + kx;
    if constexpr (PAIR) {
        // a row without a partner computes its column twice
        const bool alone = ky == 0 || 2 * ky >= p.ny;
        const size_t base[2] = {b0, alone ? b0 : (size_t)(p.ny - ky) * p.nxp + kx};
        tri64_columns<2, UNIT>(p, sm, base, lam, mean, act, up, lane);
    } else {
        const size_t base[1] = {b0};
        tri64_columns<1, UNIT>(p, sm, base, lam, mean, act, up, lane);
    }
}

}  // namespace mp
