// Krylov pressure solver (paper, Section 4: BiCGStab on the Poisson problem
// L phi = D(u*) of the FFT solver; the paper preconditions it with ILU, runs
// it in single precision to a 1e-4 stopping criterion as well as in double,
// and names a bespoke, structure-aware preconditioner as further work).
//
// L = D o G as a 7-point stencil: periodic second differences in x and y and
// the rows of the vertical operator,
//   (L x)[k] = (x_e - 2x + x_w)/dx^2 + (x_n - 2x + x_s)/dy^2
//            + sub[k] x[k-1] + diag0[k] x[k] + sup[k] x[k+1],
//   sub[k] = A[k]/V[k], sup[k] = A[k+1]/V[k], diag0[k] = -(A[k] + A[k+1])/V[k],
// with A[k] = rho_f[k]/dzn[k] (A[0] = A[nz] = 0) and V[k] = rho_c[k] dz[k].
//
// Preconditioner (precond = 1): the vertical lines of L, i.e. the vertical
// rows plus the diagonal of the horizontal part (-2/dx^2 - 2/dy^2).  Every
// column (i, j) has the same matrix, so its Thomas factors (cp[k] and the
// inverse pivots) are the plan's (krylov_tables; a one-thread kernel per solve
// took 150 us for 128 levels) and each application is one forward and one
// backward sweep per column, a thread per column, coalesced across i.  It takes the place of ILU, whose triangular
// sweeps run through the whole grid one cell after another.
//
// BiCGStab (van der Vorst 1992) with the preconditioner applied to the search
// directions, in the order of the preconditioned algorithm of Barrett et al.,
// Templates (1994): x0 = 0, shadow residual r~ = r0 = b, stop when
// ||r|| <= tol ||b|| on the recurrence residual, also after the half step on s.
// Vectors are in the field precision T (FP64 plans: double; mixed plans:
// float, whose arithmetic GB300 runs 64 times faster than FP64).  The iterate
// x = (x + alpha p^) + omega s^ is updated once per iteration: in FP64 for
// FP64 plans, and for FP32 as an unevaluated sum x_hi + x_lo of two floats
// (Knuth's TwoSum adds each FP32 increment to x_hi and carries the rounding
// error into x_lo), so the final gradient G phi is formed from a potential
// accurate to about 2^-48 without FP64 arithmetic in the loop.
// Inner products: sums in T over a few tens of a thread's elements at most (a tile's 32
// levels, a batch of a line sweep, a thread's share of a streaming kernel), block and
// global sums in FP64; the
// scalars (rho, alpha, omega, beta) live in device memory as FP64.  Each block
// of a reducing kernel writes its partial sums; the last block to finish (a
// ticket counter) adds all partials in a fixed order and forms the next
// scalar, so results are deterministic run to run and no separate reduction
// launch is needed.  The host enqueues kKryCheckEvery iterations at a time
// and then reads the scalar block to test convergence; the kernels of the
// iterations after the one that stopped return at once, so the iteration
// count and the result are those of a test after every iteration.  A denominator that is zero or not finite (rounding past the
// attainable accuracy) ends the method as a breakdown.
//
// After the solve phi is pinned as in the FFT solver (level-0 horizontal mean
// zero) and the outputs are u - G phi (w zero on the bottom and top faces).
#include <algorithm>
#include <cstddef>
#include <cstdint>

#include "krylov.h"

namespace mp {
namespace {

constexpr int kKryThreads = 256;
constexpr int kKryBlocksPerSm = 8;       // streaming kernels: 2048 threads per SM
constexpr int kKryIlp = 4;               // elements in flight per thread (streaming kernels)
constexpr int kKrySums = 2;              // partial sums per block
constexpr int kKryCheckEvery = 8;        // iterations enqueued between host convergence tests
constexpr int kTileX = 32, kTileY = 8;   // stencil kernels: a 32 x 8 tile of columns
constexpr int kTileZ = 32;               //   marching over 32 levels (one reduction per block)
constexpr int kApplyBatch = 8;           // FP32 stencil: levels whose operands load together
// line sweeps: levels loaded before use (32 FP32 or 16 FP64 values: about
// 128 bytes per thread in flight, enough to cover DRAM latency with the few
// threads one per column gives)
template <typename T> constexpr int kLineBatch = 128 / sizeof(T);

constexpr int kLineThreads = 64;         // fused line sweeps: columns per block
constexpr size_t kLineSmem = 200 * 1024; //   and their shared memory at most
constexpr size_t kSmSmem = 228 * 1024;   // shared memory of an SM
constexpr size_t kLineOwn = 2304;        // what a block of them takes beside its columns

// Scalars of the iteration, in device memory.
struct KrySc {
    double bnorm;                        // ||b||
    double rho, alpha, omega, beta;
    double relres;                       // ||r|| / ||b|| of the last completed step
    double srel;                         // ||s|| / ||b|| of the current half step
    double mean;                         // level-0 horizontal mean of phi (pin)
    int done;                            // 1: stopped
    int half;                            // 1: stop after x += alpha p^ (half-step end)
    int status;                          // 0 converged, 2 breakdown
    int iters;                           // completed iterations
};

enum Stage { kStRhs = 0, kStAlpha = 1, kStS = 2, kStOmega = 3, kStR = 4, kStMean = 5 };

template <typename T>
struct Tabs {
    const T *vsub, *vdiag, *vsup;        // vertical rows of L
    const T *lcp, *livd;                 // line preconditioner: cp[k], 1/pivot[k]
    const T *flo, *fhi;                  // divergence: rho_f[k]/V[k], rho_f[k+1]/V[k] (0 at the ends)
};

template <typename T>
struct Ws {
    T* xh;                               // the iterate: x_hi (FP64 plans: x itself)
    T* xl;                               // FP32: x_lo of x = x_hi + x_lo
    T *r, *rt, *p, *v, *ph, *sh, *t;
    double* part;                        // [nparts][kKrySums]
    KrySc* sc;
    unsigned* ticket;                    // blocks of the running reduction that have finished
};

size_t al256(size_t n) { return (n + 255) & ~size_t(255); }

constexpr int kVecX = 32, kVecY = 8, kVecZ = 8;      // four-column stencil: threads, rows and levels of a tile
dim3 vec_tiles(int nx, int ny, int nz) {
    return dim3((nx + 4 * kVecX - 1) / (4 * kVecX), (ny + kVecY - 1) / kVecY, (nz + kVecZ - 1) / kVecZ);
}

struct Shape {
    int nblk;                            // streaming kernels
    dim3 tiles;                          // stencil kernels
    int ntile;
    int nparts;                          // partial-sum slots: max of the two
};

Shape shape(int nx, int ny, int nz, int nsm) {
    Shape sh;
    sh.nblk = std::max(1, nsm) * kKryBlocksPerSm;
    sh.tiles = dim3((nx + kTileX - 1) / kTileX, (ny + kTileY - 1) / kTileY, (nz + kTileZ - 1) / kTileZ);
    sh.ntile = (int)(sh.tiles.x * sh.tiles.y * sh.tiles.z);
    sh.nparts = std::max({sh.nblk, sh.ntile, (int)(((size_t)nx * ny + kLineThreads - 1) / kLineThreads)});
    const dim3 vt = vec_tiles(nx, ny, nz);
    sh.nparts = std::max(sh.nparts, (int)(vt.x * vt.y * vt.z));
    return sh;
}

// Workspace layout: the iterate (one T field, two for FP32), seven T fields,
// the partial sums, the scalars and ticket.  With base == nullptr
// only the size is computed.
template <typename T>
Ws<T> carve(void* base, int nx, int ny, int nz, int nparts, size_t* bytes) {
    const size_t N = (size_t)nx * ny * nz;
    size_t off = 0;
    Ws<T> w{};
    auto take = [&](size_t n) -> unsigned char* {
        unsigned char* q = base ? (unsigned char*)base + off : nullptr;
        off = al256(off + n);
        return q;
    };
    w.xh = (T*)take(N * sizeof(T));
    w.xl = (sizeof(T) == 4) ? (T*)take(N * sizeof(T)) : nullptr;
    T** vecs[7] = {&w.r, &w.rt, &w.p, &w.v, &w.ph, &w.sh, &w.t};
    for (T** q : vecs) *q = (T*)take(N * sizeof(T));
    w.part = (double*)take((size_t)nparts * kKrySums * sizeof(double));
    w.sc = (KrySc*)take(sizeof(KrySc));
    w.ticket = (unsigned*)take(sizeof(unsigned));
    if (bytes) *bytes = off;
    return w;
}

template <typename T>
struct Grid {
    int nx, ny, nz;
    size_t plane, n;
    T idx, idy, idx2, idy2;
    double idx64, idy64;
};

// The scalars a finished reduction forms (a and b: the two global sums).
__device__ void finish_stage(KrySc* sc, int stage, double a, double b, double tol, int iter, int max_iter,
                             double plane) {
    if (stage == kStMean) { sc->mean = a / plane; return; }
    if (stage == kStRhs) {
        sc->bnorm = sqrt(a);
        sc->rho = a;                        // (r~, r0) = ||b||^2
        sc->alpha = sc->omega = 1.0;
        sc->beta = 0.0;
        sc->relres = sc->srel = (a > 0.0) ? 1.0 : 0.0;
        sc->done = (a > 0.0) ? 0 : 1;
        sc->half = 0;
        sc->status = 0;
        sc->iters = 0;
        return;
    }
    if (sc->done) return;
    if (stage == kStAlpha) {                // a = (r~, v)
        if (a == 0.0 || !isfinite(a)) { sc->done = 1; sc->status = 2; return; }
        sc->alpha = sc->rho / a;
    } else if (stage == kStS) {             // a = ||s||^2
        const double sn = sqrt(a);
        sc->srel = sn / sc->bnorm;
        if (sn <= tol * sc->bnorm) { sc->half = 1; sc->status = 0; }
    } else if (stage == kStOmega) {         // a = (t, s), b = (t, t)
        if (sc->half) return;
        if (b == 0.0 || !isfinite(b)) { sc->half = 1; sc->status = 2; return; }
        sc->omega = a / b;
    } else if (stage == kStR) {             // a = ||r||^2, b = (r~, r)
        sc->iters = iter;
        if (sc->half) { sc->relres = sc->srel; sc->done = 1; return; }
        sc->relres = sqrt(a) / sc->bnorm;
        if (sc->relres <= tol) { sc->done = 1; sc->status = 0; return; }
        // omega = 0 ends the method now; rho = (r~, r) = 0 would end the next
        // iteration before its first step
        const bool bad_omega = sc->omega == 0.0 || !isfinite(sc->omega);
        const bool bad_rho = (b == 0.0 || !isfinite(b)) && iter < max_iter;
        if (bad_omega || bad_rho) { sc->done = 1; sc->status = 2; return; }
        sc->beta = (b / sc->rho) * (sc->alpha / sc->omega);
        sc->rho = b;
    }
}

// What a reducing kernel does with its two block sums.
struct Reduce {
    double* part;                       // [nparts][kKrySums]
    unsigned* ticket;
    KrySc* sc;
    int nparts;                         // blocks of the launch
    int stage, iter, max_iter;
    double tol, plane;
};

// Block sum of up to two values into part[slot]; the last block of the launch
// to get here adds all partials in slot order and forms the stage's scalars.
template <int NT = kKryThreads>
__device__ __forceinline__ void block_reduce(double a, double b, const Reduce& rd, int slot) {
    __shared__ double sa[NT / 32], sb[NT / 32];
    __shared__ double fa[NT], fb[NT];
    __shared__ bool last;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
    }
    const int t = threadIdx.y * blockDim.x + threadIdx.x;
    const int wid = t >> 5, lane = t & 31;
    if (lane == 0) { sa[wid] = a; sb[wid] = b; }
    __syncthreads();
    if (t == 0) {
        double ta = 0.0, tb = 0.0;
        for (int i = 0; i < NT / 32; ++i) { ta += sa[i]; tb += sb[i]; }
        rd.part[slot * kKrySums + 0] = ta;
        rd.part[slot * kKrySums + 1] = tb;
        __threadfence();
        last = atomicAdd(rd.ticket, 1u) == (unsigned)(rd.nparts - 1);
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    // four independent sums per thread keep four loads in flight; the order
    // of the additions is fixed by the slot index
    double ga[4] = {0.0, 0.0, 0.0, 0.0}, gb[4] = {0.0, 0.0, 0.0, 0.0};
    for (int i0 = t; i0 < rd.nparts; i0 += 4 * NT) {
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int i = i0 + m * NT;
            if (i < rd.nparts) {
                ga[m] += __ldcg(&rd.part[i * kKrySums]);
                gb[m] += __ldcg(&rd.part[i * kKrySums + 1]);
            }
        }
    }
    fa[t] = (ga[0] + ga[1]) + (ga[2] + ga[3]);
    fb[t] = (gb[0] + gb[1]) + (gb[2] + gb[3]);
    __syncthreads();
    for (int s = NT / 2; s > 0; s >>= 1) {
        if (t < s) { fa[t] += fa[t + s]; fb[t] += fb[t + s]; }
        __syncthreads();
    }
    if (t == 0) {
        finish_stage(rd.sc, rd.stage, fa[0], fb[0], rd.tol, rd.iter, rd.max_iter, rd.plane);
        *rd.ticket = 0;
    }
}

__device__ __forceinline__ int tile_slot() { return blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z); }

// Column (i, j) of a stencil tile and the offsets of its periodic neighbours
// within a level.  Returns false for threads past the grid's edge.
struct Col {
    size_t c, ce, cw, cn, cs;
    int k0, k1;
};
template <typename T>
__device__ __forceinline__ bool tile_column(const Grid<T>& g, Col& cl) {
    const int i = blockIdx.x * kTileX + threadIdx.x;
    const int j = blockIdx.y * kTileY + threadIdx.y;
    cl.k0 = blockIdx.z * kTileZ;
    cl.k1 = min(g.nz, cl.k0 + kTileZ);
    if (i >= g.nx || j >= g.ny) return false;
    const size_t row = (size_t)j * g.nx;
    cl.c = row + i;
    cl.ce = row + (i == g.nx - 1 ? 0 : i + 1);
    cl.cw = row + (i == 0 ? g.nx - 1 : i - 1);
    cl.cn = (size_t)(j == g.ny - 1 ? 0 : j + 1) * g.nx + i;
    cl.cs = (size_t)(j == 0 ? g.ny - 1 : j - 1) * g.nx + i;
    return true;
}

// b = D(u, v, w) into r and r~; partials: ||b||^2.  (Stencil tiles.)
template <typename T>
__global__ void __launch_bounds__(kKryThreads) k_kry_rhs(Grid<T> g, Tabs<T> tb, const T* u, const T* v, const T* w,
                                                         T* r, T* rt, Reduce rd) {
    T acc = 0;
    Col cl;
    if (tile_column(g, cl)) {
        T wb = (cl.k0 > 0) ? w[(size_t)cl.k0 * g.plane + cl.c] : (T)0;
        for (int k = cl.k0; k < cl.k1; ++k) {
            const size_t o = (size_t)k * g.plane;
            const T wa = (k < g.nz - 1) ? w[o + g.plane + cl.c] : (T)0;
            const T d = (u[o + cl.c] - u[o + cl.cw]) * g.idx + (v[o + cl.c] - v[o + cl.cs]) * g.idy +
                        (tb.fhi[k] * wa - tb.flo[k] * wb);
            r[o + cl.c] = d;
            rt[o + cl.c] = d;
            acc += d * d;
            wb = wa;
        }
    }
    block_reduce((double)acc, 0.0, rd, tile_slot());
}

// y = L x; partials: (a, y) and, if yy, (y, y).  (Stencil tiles.)  FP32:
// the operands of kApplyBatch levels are loaded before the first is used;
// FP64 marches up the levels keeping the vertical neighbours in registers
// (the batched form needs 118 registers and measured slower).
template <typename T>
__global__ void __launch_bounds__(kKryThreads) k_kry_apply(Grid<T> g, Tabs<T> tb, const T* x, T* y, const T* a,
                                                           bool yy, Reduce rd) {
    if (rd.sc->done || rd.sc->half) return;
    T s1 = 0, s2 = 0;
    Col cl;
    if constexpr (sizeof(T) == 8) {
        if (tile_column(g, cl)) {
            T xd = (cl.k0 > 0) ? x[(size_t)(cl.k0 - 1) * g.plane + cl.c] : (T)0;
            T xc = x[(size_t)cl.k0 * g.plane + cl.c];
            for (int k = cl.k0; k < cl.k1; ++k) {
                const size_t o = (size_t)k * g.plane;
                const T xu = (k < g.nz - 1) ? x[o + g.plane + cl.c] : (T)0;
                const T o1 = (x[o + cl.ce] - (T)2 * xc + x[o + cl.cw]) * g.idx2 +
                             (x[o + cl.cn] - (T)2 * xc + x[o + cl.cs]) * g.idy2 + tb.vdiag[k] * xc +
                             tb.vsub[k] * xd + tb.vsup[k] * xu;
                y[o + cl.c] = o1;
                s1 += a[o + cl.c] * o1;
                if (yy) s2 += o1 * o1;
                xd = xc;
                xc = xu;
            }
        }
    } else if (tile_column(g, cl)) {
        constexpr int Zb = kApplyBatch;
        for (int kb = cl.k0; kb < cl.k1; kb += Zb) {
            T xc[Zb + 2], xe[Zb], xw[Zb], xn[Zb], xs[Zb], av[Zb];
            xc[0] = (kb > 0) ? x[(size_t)(kb - 1) * g.plane + cl.c] : (T)0;
#pragma unroll
            for (int i = 0; i <= Zb; ++i) {
                const int k = kb + i;
                xc[i + 1] = (k < g.nz) ? x[(size_t)k * g.plane + cl.c] : (T)0;
            }
#pragma unroll
            for (int i = 0; i < Zb; ++i) {
                const int k = kb + i;
                const size_t o = (size_t)(k < cl.k1 ? k : kb) * g.plane;
                xe[i] = x[o + cl.ce];
                xw[i] = x[o + cl.cw];
                xn[i] = x[o + cl.cn];
                xs[i] = x[o + cl.cs];
                av[i] = a[o + cl.c];
            }
#pragma unroll
            for (int i = 0; i < Zb; ++i) {
                const int k = kb + i;
                if (k < cl.k1) {
                    const T c = xc[i + 1];
                    const T o1 = (xe[i] - (T)2 * c + xw[i]) * g.idx2 + (xn[i] - (T)2 * c + xs[i]) * g.idy2 +
                                 tb.vdiag[k] * c + tb.vsub[k] * xc[i] + tb.vsup[k] * xc[i + 2];   // vsub[0] = vsup[nz-1] = 0
                    y[(size_t)k * g.plane + cl.c] = o1;
                    s1 += av[i] * o1;
                    if (yy) s2 += o1 * o1;
                }
            }
        }
    }
    block_reduce((double)s1, (double)s2, rd, tile_slot());
}

// The same for FP32 grids with nx a multiple of 4: a thread takes four adjacent
// columns (kVecX threads x kVecY rows a block) up kVecZ levels, loading the level
// above and its own level's neighbours as float4.  (One column a thread: six loads a
// point, 2.25 waves of 80-register blocks, 39 us at 256^2 x 128 for 101 MB.)
__global__ void __launch_bounds__(kKryThreads, 4) k_kry_apply4(Grid<float> g, Tabs<float> tb, const float* x, float* y,
                                                             const float* a, bool yy, Reduce rd) {
    if (rd.sc->done || rd.sc->half) return;
    const int i = 4 * (blockIdx.x * kVecX + threadIdx.x), j = blockIdx.y * kVecY + threadIdx.y;
    const int k0 = blockIdx.z * kVecZ, k1 = min(g.nz, k0 + kVecZ);
    float s1 = 0.f, s2 = 0.f;
    if (i < g.nx && j < g.ny) {
        const size_t row = (size_t)j * g.nx;
        const size_t c = row + i;
        const size_t cw = row + (i == 0 ? g.nx - 1 : i - 1), ce = row + (i + 4 == g.nx ? 0 : i + 4);
        const size_t cn = (size_t)(j == g.ny - 1 ? 0 : j + 1) * g.nx + i, cs = (size_t)(j == 0 ? g.ny - 1 : j - 1) * g.nx + i;
        auto ld = [&](const float* p, size_t q) { return *(const float4*)&p[q]; };
        const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
        float4 xd = k0 > 0 ? ld(x, (size_t)(k0 - 1) * g.plane + c) : z4;
        float4 xc = ld(x, (size_t)k0 * g.plane + c);
#pragma unroll 4
        for (int k = k0; k < k1; ++k) {
            const size_t o = (size_t)k * g.plane;
            const float4 xu = k < g.nz - 1 ? ld(x, o + g.plane + c) : z4;
            const float4 xn = ld(x, o + cn), xs = ld(x, o + cs), av = ld(a, o + c);
            const float xw = x[o + cw], xe = x[o + ce];
            const float vd = tb.vdiag[k], vb = tb.vsub[k], vp = tb.vsup[k];      // vsub[0] = vsup[nz-1] = 0
            auto pt = [&](float w, float cc, float e, float n, float s, float d, float u) {
                return (e - 2.f * cc + w) * g.idx2 + (n - 2.f * cc + s) * g.idy2 + vd * cc + vb * d + vp * u;
            };
            float4 o1;
            o1.x = pt(xw, xc.x, xc.y, xn.x, xs.x, xd.x, xu.x);
            o1.y = pt(xc.x, xc.y, xc.z, xn.y, xs.y, xd.y, xu.y);
            o1.z = pt(xc.y, xc.z, xc.w, xn.z, xs.z, xd.z, xu.z);
            o1.w = pt(xc.z, xc.w, xe, xn.w, xs.w, xd.w, xu.w);
            *(float4*)&y[o + c] = o1;
            s1 += (av.x * o1.x + av.y * o1.y) + (av.z * o1.z + av.w * o1.w);
            if (yy) s2 += (o1.x * o1.x + o1.y * o1.y) + (o1.z * o1.z + o1.w * o1.w);
            xd = xc;
            xc = xu;
        }
    }
    block_reduce((double)s1, (double)s2, rd, tile_slot());
}

// out = M^-1 in: Thomas down every column of the line matrix, one thread per
// column, kLineBatch levels loaded before use; the forward sweep leaves its
// values in out.
template <typename T>
__global__ void __launch_bounds__(kKryThreads, 2) k_kry_line(Grid<T> g, Tabs<T> tb, const T* __restrict__ in,
                                                          T* __restrict__ out, const KrySc* sc) {
    if (sc->done || sc->half) return;
    constexpr int B = kLineBatch<T>;
    const T* __restrict__ vsub = tb.vsub;
    const T* __restrict__ livd = tb.livd;
    const T* __restrict__ lcp = tb.lcp;
    for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < g.plane; c += (size_t)gridDim.x * blockDim.x) {
        T dp = 0;
        for (int kb = 0; kb < g.nz; kb += B) {
            T b[B];
#pragma unroll
            for (int i = 0; i < B; ++i) b[i] = (kb + i < g.nz) ? in[(size_t)(kb + i) * g.plane + c] : (T)0;
#pragma unroll
            for (int i = 0; i < B; ++i) {
                const int k = kb + i;
                if (k < g.nz) {
                    dp = (b[i] - __ldg(&vsub[k]) * dp) * __ldg(&livd[k]);      // vsub[0] = 0
                    out[(size_t)k * g.plane + c] = dp;
                }
            }
        }
        T xk = dp;
        for (int kb = g.nz - 2; kb >= 0; kb -= B) {
            T b[B];
#pragma unroll
            for (int i = 0; i < B; ++i) b[i] = (kb - i >= 0) ? out[(size_t)(kb - i) * g.plane + c] : (T)0;
#pragma unroll
            for (int i = 0; i < B; ++i) {
                const int k = kb - i;
                if (k >= 0) {
                    xk = b[i] - __ldg(&lcp[k]) * xk;
                    out[(size_t)k * g.plane + c] = xk;
                }
            }
        }
    }
}

// A streaming update of a column and the line solve of its result in one pass, in FP32:
// UPD 0: p = r + beta (p - omega v) (p = r at first), p^ = M^-1 p;
// UPD 1: s = r - alpha v (into r), s^ = M^-1 s, partials ||s||^2.
// A thread per column; the forward sweep's values wait in shared memory
// ([level][thread]; the last batch in registers, which lets seven blocks of 128
// levels share an SM: 1024 blocks are then one wave), so the updated vector is not read back and the sweeps'
// intermediate never leaves the SM.  Bound by the vectors it streams (5 and 4
// of them); as an update and a line kernel of its own, which wrote and re-read
// the intermediate: 24 + 27 us and 31 + 27 us of an iteration at 256^2 x 128 in
// FP32; the two fused kernels bring a solve of 8 iterations from 2.48 to 1.96 ms
// together with the four-wide kernels below.  The arithmetic of an element is unchanged.
constexpr int kFusedBatch = 16;
template <int UPD>
__global__ void __launch_bounds__(kLineThreads, 7) k_kry_line_fused(Grid<float> g, Tabs<float> tb, float* pr,
                                                                 const float* r, const float* v, float* out,
                                                                 bool first, Reduce rd) {
    using T = float;
    extern __shared__ __align__(16) unsigned char kry_smem[];
    const KrySc* sc = rd.sc;
    if (sc->done) return;
    constexpr int B = kFusedBatch;
    T* dpc = (T*)kry_smem + threadIdx.x;
    const T beta = (T)sc->beta, omega = (T)sc->omega, alpha = (T)sc->alpha;
    const size_t c = (size_t)blockIdx.x * kLineThreads + threadIdx.x;
    double sum = 0.0;
    if (c < g.plane) {
        T dp = 0, top[B];                    // the last batch's values stay in registers
        const int kt = (g.nz - 1) / B * B;   // its first level
        for (int kb = 0; kb <= kt; kb += B) {
            T a[B], b[B], d[B], acc = 0;
#pragma unroll
            for (int i = 0; i < B; ++i) {
                const size_t q = (size_t)(kb + i) * g.plane + c;
                const bool in = kb + i < g.nz;
                a[i] = in ? (UPD == 0 ? r[q] : pr[q]) : (T)0;
                b[i] = in && !(UPD == 0 && first) ? v[q] : (T)0;
                d[i] = UPD == 0 && in && !first ? pr[q] : (T)0;
            }
#pragma unroll
            for (int i = 0; i < B; ++i) {
                const int k = kb + i;
                if (k < g.nz) {
                    T x;
                    if (UPD == 0) {
                        x = first ? a[i] : a[i] + beta * (d[i] - omega * b[i]);
                    } else {
                        x = a[i] - alpha * b[i];
                        acc += x * x;
                    }
                    pr[(size_t)k * g.plane + c] = x;
                    dp = (x - __ldg(&tb.vsub[k]) * dp) * __ldg(&tb.livd[k]);      // vsub[0] = 0
                    if (kb < kt) dpc[k * kLineThreads] = dp;
                }
                top[i] = dp;
            }
            if (UPD == 1) sum += (double)acc;
        }
        T xk = 0;
#pragma unroll
        for (int i = B - 1; i >= 0; --i) {
            const int k = kt + i;
            if (k < g.nz) {
                xk = top[i] - __ldg(&tb.lcp[k]) * xk;        // lcp[nz-1] = 0
                out[(size_t)k * g.plane + c] = xk;
            }
        }
#pragma unroll 8
        for (int k = kt - 1; k >= 0; --k) {
            xk = dpc[k * kLineThreads] - __ldg(&tb.lcp[k]) * xk;
            out[(size_t)k * g.plane + c] = xk;
        }
    }
    if (UPD == 1) block_reduce<kLineThreads>(sum, 0.0, rd, blockIdx.x);
}

// Streaming kernels: thread t takes elements t + m * stride for m < kKryIlp,
// then the next kKryIlp * stride.
#define KRY_STREAM_LOOP(body)                                                              \
    {                                                                                      \
        const size_t stride = (size_t)gridDim.x * blockDim.x;                              \
        for (size_t q0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q0 < g.n;          \
             q0 += stride * kKryIlp) {                                                     \
            _Pragma("unroll") for (int m = 0; m < kKryIlp; ++m) {                          \
                const size_t q = q0 + m * stride;                                          \
                if (q < g.n) { body }                                                      \
            }                                                                              \
        }                                                                                  \
    }

// p = r (first iteration) or p = r + beta (p - omega v).
template <typename T>
__global__ void __launch_bounds__(kKryThreads) k_kry_p(Grid<T> g, T* p, const T* r, const T* v, bool first,
                                                       const KrySc* sc) {
    if (sc->done) return;
    const T beta = (T)sc->beta, omega = (T)sc->omega;
    KRY_STREAM_LOOP(p[q] = first ? r[q] : r[q] + beta * (p[q] - omega * v[q]);)
}

// s = r - alpha v (into r); partials: ||s||^2.
template <typename T>
__global__ void __launch_bounds__(kKryThreads) k_kry_s(Grid<T> g, T* r, const T* v, Reduce rd) {
    if (rd.sc->done) return;
    const T alpha = (T)rd.sc->alpha;
    T acc = 0;
    KRY_STREAM_LOOP(const T s = r[q] - alpha * v[q]; r[q] = s; acc += s * s;)
    block_reduce((double)acc, 0.0, rd, blockIdx.x);
}

// x += y: FP64 in place, FP32 as x_hi + x_lo with Knuth's TwoSum.
__device__ __forceinline__ void acc_x(double* xh, double*, size_t q, double y) { xh[q] = xh[q] + y; }
__device__ __forceinline__ void acc_x(float* xh, float* xl, size_t q, float y) {
    const float a = xh[q];
    const float s = a + y;
    const float bb = s - a;
    const float err = (a - (s - bb)) + (y - bb);
    xh[q] = s;
    xl[q] = xl[q] + err;
}

// x += alpha p^ + omega s^, r = s - omega t (r holds s); partials: ||r||^2,
// (r~, r).  After a half-step end only x += alpha p^.  (FP64 plans add the
// two terms one after the other, as (x + alpha p^) + omega s^.)
template <typename T>
__global__ void __launch_bounds__(kKryThreads) k_kry_update(Grid<T> g, T* xh, T* xl, const T* ph, const T* sh, T* r,
                                                            const T* t, const T* rt, Reduce rd) {
    const KrySc* sc = rd.sc;
    if (sc->done) return;
    const T alpha = (T)sc->alpha;
    if (sc->half) {
        KRY_STREAM_LOOP(acc_x(xh, xl, q, alpha * ph[q]);)
        block_reduce(0.0, 0.0, rd, blockIdx.x);
        return;
    }
    const T om = (T)sc->omega;
    T rr = 0, rtr = 0;
    if constexpr (sizeof(T) == 8) {
        KRY_STREAM_LOOP(xh[q] = (xh[q] + alpha * ph[q]) + om * sh[q]; const T rn = r[q] - om * t[q]; r[q] = rn;
                        rr += rn * rn; rtr += rt[q] * rn;)
    } else {
        KRY_STREAM_LOOP(acc_x(xh, xl, q, alpha * ph[q] + om * sh[q]); const T rn = r[q] - om * t[q]; r[q] = rn;
                        rr += rn * rn; rtr += rt[q] * rn;)
    }
    block_reduce((double)rr, (double)rtr, rd, blockIdx.x);
}

// The same in FP32 with the vectors taken four elements at a time (the count of
// points a multiple of 4): all seven operands of an element group are in flight, where
// four scalar elements of each did not fit 32 registers (82 us at 256^2 x 128 for 335 MB).
__global__ void __launch_bounds__(kKryThreads, 4) k_kry_update4(Grid<float> g, float* xh, float* xl, const float* ph,
                                                              const float* sh, float* r, const float* t,
                                                              const float* rt, Reduce rd) {
    const KrySc* sc = rd.sc;
    if (sc->done) return;
    const float alpha = (float)sc->alpha;
    const size_t stride = (size_t)gridDim.x * blockDim.x, n4 = g.n / 4;
    if (sc->half) {
        for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < n4; q += stride)
            for (int e = 0; e < 4; ++e) acc_x(xh, xl, 4 * q + e, alpha * ph[4 * q + e]);
        block_reduce(0.0, 0.0, rd, blockIdx.x);
        return;
    }
    const float om = (float)sc->omega;
    float rr = 0.f, rtr = 0.f;
    for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < n4; q += stride) {
        float4 h = ((float4*)xh)[q], l = ((float4*)xl)[q], p = ((const float4*)ph)[q], s = ((const float4*)sh)[q];
        float4 rv = ((float4*)r)[q], tv = ((const float4*)t)[q], w = ((const float4*)rt)[q];
        auto one = [&](float& a, float& b, float pe, float se, float& re, float te, float we) {
            const float y = alpha * pe + om * se;
            const float sum = a + y, bb = sum - a;
            b += (a - (sum - bb)) + (y - bb);
            a = sum;
            re = re - om * te;
            rr += re * re;
            rtr += we * re;
        };
        one(h.x, l.x, p.x, s.x, rv.x, tv.x, w.x);
        one(h.y, l.y, p.y, s.y, rv.y, tv.y, w.y);
        one(h.z, l.z, p.z, s.z, rv.z, tv.z, w.z);
        one(h.w, l.w, p.w, s.w, rv.w, tv.w, w.w);
        ((float4*)xh)[q] = h;
        ((float4*)xl)[q] = l;
        ((float4*)r)[q] = rv;
    }
    block_reduce((double)rr, (double)rtr, rd, blockIdx.x);
}

__device__ __forceinline__ double x_at(const double* xh, const double*, size_t q) { return xh[q]; }
__device__ __forceinline__ double x_at(const float* xh, const float* xl, size_t q) {
    return (double)xh[q] + (double)xl[q];
}

// Level-0 sum of x (the pin).
template <typename T>
__global__ void __launch_bounds__(kKryThreads) k_kry_level0(size_t plane, const T* xh, const T* xl, Reduce rd) {
    double acc = 0.0;
    for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < plane; q += (size_t)gridDim.x * blockDim.x)
        acc += x_at(xh, xl, q);
    block_reduce(acc, 0.0, rd, blockIdx.x);
}

// u_out = u - G phi with phi the iterate shifted by the pin; w zero on the
// bottom and top faces.  (Stencil tiles.)  FP64 plans: in FP64.  FP32: the
// differences of x = x_hi + x_lo are taken part by part, (x_hi' - x_hi) +
// (x_lo' - x_lo); each part's difference of two floats is rounded once,
// relative to the difference itself, so the gradient keeps FP32 accuracy
// relative to G phi (not to phi) without FP64 arithmetic.
template <typename T>
__global__ void __launch_bounds__(kKryThreads) k_kry_correct(Grid<T> g, const T* xh, const T* xl, const T* u,
                                                             const T* v, const T* w, const double* idzn, T* uo, T* vo,
                                                             T* wo, T* phi, const KrySc* sc) {
    Col cl;
    if (!tile_column(g, cl)) return;
    const double m = sc->mean;
    if constexpr (sizeof(T) == 8) {
        double xd = (cl.k0 > 0) ? xh[(size_t)(cl.k0 - 1) * g.plane + cl.c] - m : 0.0;
        for (int k = cl.k0; k < cl.k1; ++k) {
            const size_t o = (size_t)k * g.plane;
            const size_t q = o + cl.c;
            const double c = xh[q] - m;
            uo[q] = u[q] - ((xh[o + cl.ce] - m) - c) * g.idx64;
            vo[q] = v[q] - ((xh[o + cl.cn] - m) - c) * g.idy64;
            wo[q] = (k > 0) ? w[q] - (c - xd) * idzn[k] : 0.0;
            if (phi) phi[q] = c;
            xd = c;
        }
    } else {
        const size_t qd = (size_t)(cl.k0 > 0 ? cl.k0 - 1 : 0) * g.plane + cl.c;
        float hd = xh[qd], ld = xl[qd];
        for (int k = cl.k0; k < cl.k1; ++k) {
            const size_t o = (size_t)k * g.plane;
            const size_t q = o + cl.c;
            const float hc = xh[q], lc = xl[q];
            const float gx = (xh[o + cl.ce] - hc) + (xl[o + cl.ce] - lc);
            const float gy = (xh[o + cl.cn] - hc) + (xl[o + cl.cn] - lc);
            uo[q] = u[q] - gx * g.idx;
            vo[q] = v[q] - gy * g.idy;
            wo[q] = (k > 0) ? w[q] - ((hc - hd) + (lc - ld)) * (float)idzn[k] : 0.f;
            if (phi) phi[q] = (float)(((double)hc + (double)lc) - m);
            hd = hc;
            ld = lc;
        }
    }
    if (cl.k1 == g.nz) wo[g.n + cl.c] = (T)0;
}

template <typename T>
cudaError_t run(const KrylovProblem& kp, cudaStream_t st, KrylovResult* res) {
    const Shape sh = shape(kp.nx, kp.ny, kp.nz, kp.nsm);
    Ws<T> ws = carve<T>(kp.workspace, kp.nx, kp.ny, kp.nz, sh.nparts, nullptr);
    Grid<T> g;
    g.nx = kp.nx; g.ny = kp.ny; g.nz = kp.nz;
    g.plane = (size_t)kp.nx * kp.ny;
    g.n = g.plane * kp.nz;
    g.idx64 = 1.0 / kp.dx; g.idy64 = 1.0 / kp.dy;
    g.idx = (T)g.idx64; g.idy = (T)g.idy64;
    g.idx2 = (T)(g.idx64 * g.idx64); g.idy2 = (T)(g.idy64 * g.idy64);
    const int nblk = sh.nblk;
    const dim3 tb(kTileX, kTileY);
    const int cblk = (int)std::min<size_t>((size_t)nblk, (g.plane + kKryThreads - 1) / kKryThreads);
    const bool pc = kp.precond == 1;
    T* const ph = pc ? ws.ph : ws.p;          // M = I: p^ is p, s^ is s
    T* const shv = pc ? ws.sh : ws.r;
    const T* u = (const T*)kp.u; const T* v = (const T*)kp.v; const T* w = (const T*)kp.w;
    const int mi = kp.max_iter;
    cudaError_t e;
#define KRY_CHECK()                                      \
    if ((e = cudaGetLastError()) != cudaSuccess) return e
    if ((e = cudaMemsetAsync(ws.xh, 0, g.n * sizeof(T), st)) != cudaSuccess) return e;
    if (ws.xl && (e = cudaMemsetAsync(ws.xl, 0, g.n * sizeof(T), st)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(ws.ticket, 0, sizeof(unsigned), st)) != cudaSuccess) return e;
    auto rd = [&](int nparts, int stage, int it) {
        Reduce r;
        r.part = ws.part; r.ticket = ws.ticket; r.sc = ws.sc; r.nparts = nparts;
        r.stage = stage; r.iter = it; r.max_iter = mi; r.tol = kp.tol; r.plane = (double)g.plane;
        return r;
    };
    Tabs<T> tab;
    {
        const T* t = (const T*)kp.tables;
        const T** tabs[7] = {&tab.vsub, &tab.vdiag, &tab.vsup, &tab.lcp, &tab.livd, &tab.flo, &tab.fhi};
        for (const T** q : tabs) {
            *q = t;
            t += kp.nz;
        }
    }
    // the fused line sweeps hold a column of each thread in shared memory.  FP64
    // vectors keep the separate kernels: a column is twice as large, so that three
    // blocks of two warps are left on an SM for a sweep that the FP64 pipe bounds
    // (256^2 x 128: 0.82 ms an iteration against 0.73).  The same holds for tall FP32
    // columns, so they are taken where four blocks fit an SM (224 levels) or all
    // blocks are resident at once.  Eight iterations, fused / separate, us: 256^2 x 128
    // 1918 / 2092, x 224 3295 / 3469, x 256 (three blocks an SM) 4124 / 4005, x 320 (two) 5551 /
    // 4834, x 512 11453 / 7417; 512^2 x 224 11463 / 12235; 128^2 x 384 (256 blocks, two an SM) 1970 /
    // 2246, x 512 (one) 3451 / 2814; 64^2 x 800 (64 blocks) 2308 / 2645.
    const size_t lsm = (size_t)((kp.nz - 1) / kFusedBatch * kFusedBatch) * kLineThreads * sizeof(float);
    const int lblk = (int)((g.plane + kLineThreads - 1) / kLineThreads);
    const size_t per_sm = kSmSmem / (lsm + kLineOwn);
    const bool fuse = sizeof(T) == 4 && pc && lsm <= kLineSmem &&
                      (per_sm >= 4 || (size_t)lblk <= per_sm * (size_t)std::max(1, kp.nsm));
    if (fuse && lsm > 40 * 1024) {
        for (auto f : {(const void*)k_kry_line_fused<0>, (const void*)k_kry_line_fused<1>})
            if ((e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLineSmem)) !=
                cudaSuccess)
                return e;
    }
    k_kry_rhs<T><<<sh.tiles, tb, 0, st>>>(g, tab, u, v, w, ws.r, ws.rt, rd(sh.ntile, kStRhs, 0));
    KRY_CHECK();
    const dim3 vt = vec_tiles(kp.nx, kp.ny, kp.nz);
    auto apply = [&](const T* x, T* y, const T* a, bool yy, int stage, int it) {
        if constexpr (sizeof(T) == 4) {
            if (kp.nx % 4 == 0 && vt.z <= 65535u) {          // (a grid's limit: 524280 levels)
                k_kry_apply4<<<vt, dim3(kVecX, kVecY), 0, st>>>(g, tab, x, y, a, yy,
                                                                rd((int)(vt.x * vt.y * vt.z), stage, it));
                return;
            }
        }
        k_kry_apply<T><<<sh.tiles, tb, 0, st>>>(g, tab, x, y, a, yy, rd(sh.ntile, stage, it));
    };
    KrySc h{};
    if ((e = cudaMemcpyAsync(&h, ws.sc, sizeof(KrySc), cudaMemcpyDeviceToHost, st)) != cudaSuccess) return e;
    if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
    for (int it = 1; it <= mi && !h.done; ++it) {
        const bool check = (it % kKryCheckEvery == 0) || it == mi;
        if constexpr (sizeof(T) == 4) {
            if (fuse)
                k_kry_line_fused<0><<<lblk, kLineThreads, lsm, st>>>(g, tab, ws.p, ws.r, ws.v, ws.ph, it == 1,
                                                                     rd(lblk, kStS, it));
        }
        if (!fuse)
            k_kry_p<T><<<nblk, kKryThreads, 0, st>>>(g, ws.p, ws.r, ws.v, it == 1, ws.sc);
        if (pc && !fuse) k_kry_line<T><<<cblk, kKryThreads, 0, st>>>(g, tab, ws.p, ws.ph, ws.sc);
        apply(ph, ws.v, ws.rt, false, kStAlpha, it);
        if constexpr (sizeof(T) == 4) {
            if (fuse)
                k_kry_line_fused<1><<<lblk, kLineThreads, lsm, st>>>(g, tab, ws.r, nullptr, ws.v, ws.sh, false,
                                                                     rd(lblk, kStS, it));
        }
        if (!fuse)
            k_kry_s<T><<<nblk, kKryThreads, 0, st>>>(g, ws.r, ws.v, rd(nblk, kStS, it));
        if (pc && !fuse) k_kry_line<T><<<cblk, kKryThreads, 0, st>>>(g, tab, ws.r, ws.sh, ws.sc);
        apply(shv, ws.t, ws.r, true, kStOmega, it);
        bool vec = false;
        if constexpr (sizeof(T) == 4) {
            vec = g.n % 4 == 0;
            if (vec)
                k_kry_update4<<<nblk, kKryThreads, 0, st>>>(g, ws.xh, ws.xl, ph, shv, ws.r, ws.t, ws.rt,
                                                            rd(nblk, kStR, it));
        }
        if (!vec)
            k_kry_update<T><<<nblk, kKryThreads, 0, st>>>(g, ws.xh, ws.xl, ph, shv, ws.r, ws.t, ws.rt,
                                                          rd(nblk, kStR, it));
        KRY_CHECK();
        if (!check) continue;
        if ((e = cudaMemcpyAsync(&h, ws.sc, sizeof(KrySc), cudaMemcpyDeviceToHost, st)) != cudaSuccess) return e;
        if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
    }
    k_kry_level0<T><<<cblk, kKryThreads, 0, st>>>(g.plane, ws.xh, ws.xl, rd(cblk, kStMean, 0));
    k_kry_correct<T><<<sh.tiles, tb, 0, st>>>(g, ws.xh, ws.xl, u, v, w, kp.idzn, (T*)kp.u_out, (T*)kp.v_out,
                                              (T*)kp.w_out, (T*)kp.phi_out, ws.sc);
    KRY_CHECK();
#undef KRY_CHECK
    res->iterations = h.done ? h.iters : mi;
    res->rel_residual = h.relres;
    res->status = h.done ? h.status : 1;
    return cudaSuccess;
}

}  // namespace

// Vertical rows of L, the divergence's vertical weights and the Thomas factors of
// the line matrix (formed in FP64): vsub, vdiag, vsup, lcp, livd, flo, fhi, nz values each.
std::vector<double> krylov_tables(int nz, double dx, double dy, const double* acoef, const double* svol,
                                  const double* rflo, const double* rfhi) {
    const double idx = 1.0 / dx, idy = 1.0 / dy, hdiag = -2.0 * idx * idx - 2.0 * idy * idy;
    std::vector<double> t((size_t)7 * nz);
    double cp = 0.0;
    for (int k = 0; k < nz; ++k) {
        const double iv = 1.0 / svol[k];
        const double sub = acoef[k] * iv, sup = acoef[k + 1] * iv;
        const double d0 = -(acoef[k] + acoef[k + 1]) * iv;
        const double ivd = 1.0 / ((d0 + hdiag) - (k > 0 ? sub * cp : 0.0));
        cp = (k < nz - 1) ? sup * ivd : 0.0;
        const double row[7] = {sub, d0, sup, cp, ivd, rflo[k] * iv, rfhi[k] * iv};
        for (int j = 0; j < 7; ++j) t[(size_t)j * nz + k] = row[j];
    }
    return t;
}

size_t krylov_workspace_bytes(int nx, int ny, int nz, int nsm, bool fp32) {
    size_t bytes = 0;
    const int np = shape(nx, ny, nz, nsm).nparts;
    if (fp32) carve<float>(nullptr, nx, ny, nz, np, &bytes);
    else carve<double>(nullptr, nx, ny, nz, np, &bytes);
    return bytes;
}

cudaError_t krylov_run(const KrylovProblem& kp, cudaStream_t st, KrylovResult* res) {
    return kp.fp32 ? run<float>(kp, st, res) : run<double>(kp, st, res);
}

}  // namespace mp
