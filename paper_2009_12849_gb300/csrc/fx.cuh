// Fourier transforms of FP64 data in 64-bit block fixed point.
//
// GB300's FP64 pipe does 1.7 fused multiply-adds per clock and SM; its integer
// pipes do 59 64-bit additions and 15 32 x 32 + 64-bit multiply-adds (measured).
// A transform (paper, Section 4: the pressure solver's forward and backward
// FFTs) is mostly additions, so the FP64 plans' transforms run on integers: the
// elements of one transform are scaled by a power of two, the butterflies add
// and subtract 64-bit integers and multiply by twiddles of 62 bits, and the
// results are rounded to doubles.
//
// Scale.  The largest element enters below 2^T0, T0 = 62 - ceil(log2 R0) >= 58, the
// most that the first stage's radix R0 leaves room for.  What the stages after it
// can reach is known from the data: every value that a transform forms is a sum of
// its elements times numbers of modulus 1 at most, so the sum of their moduli
// bounds it.  That sum is taken while the first stage runs (of |re| + |im|, in the high
// words); where it is 2^62 or more the second stage shifts its inputs down below
// that, and nothing is taken off after it.  A spectrum of a few large
// coefficients, which does not grow, keeps its bits so, and noise loses the 2 to 4
// that its sum calls for.  The shift rounds ties up and down in turn, and twiddles that
// are a power of i are exact, so no rounding has a bias, which would add up in a
// transform's mean.
//
// Accuracy: units of 2^-61 of the sum after the first stage are 2^-61 N / sqrt(R0) / 2.4 of
// the transform's norm at most (the sum is at most sqrt(N) times the norm), 6e-17 at
// 1024 = 16 16 4, and the entry at 2^-57 of the largest element up to 0.4 sqrt(N) 2^-57,
// 9e-17, where the largest element stands alone.  Against extended precision, rms,
// fixed point / FP64 butterflies: noise 0.8e-16 / 2.1e-16 at 1024, 1.0e-16 / 2.4e-16 at 1000,
// 0.7e-16 / 2.4e-16 at 405; a 1/k^2 spectrum 1.1e-16 / 1.8e-16, 1.2e-16 / 2.0e-16,
// 0.8e-16 / 2.3e-16; a mode over 1e-3 of noise 1.5e-16 / 1.7e-16, 1.7e-16 / 1.9e-16,
// 1.2e-16 / 1.8e-16; a mode alone 0.4e-16 / 0.8e-16 to 1.1e-16.  (Taking ceil(log2 R) bits off
// at every stage, as the growth of any input would need, gave that mode over
// noise 0.9e-15 at 1024 and 5.9e-15 at 1000.  The sum and the shift cost 2 to 9% of a
// solve: 64^3 101 -> 102 us, 256^2 x 128 856 -> 895, 360x300x75 1111 -> 1159, 512^2 x 64 1802 -> 1965,
// 1024^2 x 48 5.10 -> 5.52 ms.)
// Like a floating-point FFT, the error is relative to the whole transform, not to
// each element.  A transform with a NaN or an infinity gives NaN in all its
// elements.
#pragma once
#include "kernels.cuh"

namespace mp {

struct fx {
    long long v;
    fx() = default;
    // constants: |c| <= 1 as c 2^62
    MP_HD constexpr explicit fx(double c) : v((long long)(c * 4611686018427387904.0 + (c < 0 ? -0.5 : 0.5))) {}
    MP_HD constexpr explicit fx(dd c) : v(dd_fixed(c, 62)) {}
    static MP_HD fx raw(long long v) { fx r; r.v = v; return r; }
};
MP_HD fx operator+(fx a, fx b) { return fx::raw(a.v + b.v); }
MP_HD fx operator-(fx a, fx b) { return fx::raw(a.v - b.v); }
MP_HD fx operator-(fx a) { return fx::raw(-a.v); }
MP_HD fx& operator+=(fx& a, fx b) { a.v += b.v; return a; }
MP_HD fx& operator-=(fx& a, fx b) { a.v -= b.v; return a; }
MP_HD fx operator*(int s, fx a) { return s > 0 ? a : -a; }          // s = +1 or -1

struct alignas(16) fx2 {
    fx x, y;
};
template <> struct CT<fx> { using T = fx2; };

// Balanced words: v = hi 2^32 + lo, lo signed.  The products below leave out low x
// low, which is then zero on average: left out of unsigned words it is a bias of
// half a unit that adds up in a transform's lowest frequencies (the velocities'
// errors there were three times as large).
MP_HD int fx_lo(long long v) { return (int)v; }
MP_HD int fx_hi(long long v) { return (int)(v >> 32) + (int)((unsigned)v >> 31); }

// A constant c 2^62 times data: (b a) / 2^62.
MP_HD fx operator*(fx b, fx a) {
    const int ah = fx_hi(a.v), al = fx_lo(a.v), bh = fx_hi(b.v), bl = fx_lo(b.v);
    const long long c = (long long)ah * bl + (long long)al * bh + (1ll << 29);
    return fx::raw((((long long)ah * bh) << 2) + (c >> 30));
}

MP_HD fx2 cscale(fx2 a, fx s) { a.x = s * a.x; a.y = s * a.y; return a; }

// (a w) / 2^(64 - UP); the cross products stay below 2^63 with |a| <= 2^62.5 and |w| <=
// 2^62 as complex moduli.
template <int UP> MP_HD fx2 fx_product(fx2 a, fx2 w) {
    const int rh = fx_hi(a.x.v), rl = fx_lo(a.x.v), ih = fx_hi(a.y.v), il = fx_lo(a.y.v);
    const int wrh = fx_hi(w.x.v), wrl = fx_lo(w.x.v), wih = fx_hi(w.y.v), wil = fx_lo(w.y.v);
    const long long half = 1ll << (31 - UP);
    const long long cr = (long long)rh * wrl + (long long)rl * wrh - (long long)ih * wil - (long long)il * wih + half;
    const long long ci = (long long)rh * wil + (long long)rl * wih + (long long)ih * wrl + (long long)il * wrh + half;
    fx2 o;
    o.x.v = (((long long)rh * wrh - (long long)ih * wih) << UP) + (cr >> (32 - UP));
    o.y.v = (((long long)rh * wih + (long long)ih * wrh) << UP) + (ci >> (32 - UP));
    return o;
}
// (a w) / 2^62 for w 2^62: a twiddle, a gradient symbol or a constant
MP_HD fx2 cmul(fx2 a, fx2 w) { return fx_product<2>(a, w); }
MP_HD fx2 cmulc(fx2 a, fx2 w) {
    w.y = fx::raw(-w.y.v);
    return cmul(a, w);
}

// v / 2^L (L >= 1), ties to even (rounding them up, as an odd value's half always is, is
// a bias of a quarter unit per 3-point transform).
MP_HD fx fx_shr(fx a, int L) {
    return fx::raw((a.v + (((1ll << (L - 1)) - 1) + ((a.v >> L) & 1))) >> L);
}
template <int S> struct Dft3<fx, S> {
    static MP_HD void run(fx2* x) {
        constexpr fx c(dd_sincos2pi(1, 3).s);
        const fx2 t = cadd(x[1], x[2]), d = csub(x[1], x[2]);
        fx2 m;
        m.x = x[0].x - fx_shr(t.x, 1);
        m.y = x[0].y - fx_shr(t.y, 1);
        const fx2 r = cscale(cmul_si(d, S), c);
        x[0] = cadd(x[0], t);
        x[1] = cadd(m, r);
        x[2] = csub(m, r);
    }
};
template <> struct DftConst<fx> {
    template <int M, int N, bool SIN> static MP_HD constexpr fx get(double) {
        constexpr dd_pair w = dd_sincos2pi(M, N);
        return fx(SIN ? w.s : w.c);
    }
};

// v e^{i t} with a compile-time angle (the composite register DFTs)
template <class Tw> MP_HD fx2 ct_rot_fx(fx2 v) {
    constexpr double c = Tw::re, s = Tw::im;
    fx2 o;
    if constexpr (c == 0.0) {
        o.x = s > 0 ? -v.y : v.y;
        o.y = s > 0 ? v.x : -v.x;
    } else if constexpr (s == 0.0) {
        o.x = c > 0 ? v.x : -v.x;
        o.y = c > 0 ? v.y : -v.y;
    } else if constexpr ((c > 0 ? c : -c) - (s > 0 ? s : -s) < 1e-15 && (c > 0 ? c : -c) - (s > 0 ? s : -s) > -1e-15) {
        // an odd eighth of a turn: (+-x +-y) / sqrt(2)
        constexpr fx h = DftConst<fx>::get<1, 8, false>(0.0);
        const fx a = c > 0 ? v.x : -v.x, b = s > 0 ? v.y : -v.y;
        const fx d = s > 0 ? v.x : -v.x, e = c > 0 ? v.y : -v.y;
        o.x = h * (a - b);
        o.y = h * (d + e);
    } else {
        // constants c 2^62
        constexpr fx C(Tw::wide().c), S(Tw::wide().s);
        fx2 w;
        w.x = C;
        w.y = S;
        o = cmul(v, w);
    }
    return o;
}

// Elements per thread of a length's fixed-point plan.  Powers of two: 16 (two
// stages at 256; with 8, three, the columns took 940 us of a 256^2 x 128 solve
// against 879).  Other lengths: of the candidates whose stages hold at most 16
// elements (64 registers) the one with the fewest stages, then the fewest
// elements: radices 15 and 16 of such lengths spilled 1 to 2 KB a thread (a 135^2 x
// 64 solve 286 us against 202 with 9 5 3).
MP_HD constexpr int fx_ept(int N) {
    if ((N & (N - 1)) == 0) return 16;
    int best = 8, stages = 99, held = 99;
    const int cand[4] = {12, 10, 9, 8};
    for (int c = 0; c < 4; ++c) {
        const int E = cand[c];
        int s = 0, most = 0;
        for (int m = N; m > 1; ++s) {
            const int r = ct_radix(m, E);
            const int h = ((E + r - 1) / r) * r;
            if (h > most) most = h;
            m /= r;
        }
        if (most <= 16 && s > 1 && (s < stages || (s == stages && most < held))) {
            stages = s;
            held = most;
            best = E;
        }
    }
    return best;
}
// The largest element of a transform enters below 2^T0 (moduli below 2^(T0 + 1/2),
// so that the first stage's sums stay below 2^62.5).
MP_HD constexpr int fx_t0(int N, int E) {
    int l = 0;
    while ((1 << l) < ct_stage_radix(N, 1, E)) ++l;
    return 62 - l;
}
// Sum of a butterfly's |re| + |im| in units of 2^42, rounded up: of the high words,
// |v| < (|v|'s + 1) 2^32 (below 2^31, since RAD 2^T0 <= 2^62; 1024 elements below 2^30).
template <int RAD> MP_HD int fx_sum(const fx2* x) {
    unsigned s = 2 * RAD;
#pragma unroll
    for (int r = 0; r < RAD; ++r) {
        const int a = (int)(x[r].x.v >> 32), b = (int)(x[r].y.v >> 32);
        s += (unsigned)(a ^ (a >> 31)) + (unsigned)(b ^ (b >> 31));
    }
    return (int)(s >> 10) + 1;
}
// Bits that a transform whose butterflies' sums add up to `sum` is shifted down by to
// stay below 2^62, with a 64th of it spare for the roundings of all stages (and
// half of what a word holds: the forward rows add two results).
MP_HD int fx_shift(int sum) {
    const unsigned s = (unsigned)sum + ((unsigned)sum >> 6) + 2;
    int bits = 0;
#if defined(__CUDA_ARCH__)
    bits = 32 - __clz((int)s);
#else
    while (s >> bits) ++bits;
#endif
    return bits > 20 ? bits - 20 : 0;
}

// Per transform of the block's task: its largest element's high word (as a double's)
// and the sum of its elements' moduli, zero before fx_first.
constexpr int kFxMaxBatch = 32;
struct FxTask {
    int mag[kFxMaxBatch], sum[kFxMaxBatch];
};
__device__ __forceinline__ FxTask& fx_task() {
    __shared__ FxTask t;
    return t;
}
__device__ __forceinline__ void fx_clear() {
    if (threadIdx.x < kFxMaxBatch) fx_task().mag[threadIdx.x] = fx_task().sum[threadIdx.x] = 0;
}

template <> struct StageIn<fx> {
    template <int RAD, bool SECOND> static __device__ __forceinline__ void run(fx2* x, int b, int q) {
        if constexpr (SECOND) {
            const int sh = fx_shift(fx_task().sum[b]);
            if (sh > 0) {
                // ties up and down in turn: no bias
                const long long even = (1ll << (sh - 1)) - (q & 1), odd = (1ll << (sh - 1)) - 1 + (q & 1);
#pragma unroll
                for (int r = 0; r < RAD; ++r) {
                    const long long half = (r & 1) ? odd : even;
                    x[r].x.v = (x[r].x.v + half) >> sh;
                    x[r].y.v = (x[r].y.v + half) >> sh;
                }
            }
        }
    }
};
template <class Tw> struct CtRot<fx, Tw> {
    static MP_HD fx2 run(fx2 v) { return ct_rot_fx<Tw>(v); }
};
__device__ __forceinline__ fx2 tw_load(const fx2* a) {
    const longlong2 t = __ldg((const longlong2*)a);
    fx2 r;
    r.x.v = t.x;
    r.y.v = t.y;
    return r;
}

// d in units of the transform's scale: m = (largest element's high word) gives
// the exponent E, and |d| < 2^(E - 1022) becomes |result| < 2^T0.
template <int T0> __device__ __forceinline__ long long fx_from(double d, int E) {
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    const int e = (hi >> 20) & 0x7ff;
    const unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | (e ? 0x100000u : 0u)) << 32) | lo;
    const unsigned sh = (unsigned)min(E - max(e, 1), 63);
    const long long q = (long long)((m << (T0 - 53)) >> sh);
    return ((int)hi < 0) ? -q : q;
}
// v 2^x as a double, rounded to nearest (results below the normal range become zero)
__device__ __forceinline__ double fx_to(long long v, int x, bool bad) {
    const unsigned long long a = (unsigned long long)(v < 0 ? -v : v);
    const int lz = __clzll((long long)a);
    const unsigned long long n = a << (lz & 63);
    const unsigned long long m = (n >> 11) + ((n >> 10) & 1ull);     // 53 bits (a carry goes into the exponent)
    const int e = x + 63 - lz + 1023;
    unsigned long long b = m + ((unsigned long long)(unsigned)(e - 1) << 52);
    if (e < 1 || a == 0) b = 0;
    if (e > 2046) b = 0x7ff0000000000000ull;
    if (bad) b = 0x7ff8000000000000ull;
    return __longlong_as_double((long long)(b | ((unsigned long long)v & 0x8000000000000000ull)));
}
// what transform b's record says
struct FxScale {
    int E;             // exponent field of the largest element (at least 1)
    int shift;         // before the second stage
    bool bad;          // a NaN or an infinity among them
    __device__ __forceinline__ explicit FxScale(int b) {
        const int m = fx_task().mag[b];
        E = max(m >> 20, 1);
        bad = (m >> 20) == 0x7ff;
        shift = fx_shift(fx_task().sum[b]);
    }
    // power of two of a result of a length-N transform
    template <int N> __device__ __forceinline__ int out() const { return E - 1022 - fx_t0(N, fx_ept(N)) + shift; }
    // emit(to): hands out results, to(v) = v 2^x.  A transform that can have results below
    // the normal range forms them 2^128 times as large first, in code of its own: the
    // FP64 pipe is this GPU's scarce resource, and almost none does.
    template <class Emit> __device__ __forceinline__ void results(int x, Emit&& emit) const {
        if (x >= -1022) emit([&](long long v) { return fx_to(v, x, bad); });
        else emit([&](long long v) { return fx_to(v, x + 128, bad) * 0x1p-128; });
    }
};
__device__ __forceinline__ int fx_mag(double d) { return __double2hiint(d) & 0x7fffffff; }

// Maximum and sum over butterflies into shared memory.  Where runs of the NQ
// threads of a transform are whole warps or equal parts of one, a run's lanes are
// reduced first (all of its lanes are active).
template <int NQ> struct FxRun {
    static constexpr int W = NQ % 32 == 0 ? 32 : 32 % NQ == 0 ? NQ : 1;
    static __device__ __forceinline__ unsigned mask() {
        return W == 32 ? 0xffffffffu : ((1u << (W & 31)) - 1u) << ((threadIdx.x & 31) / W * W);
    }
    static __device__ __forceinline__ bool first() { return threadIdx.x % W == 0; }
};
template <int NQ> __device__ __forceinline__ void fx_collect_max(int* to, int m) {
    if constexpr (FxRun<NQ>::W > 1) {
        m = __reduce_max_sync(FxRun<NQ>::mask(), m);
        if (!FxRun<NQ>::first()) return;
    }
    atomicMax(to, m);
}
template <int NQ> __device__ __forceinline__ void fx_collect_sum(int* to, int m) {
    if constexpr (FxRun<NQ>::W > 1) {
        m = __reduce_add_sync(FxRun<NQ>::mask(), m);
        if (!FxRun<NQ>::first()) return;
    }
    atomicAdd(to, m);
}

// First stage: fetch(b, q, r) gives what element q + r N/RAD of transform b is
// made from; fx_task() (cleared, synchronised) collects each transform's largest
// element, as a double's high word, and its sum of moduli.  RELOAD: magnitude(raw) bounds an element and
// conv(raw, E) gives it scaled by the transform's exponent E; it is fetched again
// for that (from L1) instead of waiting in registers.  Otherwise magnitude(raws, b,
// q) and conv(raws, E, b, q, x) take a butterfly's elements at once.
template <int N, int S, bool BFAST, bool RELOAD, class Fetch, class Mag, class Conv>
__device__ __forceinline__ void fx_first(fx2* buf, int nb, int bstride, Fetch&& fetch, Mag&& magnitude, Conv&& conv) {
    constexpr int E = fx_ept(N);
    static_assert(N <= 1024, "sums of moduli in 31 bits");
    int* mag = fx_task().mag;
    using SI = StageInfo<fx, N, 1, E>;
    constexpr int RAD = SI::RAD, NQ = SI::NQ, NB = (E + RAD - 1) / RAD;
    const int total = NQ * nb;
    using Raw = decltype(fetch(0, 0, Ic<0>{}));
    Raw d[RELOAD ? 1 : NB][RELOAD ? 1 : RAD];
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        const int t = threadIdx.x + i * blockDim.x;
        if (t < total) {
            int b, q, m = 0;
            bfly_map<BFAST, NQ>(t, nb, b, q);
            if constexpr (RELOAD) {
                SFor<0, RAD>::run([&](auto r) { m = max(m, magnitude(fetch(b, q, r))); });
                fx_collect_max<BFAST ? 1 : NQ>(&mag[b], m);
            } else {
                SFor<0, RAD>::run([&](auto r) { d[i][r] = fetch(b, q, r); });
            }
        }
    }
    if constexpr (!RELOAD) {
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const int t = threadIdx.x + i * blockDim.x;
            if (t < total) {
                int b, q, m = 0;
                bfly_map<BFAST, NQ>(t, nb, b, q);
                m = magnitude(d[i], b, q);
                fx_collect_max<BFAST ? 1 : NQ>(&mag[b], m);
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        const int t = threadIdx.x + i * blockDim.x;
        if (t < total) {
            int b, q;
            bfly_map<BFAST, NQ>(t, nb, b, q);
            const int ex = max(mag[b] >> 20, 1);
            fx2 x[RAD];
            if constexpr (RELOAD) SFor<0, RAD>::run([&](auto r) { x[r] = conv(fetch(b, q, r), ex); });
            else conv(d[i], ex, b, q, x);
            fx_collect_sum<BFAST ? 1 : NQ>(&fx_task().sum[b], fx_sum<RAD>(x));
            RegFFT<fx, RAD, S>::run(x);
            fx2* d0 = buf + b * bstride + q * (RAD + SPad<fx, N, E>::PAD);
#pragma unroll
            for (int r = 0; r < RAD; ++r) d0[r] = x[r];
        }
    }
    __syncthreads();
}
// elements that are double2 themselves
template <int RAD> __device__ __forceinline__ int fx_magnitude(const double2* d) {
    int m = 0;
#pragma unroll
    for (int r = 0; r < RAD; ++r) m = max(m, max(fx_mag(d[r].x), fx_mag(d[r].y)));
    return m;
}
template <int RAD, int T0> __device__ __forceinline__ void fx_convert(const double2* d, int E, fx2* x) {
#pragma unroll
    for (int r = 0; r < RAD; ++r) {
        x[r].x.v = fx_from<T0>(d[r].x, E);
        x[r].y.v = fx_from<T0>(d[r].y, E);
    }
}

// ---------------------------------------------------------------------------
// a1 + a2 (x part) of FP64 plans (the task of k_fwd_rows)
// ---------------------------------------------------------------------------
template <int NX>
__global__ void __launch_bounds__(512, 1) k_fwd_rows_fx(ProjParams p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int ny = p.ny, rows = p.rows_fwd, npair = rows / 2, bs = p.bs_row;
    const int k = blockIdx.x / p.nrb_fwd;
    const int j0 = (blockIdx.x - k * p.nrb_fwd) * rows;
    fx2* buf = (fx2*)smem_raw;
    const size_t plane = (size_t)ny * NX;
    const int kg = p.kbase + k;
    const bool below = kg > 0, above = kg < p.nz_glob - 1;
    const double cx = p.svol[kg] * p.idx, cy = p.svol[kg] * p.idy, rlo = p.rflo[kg], rhi = p.rfhi[kg];
    fx_clear();
    // the divergence goes to the transforms' buffer as doubles
    for (int r = 0; r < rows; ++r) {
        const int j = j0 + r;
        const size_t row = (size_t)k * plane + (size_t)j * NX;
        const double* ur = (const double*)p.u + row;
        const double* vr = (const double*)p.v + row;
        const double* vs = (const double*)p.v + ((size_t)k * plane + (size_t)(j == 0 ? ny - 1 : j - 1) * NX);
        const double* wr = (const double*)p.w + row;
        double* slot = (double*)&buf[(r >> 1) * bs] + (r & 1);
        constexpr int B = 4;
        for (int i0 = threadIdx.x; i0 < NX; i0 += B * blockDim.x) {
            double uc[B], um[B], vc[B], vm[B], wl[B], wh[B];
#pragma unroll
            for (int c = 0; c < B; ++c) {
                const int i = i0 + c * blockDim.x;
                uc[c] = um[c] = vc[c] = vm[c] = wl[c] = wh[c] = 0.0;
                if (i < NX && j < ny) {
                    uc[c] = ur[i];
                    um[c] = ur[i == 0 ? NX - 1 : i - 1];
                    vc[c] = vr[i];
                    vm[c] = vs[i];
                    if (below) wl[c] = wr[i];
                    if (above) wh[c] = (wr + plane)[i];
                }
            }
#pragma unroll
            for (int c = 0; c < B; ++c) {
                const int i = i0 + c * blockDim.x;
                if (i < NX)
                    slot[2 * SPad<fx, NX, fx_ept(NX)>::sp(i)] =
                        fma(cx, uc[c] - um[c], fma(cy, vc[c] - vm[c], fma(rhi, wh[c], -rlo * wl[c])));
            }
        }
    }
    __syncthreads();
    using SP = SPad<fx, NX, fx_ept(NX)>;
    const double2* in = (const double2*)buf;
    auto load = [&](int b, int q, auto r) -> double2 {
        constexpr int NQ = StageInfo<fx, NX, 1, fx_ept(NX)>::NQ;
        return in[b * bs + SP::sp(q + r * NQ)];
    };
    constexpr int RAD = StageInfo<fx, NX, 1, fx_ept(NX)>::RAD, T0 = fx_t0(NX, fx_ept(NX));
    // (the buffer is overwritten: every element waits in registers)
    fx_first<NX, -1, false, false>(
        buf, npair, bs, load, [](const double2* d, int, int) { return fx_magnitude<RAD>(d); },
        [](const double2* d, int E, int, int, fx2* x) { fx_convert<RAD, T0>(d, E, x); });
    CtFFT<fx, NX, StageInfo<fx, NX, 1, fx_ept(NX)>::NEXT, -1, BlockScope, fx_ept(NX)>::run(buf, npair, bs, (const fx2*)p.twx);
    double2* T = (double2*)p.T;
    const int nxh = p.nxh;
    for (int q = 0; q < npair; ++q) {
        const int j = j0 + 2 * q;
        if (j >= ny) break;
        const FxScale sc(q);
        const int x = sc.out<NX>() - 1;                  // the halves of the split
        const fx2* rq = buf + q * bs;
        double2* to = T + ((size_t)k * ny + j) * p.nxp;
        const bool second = j + 1 < ny;
        for (int kx = threadIdx.x; kx < nxh; kx += blockDim.x) {
            const fx2 z = rq[SP::sp(kx)];
            const fx2 zm = rq[SP::sp(kx == 0 ? 0 : NX - kx)];
            sc.results(x, [&](auto d) {
                to[kx] = make_double2(d(z.x.v + zm.x.v), d(z.y.v - zm.y.v));
                if (second) to[kx + p.nxp] = make_double2(d(z.y.v + zm.y.v), d(zm.x.v - z.x.v));
            });
        }
    }
}

// ---------------------------------------------------------------------------
// Column transforms of FP64 plans: field f as in inv_col_field, f < 0 forward
// (T -> S).
// ---------------------------------------------------------------------------
template <int NY, int S>
__device__ __forceinline__ void fx_cols_task(const ProjParams& p, fx2* buf, int k, int kx0, int f) {
    const int nxh = p.nxh, nxp = p.nxp, tw = p.tw_cols, bs = p.bs_col;
    const size_t tile = (size_t)k * NY * nxp + kx0;
    const double2* src = (S < 0 ? (const double2*)p.T : f == 2 ? (const double2*)p.G : (const double2*)p.S) + tile;
    double2* dst = (S < 0 ? (double2*)p.S
                          : f == 0 ? (double2*)p.Tp : f == 1 ? (double2*)p.Tgy : f == 2 ? (double2*)p.Tgz : (double2*)p.Tphi) + tile;
    fx_clear();
    __syncthreads();
    constexpr int NQ = StageInfo<fx, NY, 1, fx_ept(NY)>::NQ, T0 = fx_t0(NY, fx_ept(NY));
    auto fetch = [&](int c, int q, auto r) -> double2 {
        return kx0 + c < nxh ? src[(q + r * NQ) * nxp + c] : make_double2(0.0, 0.0);
    };
    constexpr int RAD = StageInfo<fx, NY, 1, fx_ept(NY)>::RAD;
    // f = 1, p^ ey: each element is scaled by its own exponent, multiplied by the
    // normalised ey and brought to the transform's scale
    const fx2* ey = (const fx2*)p.ey_fx;
    const int* eye = p.ey_exp;
    auto magnitude = [&](const double2* d, int, int q) -> int {
        if (!(S > 0 && f == 1)) return fx_magnitude<RAD>(d);
        int m = 0;
#pragma unroll
        for (int r = 0; r < RAD; ++r) {
            const int e = max(fx_mag(d[r].x), fx_mag(d[r].y)) >> 20;
            m = max(m, e == 0x7ff ? e : min(e + eye[q + r * NQ] + 1, 2046));
        }
        return m << 20;
    };
    constexpr int UP = T0 <= 59 ? 0 : 2;     // (the shift below is by E - e - eye >= 1 at least)
    static_assert(T0 <= 61, "products brought down to the transform's scale");
    auto conv = [&](const double2* d, int E, int, int q, fx2* x) {
        if (!(S > 0 && f == 1)) {
            fx_convert<RAD, T0>(d, E, x);
            return;
        }
#pragma unroll
        for (int r = 0; r < RAD; ++r) {
            const int j = q + r * NQ;
            const int e = max(max(fx_mag(d[r].x), fx_mag(d[r].y)) >> 20, 1);
            x[r].x.v = fx_from<61>(d[r].x, e);
            x[r].y.v = fx_from<61>(d[r].y, e);
            x[r] = fx_product<UP>(x[r], tw_load(&ey[j]));            // 2^(59 + UP) for 1
            const int sh = min(max(E - e - eye[j] + 59 + UP - T0, 1), 63);
            x[r].x = fx_shr(x[r].x, sh);
            x[r].y = fx_shr(x[r].y, sh);
        }
    };
    fx_first<NY, S, true, false>(buf, tw, bs, fetch, magnitude, conv);
    CtMid<fx, NY, StageInfo<fx, NY, 1, fx_ept(NY)>::NEXT, S, BlockScope, fx_ept(NY)>::run(buf, tw, bs, (const fx2*)p.twy);
    auto store = [&](int c, int q, fx2* x, int ns) {
        if (kx0 + c >= nxh) return;
        constexpr int LRAD = StageInfo<fx, NY, LastNs<fx, NY, fx_ept(NY)>::value, fx_ept(NY)>::RAD;
        const FxScale sc(c);
        int xp = sc.out<NY>();
        if (S < 0) xp += p.scale_exp;
        double2* d = dst + q * nxp + c;
        if (S > 0 && f == 0) {
            const fx2 e = tw_load((const fx2*)p.ex_fx + kx0 + c);
            xp += p.ex_exp[kx0 + c];
#pragma unroll
            for (int r = 0; r < LRAD; ++r) x[r] = cmul(x[r], e);
        }
        if constexpr (S < 0) {
            sc.results(xp, [&](auto to) {
#pragma unroll
                for (int r = 0; r < LRAD; ++r) d[r * ns * nxp] = make_double2(to(x[r].x.v), to(x[r].y.v));
            });
        } else {
            // this kernel waits for its instructions (2.6 of 8.2 cycles between a warp's issues
            // at 256^2): one copy of its stores, with the multiplication predicated
            // (512^2 x 64 inverse columns 755 us, 820 with two; the forward ones are slower so:
            // 72 against 68 at 256^2 x 128)
            const bool tiny = xp < -1022;
            if (tiny) xp += 128;
#pragma unroll
            for (int r = 0; r < LRAD; ++r) {
                double2 v = make_double2(fx_to(x[r].x.v, xp, sc.bad), fx_to(x[r].y.v, xp, sc.bad));
                if (tiny)
                    asm volatile("mul.rn.f64 %0, %0, %2;\n\tmul.rn.f64 %1, %1, %2;" : "+d"(v.x), "+d"(v.y) : "d"(0x1p-128));
                d[r * ns * nxp] = v;
            }
        }
    };
    ct_last<fx, NY, S, true, BlockScope, fx_ept(NY)>(buf, tw, bs, (const fx2*)p.twy, store);
}

template <int NY>
__global__ void __launch_bounds__(512, 1) k_fwd_cols_fx(ProjParams p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int k = blockIdx.x / p.ntiles;
    fx_cols_task<NY, -1>(p, (fx2*)smem_raw, k, (blockIdx.x - k * p.ntiles) * p.tw_cols, -1);
}

// task = (level, tile, kind): kind 0 the p^ tile's fields, kind 1 gz^ (as k_inv_cols)
template <int NY>
__global__ void __launch_bounds__(512, 1) k_inv_cols_fx(ProjParams p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int kind = blockIdx.x & 1;
    const int task = blockIdx.x >> 1;
    const int k = task / p.ntiles;
    const int kx0 = (task - k * p.ntiles) * p.tw_cols;
    if (kind == 1 && p.kbase + k == 0) return;
    const int last = kind == 1 ? 2 : p.nch == 4 ? 3 : 1;
    int f = kind == 1 ? 2 : 0;
#pragma unroll 1
    while (true) {
        fx_cols_task<NY, 1>(p, (fx2*)smem_raw, k, kx0, f);
        if (f == last) break;
        f = f == 1 ? 3 : f + 1;
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// a4 (x part) + a5 of FP64 plans (the task of k_inv_rows: one channel of
// rows_inv rows)
// ---------------------------------------------------------------------------
template <int NX>
__global__ void __launch_bounds__(512, 1) k_inv_rows_fx(ProjParams p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int ny = p.ny, nxp = p.nxp, rows = p.rows_inv, npr = rows / 2, bs = p.bs_row;
    const int ch = blockIdx.x % p.nch;
    const int t2 = blockIdx.x / p.nch;
    const int k = t2 / p.nrb_inv;
    const int j0 = (t2 - k * p.nrb_inv) * rows;
    const size_t plane = (size_t)ny * NX;
    fx2* buf = (fx2*)smem_raw;
    double* out = (ch == 0) ? (double*)p.uo : (ch == 1) ? (double*)p.vo : (ch == 2) ? (double*)p.wo : (double*)p.phi;
    const int kg = p.kbase + k;
    const bool top = kg == p.nz_glob - 1;
    if (ch == 2 && kg == 0) {
        // bottom face: w = 0
        for (int t = threadIdx.x; t < rows * NX; t += blockDim.x) {
            const int j = j0 + t / NX;
            if (j < ny) {
                out[(size_t)j * NX + (t % NX)] = 0.0;
                if (top) out[plane + (size_t)j * NX + (t % NX)] = 0.0;       // top face too
            }
        }
        return;
    }
    const double* in = (ch == 0) ? (const double*)p.u : (ch == 1) ? (const double*)p.v : (const double*)p.w;
    const bool upd = ch < 3;
    const double2* spec = inv_channel_spectrum<double>(p, ch) + (size_t)k * ny * nxp;
    fx_clear();
    __syncthreads();
    // z = A_j + i A_{j+1}, added as integers
    struct Raw {
        double2 a, c;
    };
    auto fetch = [&](int b, int q, auto r) -> Raw {
        const int j = j0 + 2 * b;
        Raw w{make_double2(0.0, 0.0), make_double2(0.0, 0.0)};
        if (j < ny) w.a = hermitian_elem<double, NX, fx_ept(NX)>(spec + (size_t)j * nxp, q, r);
        if (j + 1 < ny) w.c = hermitian_elem<double, NX, fx_ept(NX)>(spec + (size_t)(j + 1) * nxp, q, r);
        return w;
    };
    auto magnitude = [](Raw w) -> int {          // twice the largest part
        const int m = max(max(fx_mag(w.a.x), fx_mag(w.a.y)), max(fx_mag(w.c.x), fx_mag(w.c.y)));
        return m < 0x7fe00000 ? m + (1 << 20) : 0x7ff00000;
    };
    auto conv = [](Raw w, int E) -> fx2 {
        constexpr int T0 = fx_t0(NX, fx_ept(NX));
        fx2 z;
        z.x.v = fx_from<T0>(w.a.x, E) - fx_from<T0>(w.c.y, E);
        z.y.v = fx_from<T0>(w.a.y, E) + fx_from<T0>(w.c.x, E);
        return z;
    };
    fx_first<NX, 1, false, true>(buf, npr, bs, fetch, magnitude, conv);
    CtMid<fx, NX, StageInfo<fx, NX, 1, fx_ept(NX)>::NEXT, 1, BlockScope, fx_ept(NX)>::run(buf, npr, bs, (const fx2*)p.twx);
    constexpr int LRAD = StageInfo<fx, NX, LastNs<fx, NX, fx_ept(NX)>::value, fx_ept(NX)>::RAD;
    constexpr int LNB = (fx_ept(NX) + LRAD - 1) / LRAD;
    // outputs may alias inputs: a butterfly's operands are loaded before it writes
    double prev[LNB][2][LRAD];
    auto pre = [&](int b, int q, int ns, int i) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = j0 + 2 * b + h;
            const size_t row = (size_t)k * plane + (size_t)j * NX + q;
#pragma unroll
            for (int r = 0; r < LRAD; ++r) prev[i][h][r] = (upd && j < ny) ? in[row + r * ns] : 0.0;
        }
    };
    auto store = [&](int b, int q, const fx2* x, int ns, int i) {
        const FxScale sc(b);
        const int xp = sc.out<NX>();
        sc.results(xp, [&](auto to) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int j = j0 + 2 * b + h;
                if (j >= ny) continue;
                const size_t row = (size_t)k * plane + (size_t)j * NX + q;
#pragma unroll
                for (int r = 0; r < LRAD; ++r) {
                    const double val = to(h ? x[r].y.v : x[r].x.v);
                    out[row + r * ns] = upd ? prev[i][h][r] - val : val;
                    if (ch == 2 && top) out[row + r * ns + plane] = 0.0;
                }
            }
        });
    };
    ct_last_pre<fx, NX, 1, false, BlockScope, fx_ept(NX)>(buf, npr, bs, (const fx2*)p.twx, pre, store);
}

}  // namespace mp
