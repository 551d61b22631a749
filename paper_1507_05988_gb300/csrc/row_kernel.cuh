// row_kernel.cuh -- the row stage of the FCN z-step: FFTs along tau fused with
// the nonlinear half steps (Ma & Lin, arXiv:1507.05988, Sec. 3.1 first/third
// loops, Sec. 3.2, Eqs. (Anhalf)/(Anhalf1), and the re-organised step of
// Sec. 4 where the nonlinear part and the transforms share the radial
// decomposition).
//
// One row (fixed radial index m) is one independent unit of work, on Nt/16
// threads with E = 16 complex values each (E = Nt when Nt < 16; E = 4 on
// grids of few rows), or two adjacent rows on as many threads in packed
// arithmetic.
//
// Transform: in-place decimation-in-time FFT (one radix 2/4/8 pass for the
// factor left by radix 16, then radix-16 passes) in one padded shared-memory
// buffer with the butterfly operands in registers; every pass reads and
// writes the same positions in the same thread, so one barrier per pass
// suffices.  The forward transform takes the time samples in mixed-radix
// digit-reversed order (tpos) and leaves natural frequency order; the
// inverse transform is its exact adjoint (the forward passes in reverse
// order, transposed, with conjugate constants).  The first inverse pass
// reads HBM directly and the last forward pass writes HBM directly, in
// natural frequency order; both are coalesced (consecutive threads touch
// consecutive complex values).  Shared-memory rows are padded by one value
// per 16 so that the passes and the nonlinear stage's per-thread samples are
// free of bank conflicts.
//
// Nonlinear half step (Eq. (nonlinearpart)):  A <- A exp(h N(I, rho)).
// rho(tau) follows Eq. (ionization) integrated by RK4 along tau from
// rho(tau_min) = 0, with the RK4 midpoint intensity the mean of the two
// neighbours.  Because the ODE is linear in u = rho/rho_nt, one RK4 step is
// u_{p+1} = u_p + c_p (1 - u_p) with c_p a function of I_p and I_{p+1} only, so
// u_p = c_0 (+) c_1 (+) ... (+) c_{p-1} for the associative, commutative
// operation a (+) b = a + b - a b = 1 - (1-a)(1-b).  That makes the
// integration an exclusive parallel scan: sequential over each thread's 16
// points, warp shuffles across threads, and (rows wider than a warp) an FP64
// scan of the warp totals.  (+) never cancels (all terms are in [0, 1]), so
// the scan keeps the relative precision of the working type.
#pragma once
#include <type_traits>

#include "pack.cuh"

namespace fcn {
namespace {

// The element of a thread from the values of its rows (x[0 .. L-1]), and back.
template <typename V>
__device__ __forceinline__ cx<V> pack_rows(const cx<typename Pack<V>::S> *x) {
    if constexpr (Pack<V>::L == 2) return mk(pk2{x[0].x, x[1].x}, pk2{x[0].y, x[1].y});
    else return x[0];
}
template <typename V>
__device__ __forceinline__ cx<typename Pack<V>::S> row_of(cx<V> v, int lane) {
    if constexpr (Pack<V>::L == 2) return lane ? mk(v.x.b, v.y.b) : mk(v.x.a, v.y.a);
    else return v;
}

constexpr int ilog2(int n) { return n <= 1 ? 0 : 1 + ilog2(n / 2); }

// FP64 scratch per CTA for the cross-warp parts of the row scans and
// reductions (rows per CTA x warps per row x values <= 64)
constexpr int kRowScratch = 64;

// NT is the row length with the FFT plan in its high bits (fft_tag); N is
// the length itself.
template <int NT>
struct RowCfg {
    static constexpr int N = fft_nt(NT);                    // points per row
    static constexpr int PLAN = fft_plan(NT);               // FFT decomposition
    static constexpr int E = PLAN == 2 ? 4 : N < 16 ? N : 16;   // values per thread
    static constexpr int TPR = N / E;                       // threads per row
    static constexpr int THREADS = TPR >= 256 ? TPR : 256;  // CTA size
    static constexpr int PADN = N >= 16 ? N + N / 16 : N;
    static constexpr int NPASS = fft_npass(NT);
    static constexpr int WARPS_PER_ROW = TPR > 32 ? TPR / 32 : 1;
    static_assert(fft_radix(NT, NPASS - 1) == E, "the last pass has the radix of a thread's samples");
};

// Pass P of the transform: radix R (fft_radix: the plan's sequence, its last
// pass radix 16) and Ns, the product of the radices of the earlier passes.
template <int NT, int P>
struct PassCfg {
    static constexpr int R = fft_radix(NT, P);
    static constexpr int NS = fft_ns(NT, P);
};

__host__ __device__ __forceinline__ int pidx(int i, int nt) { return nt >= 16 ? i + (i >> 4) : i; }

// cos(2 pi m / 16)
__host__ __device__ constexpr double cos16(int m) {
    m &= 15;
    return m == 0 ? 1.0
         : m == 1 ? 0.92387953251128675613
         : m == 2 ? 0.70710678118654752440
         : m == 3 ? 0.38268343236508977173
         : m == 4 ? 0.0
         : m == 5 ? -0.38268343236508977173
         : m == 6 ? -0.70710678118654752440
         : m == 7 ? -0.92387953251128675613
         : m == 8 ? -1.0
         : m == 9 ? -0.92387953251128675613
         : m == 10 ? -0.70710678118654752440
         : m == 11 ? -0.38268343236508977173
         : m == 12 ? 0.0
         : m == 13 ? 0.38268343236508977173
         : m == 14 ? 0.70710678118654752440
         : 0.92387953251128675613;
}

// o * exp(DIR 2 pi i m / 16); exact shortcuts for the quarter turns.
//
// FP32 constants: a float (cos, sin) pair of a codelet or twiddle angle
// carries a phase and a modulus error of up to ~6e-8.  The same constants act
// on every row at every z-step, so such errors do not average out: they add
// up coherently over the steps (field error ~5e-7 per step, energy drift
// ~1e-8 per step on a 1024 x 4096 pulse).  So every non-trivial FP32 constant
// is applied as a two-float (hi + lo) pair inside the FMAs that multiply by
// it: the pi/8 family here, 1/sqrt(2) for the pi/4 family, and the twiddles
// (tw_mul).  Together with the inverse transform being the exact adjoint of
// the forward one (inverse_fft), the constants then leave errors at the
// level of the random rounding of the arithmetic only.
__device__ __forceinline__ void c16f_pair2(int m, float *ch, float *cl, float *sh, float *sl) {
    // cos(pi/8), sin(pi/8) = hi + lo (hi the nearest float, lo the nearest
    // float to the rest; residual below 7e-16)
    constexpr float C8H = 0.9238795042037964f, C8L = 2.830748968563057e-08f;
    constexpr float S8H = 0.3826834261417389f, S8L = 6.2233507236442165e-09f;
    switch (m & 15) {
        case 1: *ch = C8H; *cl = C8L; *sh = S8H; *sl = S8L; break;
        case 3: *ch = S8H; *cl = S8L; *sh = C8H; *sl = C8L; break;
        case 5: *ch = -S8H; *cl = -S8L; *sh = C8H; *sl = C8L; break;
        case 7: *ch = -C8H; *cl = -C8L; *sh = S8H; *sl = S8L; break;
        case 9: *ch = -C8H; *cl = -C8L; *sh = -S8H; *sl = -S8L; break;
        case 11: *ch = -S8H; *cl = -S8L; *sh = -C8H; *sl = -C8L; break;
        case 13: *ch = S8H; *cl = S8L; *sh = -C8H; *sl = -C8L; break;
        default: *ch = C8H; *cl = C8L; *sh = -S8H; *sl = -S8L; break;        // 15
    }
}

template <typename V, int DIR>
__device__ __forceinline__ cx<V> rot16(cx<V> o, int m) {
    using T = typename Pack<V>::S;
    const auto K = [](T c) { return Pack<V>::splat(c); };
    m &= 15;
    if (m == 0) return o;
    if (m == 8) return mk(-o.x, -o.y);
    if (m == 4) return DIR > 0 ? mk(-o.y, o.x) : mk(o.y, -o.x);
    if (m == 12) return DIR > 0 ? mk(o.y, -o.x) : mk(-o.y, o.x);
    if constexpr (sizeof(T) == 4) {
        if ((m & 1) == 0) {
            // odd multiples of pi/4: (c, s) = (+-1, +-1)/sqrt(2)
            constexpr float H_HI = 0.70710676908493042f;       // float(1/sqrt 2)
            constexpr float H_LO = 1.2101617485882343e-8f;     // 1/sqrt 2 - H_HI
            const bool sc = m == 2 || m == 14;                 // cos > 0
            const bool ss = (DIR > 0) == (m == 2 || m == 6);   // sin > 0
            const V p = o.x + o.y, d = o.x - o.y;
            const V re = sc ? (ss ? d : p) : (ss ? -p : -d);   // +-x -+ y
            const V im = sc ? (ss ? p : -d) : (ss ? d : -p);
            return mk(vfma(re, K(H_HI), re * K(H_LO)), vfma(im, K(H_HI), im * K(H_LO)));
        }
        float ch, cl, sh, sl;
        c16f_pair2(m, &ch, &cl, &sh, &sl);
        if (DIR < 0) { sh = -sh; sl = -sl; }
        // (o.x + i o.y)(c + i s), the lo parts first
        const V lre = vfma(o.x, K(cl), -o.y * K(sl));
        const V lim = vfma(o.x, K(sl), o.y * K(cl));
        return mk(vfma(o.x, K(ch), vfma(-o.y, K(sh), lre)), vfma(o.x, K(sh), vfma(o.y, K(ch), lim)));
    } else {
        const T c = T(cos16(m));
        const T s = T(DIR) * T(cos16(m - 4));
        return mk(o.x * c - o.y * s, o.x * s + o.y * c);
    }
}

// Complex add / subtract; FP32 as one packed f32x2 instruction (each lane an
// IEEE single add, the same result as two scalar adds).
__device__ __forceinline__ cx<float> cadd2(cx<float> a, cx<float> b) {
    unsigned long long ra, rb, rc;
    asm("mov.b64 %0, {%1, %2};" : "=l"(ra) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(rb) : "f"(b.x), "f"(b.y));
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(rc) : "l"(ra), "l"(rb));
    cx<float> r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(rc));
    return r;
}
__device__ __forceinline__ cx<float> csub2(cx<float> a, cx<float> b) {
    unsigned long long ra, rb, rc;
    asm("mov.b64 %0, {%1, %2};" : "=l"(ra) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(rb) : "f"(b.x), "f"(b.y));
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(rc) : "l"(ra), "l"(rb));
    cx<float> r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(rc));
    return r;
}
__device__ __forceinline__ cx<double> cadd2(cx<double> a, cx<double> b) { return a + b; }
__device__ __forceinline__ cx<double> csub2(cx<double> a, cx<double> b) { return a - b; }
__device__ __forceinline__ cx<pk2> cadd2(cx<pk2> a, cx<pk2> b) { return a + b; }
__device__ __forceinline__ cx<pk2> csub2(cx<pk2> a, cx<pk2> b) { return a - b; }

// In-register DFT of size R (power of two <= 16), natural order in and out,
// X_k = sum_n x_n exp(DIR 2 pi i n k / R), by radix-2 decimation in time.
template <typename T, int R, int DIR>
struct Dft {
    __device__ __forceinline__ static void run(cx<T> *v) {
        cx<T> e[R / 2], o[R / 2];
#pragma unroll
        for (int k = 0; k < R / 2; ++k) { e[k] = v[2 * k]; o[k] = v[2 * k + 1]; }
        Dft<T, R / 2, DIR>::run(e);
        Dft<T, R / 2, DIR>::run(o);
#pragma unroll
        for (int k = 0; k < R / 2; ++k) {
            const int m = k * (16 / R);
            cx<T> t = rot16<T, DIR>(o[k], m);
            if ((m & 7) == 4) {
                // quarter turn: t is o with its parts swapped, which the
                // scalar adds take as operands at no cost
                v[k] = e[k] + t;
                v[k + R / 2] = e[k] - t;
            } else {
                v[k] = cadd2(e[k], t);
                v[k + R / 2] = csub2(e[k], t);
            }
        }
    }
};
// Four-point DFT in place (no multiplications).
template <int DIR, typename V>
__device__ __forceinline__ void dft4(cx<V> &a, cx<V> &b, cx<V> &c, cx<V> &d) {
    const cx<V> p = cadd2(a, c), m = csub2(a, c), q = cadd2(b, d);
    const V rx = b.x - d.x, ry = b.y - d.y;
    a = cadd2(p, q);
    c = csub2(p, q);
    // m +- DIR i (b - d)
    b = DIR > 0 ? mk(m.x - ry, m.y + rx) : mk(m.x + ry, m.y - rx);
    d = DIR > 0 ? mk(m.x + ry, m.y - rx) : mk(m.x - ry, m.y + rx);
}
// R = 16 as 4 x 4: with n = 4 n1 + n2 and k = k1 + 4 k2,
//   X_k = sum_n2 W16^(n2 k1) (sum_n1 x_n W4^(n1 k1)) W4^(n2 k2):
// 8 rotations (4 by odd multiples of pi/8, 4 of pi/4) against the 10 of the
// radix-2 recursion.
template <typename T, int DIR>
struct Dft<T, 16, DIR> {
    __device__ __forceinline__ static void run(cx<T> *v) {
#pragma unroll
        for (int n2 = 0; n2 < 4; ++n2) dft4<DIR>(v[n2], v[4 + n2], v[8 + n2], v[12 + n2]);   // v[4 k1 + n2]
#pragma unroll
        for (int k1 = 1; k1 < 4; ++k1)
#pragma unroll
            for (int n2 = 1; n2 < 4; ++n2) v[4 * k1 + n2] = rot16<T, DIR>(v[4 * k1 + n2], n2 * k1);
        cx<T> x[16];
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) {
            dft4<DIR>(v[4 * k1], v[4 * k1 + 1], v[4 * k1 + 2], v[4 * k1 + 3]);
#pragma unroll
            for (int k2 = 0; k2 < 4; ++k2) x[k1 + 4 * k2] = v[4 * k1 + k2];
        }
#pragma unroll
        for (int k = 0; k < 16; ++k) v[k] = x[k];
    }
};
template <typename T, int DIR>
struct Dft<T, 1, DIR> {
    __device__ __forceinline__ static void run(cx<T> *) {}
};

// One twiddle as loaded: FP32 tables hold each as a two-float pair, 16 bytes
// per entry (hi.x, hi.y, lo.x, lo.y); FP64 tables one complex double.
template <typename T>
struct Twiddle;
template <>
struct Twiddle<float> {
    float x, y, z, w;
};
template <>
struct Twiddle<double> {
    double x, y;
};
__device__ __forceinline__ Twiddle<float> ld_tw(const cx<float> *__restrict__ tw, int e) {
    Twiddle<float> r;
    asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w)
                 : "l"(reinterpret_cast<const float4 *>(tw) + e));
    return r;
}
__device__ __forceinline__ Twiddle<double> ld_tw(const cx<double> *__restrict__ tw, int e) {
    Twiddle<double> r;
    asm volatile("ld.global.nc.v2.f64 {%0, %1}, [%2];" : "=d"(r.x), "=d"(r.y) : "l"(tw + e));
    return r;
}

// v * W (DIR < 0) or v * conj(W) (DIR > 0).
template <typename V, int DIR>
__device__ __forceinline__ cx<V> tw_mul(cx<V> v, const Twiddle<typename Pack<V>::S> &w) {
    using T = typename Pack<V>::S;
    if constexpr (sizeof(T) == 4) {
        const auto K = [](T c) { return Pack<V>::splat(c); };
        const float hy = DIR > 0 ? -w.y : w.y;
        const float ly = DIR > 0 ? -w.w : w.w;
        const V lre = vfma(v.x, K(w.z), -v.y * K(ly));
        const V lim = vfma(v.x, K(ly), v.y * K(w.z));
        return mk(vfma(v.x, K(w.x), vfma(-v.y, K(hy), lre)), vfma(v.x, K(hy), vfma(v.y, K(w.x), lim)));
    } else {
        return cmul(v, mk(w.x, DIR > 0 ? -w.y : w.y));
    }
}

// The thread's twiddles of pass P, m = 0 .. count - 1 in the order the pass
// uses them (butterfly i, factor r).  The first kTwPre of them are loaded
// ahead, before the barrier in front of the pass, while the sample registers
// are free (the samples are in shared memory): their latency is then not
// waited for behind the operands'.
constexpr int kTwPre = 8;
template <int NT, int P>
struct PassTw {
    static constexpr int R = PassCfg<NT, P>::R;
    static constexpr int NS = PassCfg<NT, P>::NS;
    static constexpr int COUNT = NS > 1 ? RowCfg<NT>::E / R * (R - 1) : 0;
    static constexpr int PRE = COUNT < kTwPre ? COUNT : kTwPre;
    __device__ __forceinline__ static int entry(int t, int m) {
        const int i = m / (R - 1), r = m % (R - 1) + 1;
        return tw_offset(NT, P) + (r - 1) * NS + ((t + RowCfg<NT>::TPR * i) & (NS - 1));   // P > 0
    }
};
template <typename T>
struct TwAhead {
    Twiddle<T> w[kTwPre];
};
template <int NT, int P, typename T>
__device__ __forceinline__ void tw_ahead(TwAhead<T> &a, const cx<T> *__restrict__ tw, int t) {
    if constexpr (P >= 0 && P < RowCfg<NT>::NPASS) {
#pragma unroll
        for (int m = 0; m < PassTw<NT, P>::PRE; ++m)
            a.w[m] = ld_tw(tw, FCN_IDX((PassTw<NT, P>::entry(t, m)), tw_size(NT), 3));
    }
}
template <int NT, int P, typename T>
__device__ __forceinline__ Twiddle<T> tw_get(const TwAhead<T> &a, const cx<T> *__restrict__ tw, int t, int m) {
    if (m < PassTw<NT, P>::PRE) return a.w[m];
    return ld_tw(tw, FCN_IDX((PassTw<NT, P>::entry(t, m)), tw_size(NT), 3));
}

// Adjoint of Dft<T, R, -1>: the same butterflies transposed, with the
// conjugate constants (decimation in frequency).  Exact transpose in exact
// arithmetic, so that Inverse(Forward(x)) = x to first order in the errors of
// the rounded constants.
template <typename T, int R>
struct DftAdj {
    __device__ __forceinline__ static void run(cx<T> *v) {
        cx<T> e[R / 2], o[R / 2];
#pragma unroll
        for (int k = 0; k < R / 2; ++k) {
            const int m = k * (16 / R);
            const cx<T> a = v[k], b = v[k + R / 2];
            e[k] = cadd2(a, b);
            if (m == 4) {
                o[k] = mk(b.y - a.y, a.x - b.x);          // i (a - b)
            } else if (m == 12) {
                o[k] = mk(a.y - b.y, b.x - a.x);          // -i (a - b)
            } else {
                o[k] = rot16<T, +1>(csub2(a, b), m);
            }
        }
        DftAdj<T, R / 2>::run(e);
        DftAdj<T, R / 2>::run(o);
#pragma unroll
        for (int k = 0; k < R / 2; ++k) { v[2 * k] = e[k]; v[2 * k + 1] = o[k]; }
    }
};
template <typename T>
struct DftAdj<T, 16> {
    __device__ __forceinline__ static void run(cx<T> *v) {
        // the steps of Dft<T, 16, -1> transposed, in reverse order
        cx<T> x[16];
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) {
#pragma unroll
            for (int k2 = 0; k2 < 4; ++k2) x[4 * k1 + k2] = v[k1 + 4 * k2];
            dft4<+1>(x[4 * k1], x[4 * k1 + 1], x[4 * k1 + 2], x[4 * k1 + 3]);                  // x[4 k1 + n2]
        }
#pragma unroll
        for (int k1 = 1; k1 < 4; ++k1)
#pragma unroll
            for (int n2 = 1; n2 < 4; ++n2) x[4 * k1 + n2] = rot16<T, +1>(x[4 * k1 + n2], n2 * k1);
#pragma unroll
        for (int n2 = 0; n2 < 4; ++n2) {
            dft4<+1>(x[n2], x[4 + n2], x[8 + n2], x[12 + n2]);                                // x[4 n1 + n2]
#pragma unroll
            for (int n1 = 0; n1 < 4; ++n1) v[4 * n1 + n2] = x[4 * n1 + n2];
        }
    }
};
template <typename T>
struct DftAdj<T, 1> {
    __device__ __forceinline__ static void run(cx<T> *) {}
};

// Twiddle and butterfly of forward pass P for this thread's butterflies
// (operands already in v[i*R + r]).
template <typename T, int NT, int P>
__device__ __forceinline__ void pass_compute(cx<T> (&v)[RowCfg<NT>::E], int t,
                                             const cx<typename Pack<T>::S> *__restrict__ tw,
                                             const TwAhead<typename Pack<T>::S> &ahead) {
    constexpr int R = PassCfg<NT, P>::R;
    constexpr int NB = RowCfg<NT>::E / R;
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        if (PassTw<NT, P>::COUNT > 0) {
#pragma unroll
            for (int r = 1; r < R; ++r)
                v[i * R + r] = tw_mul<T, -1>(v[i * R + r], tw_get<NT, P>(ahead, tw, t, i * (R - 1) + r - 1));
        }
        Dft<T, R, -1>::run(&v[i * R]);
    }
}

// Adjoint of forward pass P: the transposed butterfly, then the conjugate
// twiddles.
template <typename T, int NT, int P>
__device__ __forceinline__ void pass_compute_adj(cx<T> (&v)[RowCfg<NT>::E], int t,
                                                 const cx<typename Pack<T>::S> *__restrict__ tw,
                                                 const TwAhead<typename Pack<T>::S> &ahead) {
    constexpr int R = PassCfg<NT, P>::R;
    constexpr int NB = RowCfg<NT>::E / R;
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        DftAdj<T, R>::run(&v[i * R]);
        if (PassTw<NT, P>::COUNT > 0) {
#pragma unroll
            for (int r = 1; r < R; ++r)
                v[i * R + r] = tw_mul<T, +1>(v[i * R + r], tw_get<NT, P>(ahead, tw, t, i * (R - 1) + r - 1));
        }
    }
}

// Butterfly i of thread t in pass P: the thread's butterflies are adjacent in
// pass 0 (its positions are then the contiguous E t .. E t + E - 1) and TPR
// apart in the others.
template <int NT, int P>
__device__ __forceinline__ int bfly(int t, int i) {
    if constexpr (P == 0) return RowCfg<NT>::E / PassCfg<NT, 0>::R * t + i;
    else return t + RowCfg<NT>::TPR * i;
}

// Makes what pass P - 1 stored visible to pass P (or the reverse, in the
// inverse transform).  In plans 0 and 2 every pass from 1 on has one butterfly of
// radix E per thread, so both passes cover a block of NS_P E positions with
// the same NS_P consecutive threads: up to 32 of them are one warp, and only
// the last exchange of rows above 512 points (Nt = 4096: passes 1 and 2)
// needs the whole CTA.  Measured on the middle launch: see RowForm.
template <int NT, int P>
__device__ __forceinline__ void pass_sync() {
    if constexpr (RowCfg<NT>::PLAN != 1 && fft_ns(NT, P) <= 32) __syncwarp();
    else __syncthreads();
}

// Operands of forward pass P (in-place decimation in time): butterfly j
// combines the positions base + r NS (r < R), base = (j / NS) NS R + j mod NS,
// and writes its outputs back to them.
template <typename T, int NT, int P>
__device__ __forceinline__ void pass_load(cx<T> (&v)[RowCfg<NT>::E], const cx<T> *S, int t) {
    using C = RowCfg<NT>;
    constexpr int R = PassCfg<NT, P>::R;
    constexpr int NS = PassCfg<NT, P>::NS;
    constexpr int NB = C::E / R;
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        const int j = bfly<NT, P>(t, i);
        const int base = (j / NS) * NS * R + (j & (NS - 1));
#pragma unroll
        for (int r = 0; r < R; ++r) v[i * R + r] = S[FCN_IDX(pidx(base + r * NS, fft_nt(NT)), C::PADN, 1)];
    }
}

template <typename T, int NT, int P>
__device__ __forceinline__ void pass_store(const cx<T> (&v)[RowCfg<NT>::E], cx<T> *S, int t) {
    using C = RowCfg<NT>;
    constexpr int R = PassCfg<NT, P>::R;
    constexpr int NS = PassCfg<NT, P>::NS;
    constexpr int NB = C::E / R;
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        const int j = bfly<NT, P>(t, i);
        const int base = (j / NS) * NS * R + (j & (NS - 1));
#pragma unroll
        for (int r = 0; r < R; ++r) S[FCN_IDX(pidx(base + r * NS, fft_nt(NT)), C::PADN, 2)] = v[i * R + r];
    }
}

// Inverse transform: the exact adjoint of the forward transform, i.e. the
// forward passes in reverse order, each applying the transposed butterfly
// and the conjugate twiddles in place (input already in registers in the
// last forward pass's order, i.e. natural frequency order; the result of the
// last pass, scaled by sc, stays in registers at the positions of forward
// pass 0, the forward transform's input order).  Every pass reads and writes
// the same positions in the same thread, so one synchronisation per pass
// (before other threads read them, pass_sync) suffices.
template <typename T, int NT, int P>
__device__ __forceinline__ void inverse_fft(cx<T> (&v)[RowCfg<NT>::E], cx<T> *S, int t,
                                            const cx<typename Pack<T>::S> *tw, TwAhead<typename Pack<T>::S> &ahead,
                                            typename Pack<T>::S sc) {
    using C = RowCfg<NT>;
    if constexpr (P >= 0) {
        if (P + 1 < C::NPASS) pass_load<T, NT, P>(v, S, t);
        pass_compute_adj<T, NT, P>(v, t, tw, ahead);
        if constexpr (P == 0) {
            // sc: the 1/Nt of the inverse transform
            const T s = Pack<T>::splat(sc);
#pragma unroll
            for (int e = 0; e < C::E; ++e) v[e] = mk(v[e].x * s, v[e].y * s);
        } else {
            pass_store<T, NT, P>(v, S, t);
            tw_ahead<NT, P - 1>(ahead, tw, t);
            pass_sync<NT, P>();
            inverse_fft<T, NT, P - 1>(v, S, t, tw, ahead, sc);
        }
    }
}

// Forward transform in place: the operands of pass 0 in registers (time
// samples in the digit-reversed order of tpos), the output of the last pass
// (natural frequency order, positions j + r NS) left in registers.
template <typename T, int NT, int P>
__device__ __forceinline__ void forward_fft(cx<T> (&v)[RowCfg<NT>::E], cx<T> *S, int t,
                                            const cx<typename Pack<T>::S> *tw,
                                            TwAhead<typename Pack<T>::S> &ahead) {
    using C = RowCfg<NT>;
    if constexpr (P < C::NPASS) {
        if constexpr (P > 0) pass_load<T, NT, P>(v, S, t);
        pass_compute<T, NT, P>(v, t, tw, ahead);
        if constexpr (P + 1 < C::NPASS) {
            pass_store<T, NT, P>(v, S, t);
            tw_ahead<NT, P + 1>(ahead, tw, t);
            pass_sync<NT, P + 1>();
        }
        forward_fft<T, NT, P + 1>(v, S, t, tw, ahead);
    }
}

// Padded shared-memory index of the e-th of the E samples a thread owns,
// whose first sits at unpadded position p0 (tpos): when the sample stride
// NSL is a multiple of 16 the padding is linear in e, so that the indices
// are one base plus compile-time offsets.
template <int NT, int NSL>
__host__ __device__ __forceinline__ int own_idx(int q0, int p0, int e) {
    if constexpr (fft_nt(NT) >= 16 && NSL % 16 == 0) return q0 + e * (NSL + NSL / 16);
    else return pidx(p0 + e * NSL, fft_nt(NT));
}

// Position in S of time sample tau.  The forward transform takes its input
// in mixed-radix digit-reversed order: the least significant digit of tau
// (radix R of the last pass) is the most significant digit of the position
// (place value NS of the last pass), and so on.  With the last pass of
// radix E, a thread's E consecutive samples tau = E t + e sit at
// tpos(E t) + e NS_last.
template <int NT>
__host__ __device__ __forceinline__ int tpos(int tau) {
    int p = 0;
#pragma unroll
    for (int s = RowCfg<NT>::NPASS - 1; s >= 0; --s) {
        p += (tau % fft_radix(NT, s)) * fft_ns(NT, s);
        tau /= fft_radix(NT, s);
    }
    return p;
}

// Time-domain rows between HBM (natural order) and S (digit-reversed
// positions, tpos).  Consecutive tau sit NS_last apart in S, which for the
// usual sizes is one bank (4096 points: 272 values apart): lanes moving
// consecutive tau would meet a 32-way bank conflict on every access of S.
// Instead, per instruction, lanes 2b and 2b+1 move the two 16-byte halves of
// one 32-byte sector of line b of a group of 16 consecutive 128-byte lines:
// whole sectors to and from HBM, and the 16 lines' values sit in different
// banks of S (their positions differ in the higher digits).  A thread moves
// its E values as E / CPC 16-byte chunks.  Needs whole warps per row and
// whole groups of 16 lines; otherwise the per-value coalesced loop is used.
template <typename T, int NT>
struct RowIo {
    static constexpr int N = fft_nt(NT);
    static constexpr int CPC = 16 / (int)sizeof(cx<T>);   // values per 16-byte chunk
    static constexpr int LW = 128 / (int)sizeof(cx<T>);   // values per 128-byte line
    static constexpr int UNITS = RowCfg<NT>::E / CPC;      // chunks per thread
    static constexpr int NSL = PassCfg<NT, RowCfg<NT>::NPASS - 1>::NS;
    static constexpr bool OK = RowCfg<NT>::E == 16 && RowCfg<NT>::TPR % 32 == 0 &&
                               (N * (int)sizeof(cx<T>)) % 2048 == 0 && UNITS % 4 == 0;
};

// The row at p can move in 16-byte chunks (complex<double> is 16-byte aligned
// by its type; a float row needs a 16-byte aligned start).
template <typename T, int NT>
__device__ __forceinline__ bool row_io_chunks(const cx<T> *p) {
    if constexpr (!RowIo<T, NT>::OK) return false;
    else return sizeof(T) == 8 || (reinterpret_cast<uintptr_t>(p) & 15) == 0;
}

// Field values bypass L1 (each is read once; the twiddle table, read by
// every row, then stays there).
__device__ __forceinline__ cx<float> ld_field(const cx<float> *p) {
    const float2 q = __ldcg(reinterpret_cast<const float2 *>(p));
    return mk(q.x, q.y);
}
__device__ __forceinline__ cx<double> ld_field(const cx<double> *p) {
    const double2 q = __ldcg(reinterpret_cast<const double2 *>(p));
    return mk(q.x, q.y);
}
template <typename T>
__device__ __forceinline__ void ld_chunk(const cx<T> *p, cx<T> *v) {
    if constexpr (sizeof(T) == 4) {
        const float4 q = __ldcg(reinterpret_cast<const float4 *>(p));
        v[0] = mk(q.x, q.y);
        v[1] = mk(q.z, q.w);
    } else {
        v[0] = ld_field(p);
    }
}

template <typename T>
__device__ __forceinline__ void st_chunk(cx<T> *p, const cx<T> *v) {
    if constexpr (sizeof(T) == 4) *reinterpret_cast<float4 *>(p) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
    else *p = v[0];
}

// Visits the thread's chunks: f(tau, q0, p0) with tau the chunk's first time
// sample and (q0, p0) the padded and unpadded S positions of tau rounded down
// to a multiple of 16 (own_idx then places tau & 15 and the next values).
template <typename T, int NT, typename F>
__host__ __device__ __forceinline__ void row_chunks(int t, F f) {
    using IO = RowIo<T, NT>;
    const int lane = t & 31, w = t >> 5;
#pragma unroll
    for (int gi = 0; gi < IO::UNITS / 4; ++gi) {
        const int line = 16 * (w * (IO::UNITS / 4) + gi) + (lane >> 1);
        const int tl = line * IO::LW;
        const int p0 = tpos<NT>(tl & ~15);
        const int q0 = pidx(p0, IO::N);
#pragma unroll
        for (int j = 0; j < 4; ++j) f(tl + (2 * j + (lane & 1)) * IO::CPC, q0, p0);
    }
}

// The same sector-wise order for a row of reals (the rho output from the u
// rows): 16-byte chunks of RC reals, 128-byte lines of 8 RC reals.  Used with
// FFT plan 0, where it cuts the wavefronts at every Nt (4096 float points:
// 2 instead of 8); with plan 1 it would not at every Nt, and the per-value
// loop stays.
template <typename T, int NT>
struct RowIoReal {
    static constexpr int N = fft_nt(NT);
    static constexpr int RC = 16 / (int)sizeof(T);        // reals per 16-byte chunk
    static constexpr int LW = 128 / (int)sizeof(T);       // reals per 128-byte line
    static constexpr int UNITS = RowCfg<NT>::E / RC;       // chunks per thread
    static constexpr bool OK = fft_plan(NT) == 0 && RowCfg<NT>::E == 16 && RowCfg<NT>::TPR % 32 == 0 &&
                               (N * (int)sizeof(T)) % 2048 == 0 && UNITS % 4 == 0;
};

template <typename T, int NT>
__device__ __forceinline__ bool row_io_real_chunks(const T *p) {
    if constexpr (!RowIoReal<T, NT>::OK) return false;
    else return (reinterpret_cast<uintptr_t>(p) & 15) == 0;
}

// Visits the thread's chunks of a real row: f(tau), tau the chunk's first
// time sample (a chunk never crosses a multiple of 16).
template <typename T, int NT, typename F>
__host__ __device__ __forceinline__ void row_real_chunks(int t, F f) {
    using IO = RowIoReal<T, NT>;
    const int lane = t & 31, w = t >> 5;
#pragma unroll
    for (int gi = 0; gi < IO::UNITS / 4; ++gi) {
        const int line = 16 * (w * (IO::UNITS / 4) + gi) + (lane >> 1);
#pragma unroll
        for (int j = 0; j < 4; ++j) f(line * IO::LW + (2 * j + (lane & 1)) * IO::RC);
    }
}

// ---------------------------------------------------------------------------
// Nonlinear half step
// ---------------------------------------------------------------------------

template <typename V>
__device__ __forceinline__ V ipow(V x, int k) {
    V r = Pack<V>::splat(typename Pack<V>::S(1));
    while (k) {
        if (k & 1) r = r * x;
        x = x * x;
        k >>= 1;
    }
    return r;
}

// x^K with K a compile-time constant when KT > 0 (squarings unrolled), the
// runtime exponent k otherwise.
template <int KT, typename V>
__device__ __forceinline__ V powk(V x, int k) {
    if constexpr (KT == 8) {
        const V x2 = x * x, x4 = x2 * x2;
        return x4 * x4;
    } else if constexpr (KT == 7) {
        const V x2 = x * x, x4 = x2 * x2;
        return x4 * x2 * x;
    } else {
        return ipow(x, k);
    }
}

template <typename T>
__device__ __forceinline__ T uplus(T a, T b) { return a + b - a * b; }

// RK4 increment of u over one dtau cell (du/dtau = w (1 - u), w = sigma_K
// I^K): with xa, xb, xm = dtau w at the cell's ends and midpoint,
// u_next = u + c (1 - u),
//   6 c = xa + 2 xm t1 + 2 xm t2 + xb t3,
//   t1 = 1 - xa/2,  t2 = 1 - (xm/2) t1,  t3 = 1 - xm t2.
// Returns 6 c (the caller folds the 1/6 into the (+) update).
template <typename V>
__device__ __forceinline__ V rk4_coef6(V xa, V xb, V xm) {
    const V one = Pack<V>::splat(typename Pack<V>::S(1)), mh = Pack<V>::splat(typename Pack<V>::S(-0.5));
    const V t1 = vfma(mh, xa, one);
    const V t2 = vfma(mh * xm, t1, one);
    const V t3 = vfma(-xm, t2, one);
    const V acc = vfma(xm + xm, t1 + t2, xa);
    return vfma(xb, t3, acc);
}

// run (+) c for c = c6 / 6: run + c (1 - run)
template <typename V>
__device__ __forceinline__ V uplus6(V run, V c6) {
    const V k = Pack<V>::splat(typename Pack<V>::S(1.0 / 6.0));
    return vfma(c6, vfma(-run, k, k), run);
}

// Exclusive (+)-scan of one value per thread and row across the TPR threads
// of a unit.  Returns the carry entering this thread.  FP64 carries between
// warps.
template <typename T, int NT>
__device__ __forceinline__ T row_scan_exclusive(T tot, int t, double *scr, int rloc) {
    using C = RowCfg<NT>;
    if (C::TPR == 1) return T(0);
    constexpr int W = C::TPR < 32 ? C::TPR : 32;
    const int lane = t & (W - 1);
    T incl = tot;
#pragma unroll
    for (int d = 1; d < W; d <<= 1) {
        T y = __shfl_up_sync(0xffffffffu, incl, d, W);
        if (lane >= d) incl = uplus(incl, y);
    }
    T excl = __shfl_up_sync(0xffffffffu, incl, 1, W);
    if (lane == 0) excl = T(0);
    if (C::WARPS_PER_ROW > 1) {
        const int w = t >> 5;
        if (lane == 31) scr[FCN_IDX(rloc * C::WARPS_PER_ROW + w, 32, 14)] = double(incl);
        __syncthreads();
        if (t < 32) {
            // FP64 exclusive scan of the warp totals of this row (<= 16)
            double x = (lane < C::WARPS_PER_ROW) ? scr[FCN_IDX(rloc * C::WARPS_PER_ROW + lane, 32, 15)] : 0.0;
            double in = x;
            // log2(warps per row) levels: the FP64 latency of this serial
            // part is paid while the row's other warps wait at the barrier
#pragma unroll
            for (int d = 1; d < C::WARPS_PER_ROW; d <<= 1) {
                double y = __shfl_up_sync(0xffffffffu, in, d, 32);
                if (lane >= d) in = in + y - in * y;
            }
            double ex = __shfl_up_sync(0xffffffffu, in, 1, 32);
            if (lane == 0) ex = 0.0;
            __syncwarp();
            if (lane < C::WARPS_PER_ROW) scr[FCN_IDX(rloc * C::WARPS_PER_ROW + lane, 32, 16)] = ex;
        }
        __syncthreads();
        // the carries are not rewritten before the caller's next barrier
        const T wc = T(scr[FCN_IDX(rloc * C::WARPS_PER_ROW + w, 32, 17)]);
        excl = uplus(wc, excl);
    }
    return excl;
}

template <typename T>
constexpr double u_idle();

// u = rho/rho_nt along tau of the unit's rows: in, U[position] = |A|^2 of
// every sample (positions of tpos, padded; complete for every thread); out,
// U[position] = u.  Each thread owns E contiguous points p = E t + e: the RK4
// coefficients of the cells (p, p+1) (the last one needs the next thread's
// first point), the thread's own exclusive (+)-scan in registers, then the
// row scan for the carry that enters it.  Ends with a barrier.  Out of line:
// few rows need it in most launches (nl_plan), and inlined it would weigh on
// the register allocation of the path that all others take.  OUT: the launch
// may write u or its maximum.  Otherwise only the plasma phase and the
// saturation read it, and without them it stays unformed (decided here: as a
// branch of the caller it cost its register allocation 1 % of a 128 x 256 FP64
// run).  Loss alone, 1024 x 4096 points that all ionise, a step: FP32 93 -> 80
// us, FP64 2320 -> 2005.
template <typename V, int NT, int KT, int MB, bool OUT>
__device__ __noinline__ void u_rows(V *U, int t, const NLCoef<typename Pack<V>::S> *cp, double *scr, int rloc) {
    if (!OUT && !(cp->flags & (PH_PLASMA | PH_MPI_SAT))) return;
    using C = RowCfg<NT>;
    using T = typename Pack<V>::S;
    constexpr int E = C::E, L = Pack<V>::L;
    constexpr int NSL = PassCfg<NT, C::NPASS - 1>::NS;
    static_assert(PassCfg<NT, C::NPASS - 1>::R == E, "a thread's samples differ in the last digit only");
    const V isr = Pack<V>::splat(cp->is_root), half = Pack<V>::splat(T(0.5));
    const int K = cp->K;
    // the thread's samples tau = E t + e sit at p0 + e NSL (tpos)
    const int p0 = tpos<NT>(E * t);
    const int q0 = pidx(p0, fft_nt(NT));
    const bool last_thread = (t == C::TPR - 1);
    // j = |A|^2 is_root: x = dtau sigma_K Ihat^K = j^K
    V jv[E + 1];
#pragma unroll
    for (int e = 0; e < E; ++e) jv[e] = U[FCN_IDX((own_idx<NT, NSL>(q0, p0, e)), C::PADN, 8)] * isr;
    jv[E] = last_thread ? Pack<V>::splat(T(0)) : U[FCN_IDX(pidx(tpos<NT>(E * (t + 1)), fft_nt(NT)), C::PADN, 8)] * isr;
    // the thread's exclusive local prefixes of the (+)-scan; u at point e is
    // carry (+) lp[e] once the carry is known
    V lp[E];
#pragma unroll
    for (int e = 0; e < E; ++e) lp[e] = Pack<V>::splat(T(0));
    V run = Pack<V>::splat(T(0));
    T jmax = T(0);
#pragma unroll
    for (int e = 0; e <= E; ++e) {
        if constexpr (L == 2) jmax = fmaxf(jmax, fmaxf(jv[e].a, jv[e].b));
        else jmax = fmax(jmax, jv[e]);
    }
    // Where every j^K of the thread's cells underflows to zero (the pulse's
    // wings), every RK4 increment is exactly zero and u keeps its entering
    // value: the arithmetic below would give the same bits.
    if (!(KT == 8 && jmax < T(u_idle<T>()))) {
        V ja = jv[0];
        V xa = powk<KT>(ja, K);
#pragma unroll
        for (int e = 0; e < E; ++e) {
            lp[e] = run;
            if ((e + 1 < E) || !last_thread) {
                const V jb = jv[e + 1];
                const V xb = powk<KT>(jb, K);
                const V xm = powk<KT>(half * (ja + jb), K);
                run = uplus6(run, rk4_coef6(xa, xb, xm));
                ja = jb;
                xa = xb;
            }
        }
    }
    V carry;
    if constexpr (L == 2) {
        carry.a = row_scan_exclusive<T, NT>(run.a, t, scr, rloc);
        if (C::WARPS_PER_ROW > 1) __syncthreads();          // the scratch is reused
        carry.b = row_scan_exclusive<T, NT>(run.b, t, scr, rloc);
    } else {
        carry = row_scan_exclusive<T, NT>(run, t, scr, rloc);
    }
    const V omc = Pack<V>::splat(T(1)) - carry;
    __syncthreads();                                        // every thread has read its neighbour's |A|^2
#pragma unroll
    for (int e = 0; e < E; ++e) U[FCN_IDX((own_idx<NT, NSL>(q0, p0, e)), C::PADN, 28)] = vfma(lp[e], omc, carry);
    __syncthreads();
}

// j below which j^8 rounds to zero (j^8 < half the smallest denormal: 2.4e-6
// in FP32, 4e-41 in FP64).
template <typename T>
constexpr double u_idle() { return sizeof(T) == 4 ? 2e-6 : 1e-41; }

// ---- the nonlinear step of rows that ionise too little to matter ----
// Where, over a whole row, the plasma phase and the loss exponent stay below
// a small part of the rounding of the field (nl_plan: 2^-32 in FP32, 2^-61 in
// FP64, against the 2^-25 and 2^-54 that rounding A itself can turn it by),
// the half step is the Kerr rotation alone,
//   A <- A exp(i h sum_j kerr_j |A|^(2 j + 2)),
// pointwise: no scan along tau, so the samples can stay in the registers
// they leave the inverse transform in and enter the forward one from.  That
// takes 6 of 11 block barriers and 3 shared-memory round trips per point out
// of the middle launch.  The two half steps of a middle launch stay two
// rotations with their own roundings: a run continued from its saved field
// (closing, then opening half step) has the same bits as one that was not
// interrupted.
// Only the rows through a filament's core ionise more (|A|^2 above ~2e16
// W/m^2 for 2 mm steps); they take u_rows and nl_full.
//
// u at the end of the row is at most Nt max(c) with c <= max j^K (the RK4
// increment's weights add up to 1 and every factor is in [0, 1]).
// Returns -1: full half step; 0: nothing to do; 1..4: range of the phase
// (nl_kerr): below 1/16 (FP32) or 2^-12 (FP64), 1/64 (FP64 only), 0.78 (no
// reduction needed), 1e4.  Monotone in cmax.
template <typename T, int NT, int KT>
__device__ __forceinline__ int nl_plan(float cmax, const NLCoef<T> &c) {
    constexpr float kNeg = sizeof(T) == 4 ? 2.3283064e-10f : 4.3368087e-19f;       // 2^-32, 2^-61
    constexpr float kSkip = sizeof(T) == 4 ? 7.450580596923828e-9f : 6.9388939e-18f;  // 2^-27, 2^-57
    constexpr float kSmall = sizeof(T) == 4 ? 0.0625f : 2.44140625e-4f;
    constexpr float kMid = sizeof(T) == 4 ? 0.0f : 0.015625f;
    const float ihm = cmax * float(c.inv_is);
    const float pk = fabsf(float(c.hk[0])) +
                     ihm * (fabsf(float(c.hk[1])) + ihm * (fabsf(float(c.hk[2])) + ihm * fabsf(float(c.hk[3]))));
    const float phib = ihm * pk;
    const float ub = float(fft_nt(NT)) * powk<KT>(cmax * float(c.is_root), c.K);
    const float plb = fabsf(float(c.hplasma)) * ub;
    const float lnb = fabsf(float(c.hloss)) * powk<(KT > 0 ? KT - 1 : 0)>(ihm, c.K - 1);
    if (plb < kNeg && lnb < kNeg && phib < 1.0e4f)
        return phib < kSkip ? 0 : phib < kSmall ? 1 : phib < kMid ? 2 : phib < 0.78f ? 3 : 4;
    return -1;                                     // also for NaN or infinite bounds
}

// Largest part of the thread's values in modulus, as ordered unsigned bits
// (float: its bits; double: its high word; NaN above infinity).  The largest
// |A|^2 lies between its square and twice that.
template <typename V, int E>
__device__ __forceinline__ unsigned thread_max(const cx<V> (&v)[E]) {
    if constexpr (sizeof(typename Pack<V>::S) == 8) {
        unsigned m = 0;
#pragma unroll
        for (int e = 0; e < E; ++e)
            m = max(m, max((unsigned)__double2hiint(v[e].x) & 0x7fffffffu, (unsigned)__double2hiint(v[e].y) & 0x7fffffffu));
        return m;
    } else {
        float m = 0.f;
        auto acc = [&](float x, float y) {
            asm("max.NaN.f32 %0, %0, %1;" : "+f"(m) : "f"(fabsf(x)));
            asm("max.NaN.f32 %0, %0, %1;" : "+f"(m) : "f"(fabsf(y)));
        };
#pragma unroll
        for (int e = 0; e < E; ++e) {
            if constexpr (Pack<V>::L == 2) {
                acc(v[e].x.a, v[e].y.a);
                acc(v[e].x.b, v[e].y.b);
            } else {
                acc(v[e].x, v[e].y);
            }
        }
        return __float_as_uint(m);
    }
}

// Bound of |A|^2 over the CTA's rows from the threads' thread_max, rounded
// up to float, in every thread (NaN or an overflow reads as NaN or infinity).
// One block barrier; two calls in a row take different halves of the scratch
// (slot 0, 1).
template <int TH, typename T>
__device__ __forceinline__ float cta_bound(unsigned m, double *scr, int slot) {
    unsigned *ws = reinterpret_cast<unsigned *>(scr) + 16 * slot;
    m = __reduce_max_sync(0xffffffffu, m);
    if constexpr (TH > 32) {
        if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = m;
        __syncthreads();
        m = __reduce_max_sync(0xffffffffu, ws[threadIdx.x & (TH / 32 - 1)]);
    }
    float f;
    // (the largest high word is a NaN's, and adding 1 would make it a zero)
    if constexpr (sizeof(T) == 8) f = m < 0x7ff00000u ? __double2float_ru(__hiloint2double((int)(m + 1), 0)) : INFINITY;
    else f = __uint_as_float(m);
    return f * f * 2.00001f;
}

// sin(phi) = phi (1 + phi^2 ps) and cos(phi) - 1 = phi^2 pc for |phi| below
// the tier's bound (nl_plan): Taylor polynomials, the terms left out below
// 2^-33 (FP32) and 2^-58 (FP64), but for the FP32 sine, which stops at phi^9
// also near pi/4 (tiers 3 and 4): there it is 2^-29 too large.  The roundings
// of its coefficients and steps leave it as much too small: rows turned by
// 0.70 to 0.785 lose 0.8e-10 to 1.2e-10 of |A|^2 per half step (2000 of them,
// measured), and 2.6e-10 with the phi^11 term.
template <int TIER, typename V>
__device__ __forceinline__ void expi_poly(V p2, V *ps_out, V *pc_out) {
    using T = typename Pack<V>::S;
    const auto K = [](double c) { return Pack<V>::splat(T(c)); };
    V ps, pc;
    if constexpr (TIER == 1) {
        ps = vfma(p2, K(8.33333333333333333333e-3), K(-1.66666666666666666667e-1));
        pc = vfma(p2, K(4.16666666666666666667e-2), K(-0.5));
    } else {
        if constexpr (sizeof(T) == 4 || TIER == 2) {
            ps = vfma(p2, K(2.75573192239858906526e-6), K(-1.98412698412698412698e-4));
            pc = vfma(p2, K(-2.75573192239858906526e-7), K(2.48015873015873015873e-5));
        } else {
            ps = vfma(p2, K(2.81145725434552076320e-15), K(-7.64716373181981647590e-13));
            ps = vfma(p2, ps, K(1.60590438368216145994e-10));
            ps = vfma(p2, ps, K(-2.50521083854417187751e-8));
            ps = vfma(p2, ps, K(2.75573192239858906526e-6));
            ps = vfma(p2, ps, K(-1.98412698412698412698e-4));
            pc = vfma(p2, K(4.77947733238738529743e-14), K(-1.14707455977297247139e-11));
            pc = vfma(p2, pc, K(2.08767569878680989792e-9));
            pc = vfma(p2, pc, K(-2.75573192239858906526e-7));
            pc = vfma(p2, pc, K(2.48015873015873015873e-5));
        }
        ps = vfma(p2, ps, K(8.33333333333333333333e-3));
        ps = vfma(p2, ps, K(-1.66666666666666666667e-1));
        pc = vfma(p2, pc, K(-1.38888888888888888889e-3));
        pc = vfma(p2, pc, K(4.16666666666666666667e-2));
        pc = vfma(p2, pc, K(-0.5));
    }
    *ps_out = ps;
    *pc_out = pc;
}

// Quadrant n of the reduced angle: (sin r, cos r - 1) -> (sin x, cos x - 1)
// for x = n pi/2 + r (cos - 1 kept without adding 1 where n = 0).
template <typename T>
__device__ __forceinline__ void expi_quadrant(int n, T &s, T &cm1) {
    const T sr = s, cr = cm1 + T(1);
    const T s1 = (n & 1) ? cr : sr, c1 = (n & 1) ? sr : cr;
    s = (n & 2) ? -s1 : s1;
    const T c = ((n + 1) & 2) ? -c1 : c1;
    if (n & 3) cm1 = c - T(1);
}

// sin(phi) and cos(phi) - 1 for |phi| < 1e4: Cody & Waite's reduction
// phi = n pi/2 + r with pi/2 as two words (n PIO2_HI exact inside the FMA),
// then the polynomials for |r| < pi/4.
template <typename V>
__device__ __forceinline__ void expi_m1_reduced(V phi, V *s, V *cm1) {
    using T = typename Pack<V>::S;
    constexpr T HI = sizeof(T) == 4 ? T(1.57079637050628662109) : T(1.57079632679489655800);
    constexpr T LO = sizeof(T) == 4 ? T(-4.37113900018624283e-8) : T(6.12323399573676603587e-17);
    if constexpr (Pack<V>::L == 2) {
        const pk2 n = {rintf(phi.a * 0.636619772367581343076f), rintf(phi.b * 0.636619772367581343076f)};
        V r = vfma(-n, Pack<V>::splat(HI), phi);
        r = vfma(-n, Pack<V>::splat(LO), r);
        const V r2 = r * r;
        V ps, pc;
        expi_poly<3, V>(r2, &ps, &pc);
        *s = vfma(r * r2, ps, r);
        *cm1 = r2 * pc;
        expi_quadrant<float>(int(n.a), s->a, cm1->a);
        expi_quadrant<float>(int(n.b), s->b, cm1->b);
    } else {
        const T n = rint(phi * T(0.636619772367581343076));
        V r = vfma(-n, HI, phi);
        r = vfma(-n, LO, r);
        const V r2 = r * r;
        V ps, pc;
        expi_poly<3, V>(r2, &ps, &pc);
        *s = vfma(r * r2, ps, r);
        *cm1 = r2 * pc;
        expi_quadrant<T>(int(n), *s, *cm1);
    }
}

// A <- A exp(i phi) for the thread's values, in delta form (A +
// A (exp(i phi) - 1), one rounding per component; see nl_full).  Below pi/4
// the common factor phi of sin and cos - 1 enters last:
//   A + phi (A (phi pc + i (1 + phi^2 ps))).
// With Kerr orders n2 and n4 alone (NLCoef::kerr2) phi comes from |A|^2 with
// the intensity scale (a power of two) in the coefficients.
template <int TIER, bool KERR2, typename V, int E, typename T = typename Pack<V>::S>
__device__ __forceinline__ void nl_kerr_tier(cx<V> (&v)[E], const NLCoef<T> &c) {
    const auto K = [](T x) { return Pack<V>::splat(x); };
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const cx<V> a = v[e];
        const V i2 = vfma(a.x, a.x, a.y * a.y);
        V phi;
        if constexpr (KERR2) {
            phi = i2 * vfma(i2, K(c.kf[1]), K(c.kf[0]));
        } else {
            const V ih = i2 * K(c.inv_is);
            V p = vfma(ih, K(c.hk[3]), K(c.hk[2]));
            p = vfma(ih, p, K(c.hk[1]));
            phi = ih * vfma(ih, p, K(c.hk[0]));
        }
        if constexpr (TIER == 4) {
            V s, cm1;
            expi_m1_reduced<V>(phi, &s, &cm1);
            const V dx = vfma(a.x, cm1, -(a.y * s));
            const V dy = vfma(a.y, cm1, a.x * s);
            v[e] = mk(a.x + dx, a.y + dy);
        } else {
            const V p2 = phi * phi;
            V ps, pc;
            expi_poly<TIER, V>(p2, &ps, &pc);
            const V s1 = vfma(p2, ps, K(T(1))), c1 = phi * pc;
            const V tx = vfma(a.x, c1, -(a.y * s1));
            const V ty = vfma(a.y, c1, a.x * s1);
            v[e] = mk(vfma(phi, tx, a.x), vfma(phi, ty, a.y));
        }
    }
}
template <typename V, int E, typename T = typename Pack<V>::S>
__device__ __forceinline__ void nl_kerr(cx<V> (&v)[E], const NLCoef<T> &c, int tier) {
    if (tier <= 0) return;
    if (!c.kerr2) return nl_kerr_tier<4, false, V, E>(v, c);      // n6, n8 terms: one form for every phase
    if (tier == 1) nl_kerr_tier<1, true, V, E>(v, c);
    else if (sizeof(T) == 8 && tier == 2) nl_kerr_tier<2, true, V, E>(v, c);
    else if (tier == 3) nl_kerr_tier<3, true, V, E>(v, c);
    else nl_kerr_tier<4, true, V, E>(v, c);
}

// exp(x) - 1: the loss exponent is tiny except near the peak, where the
// series is exact to rounding (FP32: x^3/6 < 2e-13; FP64: x^6/720 < 2e-27).
__device__ __forceinline__ float expm1_of(float x) {
    if (fabsf(x) < 1.0e-4f) return fmaf(0.5f * x, x, x);
    return expm1f(x);
}
__device__ __forceinline__ double expm1_of(double x) {
    if (fabs(x) < 1.0e-4) {
        double p = fma(x, 1.0 / 120.0, 1.0 / 24.0);
        p = fma(x, p, 1.0 / 6.0);
        p = fma(x, p, 0.5);
        return fma(x * x, p, x);
    }
    return expm1(x);
}
__device__ __forceinline__ pk2 expm1_of(pk2 x) { return {expm1_of(x.a), expm1_of(x.b)}; }
// sin and cos - 1 of any finite phase: the reduction of tier 3 where it
// holds, the library beyond.
template <typename V>
__device__ __forceinline__ void expi_any(V phi, V *s, V *cm1) {
    using T = typename Pack<V>::S;
    expi_m1_reduced<V>(phi, s, cm1);
    auto far = [](T x, T *sn, T *cm) {
        if (!(fabs(x) < T(1.0e4))) {
            T c;
            if constexpr (sizeof(T) == 4) sincosf(x, sn, &c);
            else sincos(x, sn, &c);
            *cm = c - T(1);
        }
    };
    if constexpr (Pack<V>::L == 2) {
        far(phi.a, &s->a, &cm1->a);
        far(phi.b, &s->b, &cm1->b);
    } else {
        far(phi, s, cm1);
    }
}

// The full half step A <- A exp(h N(|A|^2, u)) of one value, with h and the
// physics switches folded into the coefficients:
//   phi = Ihat (hk0 + Ihat (hk1 + Ihat (hk2 + Ihat hk3))) - hplasma u,
//   lnamp = -hloss Ihat^(K-1) (1 - sat u),  A <- A exp(lnamp + i phi),
// in delta form: A D with D = amp exp(i phi) - 1 = (em1 + cm1 + em1 cm1) +
// i s (1 + em1), em1 = amp - 1, formed first and added to A with one rounding
// per component.  (A float cosine that rounds to 1 for small phases gives
// |(cos, sin)|^2 = 1 + phi^2 > 1, a systematic energy gain in the pulse's
// weak tails; and folding the terms into A one FMA at a time rounds A plus
// the first-order part before the second-order part is added, which raised
// |A| by ~1e-8 of the energy per step on a Kerr-phase pulse.)
template <int KT, typename V, typename T = typename Pack<V>::S>
__device__ __forceinline__ cx<V> nl_full(cx<V> a, V u, const NLCoef<T> &c) {
    const auto K = [](T x) { return Pack<V>::splat(x); };
    const V ih = vfma(a.x, a.x, a.y * a.y) * K(c.inv_is);
    V p = vfma(ih, K(c.hk[3]), K(c.hk[2]));
    p = vfma(ih, p, K(c.hk[1]));
    p = vfma(ih, p, K(c.hk[0]));
    const V phi = vfma(K(-c.hplasma), u, ih * p);
    const V lna = -(K(c.hloss) * vfma(K(-c.sat), u, K(T(1)))) * powk<(KT > 0 ? KT - 1 : 0)>(ih, c.K - 1);
    V s, cm1;
    expi_any<V>(phi, &s, &cm1);
    const V em1 = expm1_of(lna);
    const V dre = vfma(em1, cm1, em1 + cm1);
    const V dim = vfma(s, em1, s);
    const V dx = vfma(a.x, dre, -(a.y * dim));
    const V dy = vfma(a.y, dre, a.x * dim);
    return mk(a.x + dx, a.y + dy);
}

// Totals over the TPR threads of each row of a CTA of TH threads: sums of
// s[k] in FP64, sums (k < NA) or maxima of m[k] in T.  Every thread leaves its
// partials in shared memory (smem: free for all, no barrier needed before);
// G of them each go to one lane, the lanes of a row combine theirs by
// shuffles, and the row's first lane calls out(unit of the CTA, s, m).  No
// barrier after: the caller has one before smem is written again.
//
// FP64 units bound it: a warp's FP64 instruction holds one of an SM's four
// schedulers' FP64 lanes for 64 cycles, so a tree of shuffles in every warp
// (5 levels x 4 FP64 values, of which most lanes are idle work) took as long
// as the row's transform.  Here one warp adds for 256 threads, 13 FP64
// additions deep, and maxima and counts are in T.  Last stage with rho and
// statistics, 8 x 1024 rows of 4096 points, FP32: 303 -> 209-215 us; with the
// step-doubling sums 336-353 -> 264-285 us.
constexpr int row_red_group(int tpr) { return tpr >= 256 ? tpr / 32 : tpr >= 8 ? 8 : tpr; }
template <typename T, int NT, int TH, int NS, int NA, int NX, typename F>
__device__ __forceinline__ void row_totals(const double (&s)[NS], const T (&m)[NA + NX + 1], unsigned char *smem,
                                           F out) {
    using C = RowCfg<NT>;
    if constexpr (C::TPR == 1) return out((int)threadIdx.x, s, m);
    constexpr int G = row_red_group(C::TPR), LPR = C::TPR / G, NM = NA + NX;
    constexpr int STRIDE = G > 1 ? TH + TH / G : TH;          // padded: conflict-free for writers and readers
    static_assert(C::TPR == 1 || STRIDE * (NS * 8 + NM * (int)sizeof(T)) <= TH * C::PADN / C::TPR * 2 * (int)sizeof(T), "row storage");
    static_assert(LPR <= 32, "a row's lanes are in one warp");
    double *P = reinterpret_cast<double *>(smem);
    T *Q = reinterpret_cast<T *>(P + NS * STRIDE);
    const int tid = threadIdx.x;
    const int pos = G > 1 ? tid + tid / G : tid;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NS; ++k) P[FCN_IDX(k * STRIDE + pos, NS * STRIDE, 18)] = s[k];
#pragma unroll
    for (int k = 0; k < NM; ++k) Q[FCN_IDX(k * STRIDE + pos, NM * STRIDE, 19)] = m[k];
    __syncthreads();
    if ((tid & ~31) >= TH / G) return;
    const bool on = tid < TH / G;
    const int p0 = on ? (G > 1 ? tid * (G + 1) : tid) : 0;
    double x[NS];
    T y[NM + 1];
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        x[k] = P[FCN_IDX(k * STRIDE + p0, NS * STRIDE, 20)];
#pragma unroll
        for (int g = 1; g < G; ++g) x[k] += P[FCN_IDX(k * STRIDE + p0 + g, NS * STRIDE, 20)];
    }
#pragma unroll
    for (int k = 0; k < NM; ++k) {
        y[k] = Q[FCN_IDX(k * STRIDE + p0, NM * STRIDE, 21)];
#pragma unroll
        for (int g = 1; g < G; ++g) {
            const T o = Q[FCN_IDX(k * STRIDE + p0 + g, NM * STRIDE, 21)];
            y[k] = k < NA ? y[k] + o : fmax(y[k], o);
        }
    }
#pragma unroll
    for (int d = LPR / 2; d >= 1; d >>= 1) {
#pragma unroll
        for (int k = 0; k < NS; ++k) x[k] += __shfl_down_sync(0xffffffffu, x[k], d, LPR);
#pragma unroll
        for (int k = 0; k < NM; ++k) {
            const T o = __shfl_down_sync(0xffffffffu, y[k], d, LPR);
            y[k] = k < NA ? y[k] + o : fmax(y[k], o);
        }
    }
    if (on && (tid & (LPR - 1)) == 0) out(tid / LPR, x, y);
}

// Compensated (Kahan) FP32 running sum: the per-thread partials of the FP32
// path keep float relative accuracy whatever the count; rows and the final
// reductions are FP64.
struct KahanF {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float v) {
        const float y = v - c;
        const float t2 = s + y;
        c = (t2 - s) - y;
        s = t2;
    }
    __device__ __forceinline__ double sum() const { return double(s) - double(c); }
};
template <typename T>
struct PlainSum {
    T s = T(0);
    __device__ __forceinline__ void add(T v) { s += v; }
    __device__ __forceinline__ double sum() const { return double(s); }
};

// MB: minimum resident CTAs per SM requested from the compiler (register cap
// 64K / (MB TH)).  One CTA of TH threads processes the rows of TH/TPR units
// from row_base on, of one pulse; TH and MB by form (RowForm), in the work-list
// kernel by the list's largest Nt.  Every thread of the CTA must call it
// (barriers inside).
enum : int { ROW_PLAIN = 0, ROW_OUT = 1, ROW_DIFF = 2 };
// The mode that launches with these operations take.
__host__ __device__ constexpr int row_mode(int ops) {
    return (ops & OP_DIFF) ? ROW_DIFF : (ops & (OP_RHO | OP_STATS | OP_SPEC)) ? ROW_OUT : ROW_PLAIN;
}
// Whether a mode's u rows have a place of their own behind the scratch
// (otherwise the storage of S).  The kernel's layout and the shared memory of
// its launches both follow from this.
__host__ __device__ constexpr bool row_keeps_u(int mode) { return mode != ROW_PLAIN; }
// The buffers of one pulse (RowArgs names them).
template <typename T>
struct RowBufs {
    cx<T> *field;
    T *rho;
    double *stats;
    const cx<T> *in, *cmp;
    double *diff;
};

// One row stage of TH / TPR units of rows (a unit: one row, or the two
// adjacent rows of a pair); row_base: the first unit's first row.
//
// MODE: what the kernel is compiled for -- ROW_PLAIN: neither rho nor
// statistics (the launches of almost every z-step), ROW_OUT: also those,
// ROW_DIFF: also the step-doubling norm's sums (OP_DIFF).  The code of the
// outputs then does not weigh on the register allocation of the others.
template <typename V, int NT, int KT, int TH, int MB, int MODE>
__device__ __forceinline__ void row_body(const RowArgs<typename Pack<V>::S> &a,
                                         const RowBufs<typename Pack<V>::S> &bf, int row_base, int ops,
                                         unsigned char *smem_raw) {
    using T = typename Pack<V>::S;
    constexpr bool DIFFK = MODE == ROW_DIFF;
    using C = RowCfg<NT>;
    constexpr int E = C::E;
    constexpr int L = Pack<V>::L;
    constexpr int RPC = TH / C::TPR;
    constexpr int PL = C::NPASS - 1;
    constexpr int RL = PassCfg<NT, PL>::R;
    constexpr int NSL = PassCfg<NT, PL>::NS;
    static_assert(RPC * C::TPR == TH, "CTA size must hold whole rows");
    // shared memory: the rows S, the FP64 scratch, then the u rows U of the
    // modes that keep them (row_keeps_u)
    cx<V> *S_all = reinterpret_cast<cx<V> *>(smem_raw);
    double *scr = reinterpret_cast<double *>(S_all + RPC * C::PADN);
    // u rows: behind the scratch where an output may need them, else in the
    // storage of S (the samples are then in registers)
    V *U_all = row_keeps_u(MODE) ? reinterpret_cast<V *>(scr + kRowScratch) : reinterpret_cast<V *>(smem_raw);

#ifdef FCN_CHECKED
    {
        unsigned dsm;
        asm volatile("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dsm));
        if (threadIdx.x == 0)
            FCN_IDX((sizeof(cx<T>) + (row_keeps_u(MODE) ? sizeof(T) : 0)) * L * RPC * C::PADN +
                        sizeof(double) * kRowScratch - 1,
                    dsm, 25);
    }
#endif
    const int tid = threadIdx.x;
    const int rloc = tid / C::TPR;
    const int t = tid - rloc * C::TPR;
    const int row = row_base + rloc * L;             // the unit's first row
    const bool valid = row < a.nr;
    // rows of the unit that exist (a pair's second row is missing at the end
    // of an odd Nr: it then computes on a copy of the first and stores nothing)
    const int nrow = min(L, a.nr - row);
    cx<V> *S = S_all + rloc * C::PADN;
    V *U = U_all + rloc * C::PADN;
    cx<T> *g[L];
    const cx<T> *src[L];                             // the rows' input: the field itself, or a separate source
#pragma unroll
    for (int k = 0; k < L; ++k) {
        const size_t r = valid ? row + (k < nrow ? k : 0) : 0;
        g[k] = bf.field + r * C::N;
        src[k] = bf.in ? bf.in + r * C::N : g[k];
    }

    cx<V> v[E];
    bool in_regs = false;                            // v holds the time samples at the positions of pass 0
    if (ops & OP_IFFT) {
        // the inverse's first pass (the adjoint of the last forward pass) takes
        // its operands straight from HBM: X[j + r*NS], j = t + TPR*i, coalesced
#pragma unroll
        for (int i = 0; i < E / RL; ++i) {
            const int j = t + C::TPR * i;
#pragma unroll
            for (int r = 0; r < RL; ++r) {
                cx<T> x[L];
#pragma unroll
                for (int k = 0; k < L; ++k)
                    x[k] = valid ? ld_field(&src[k][FCN_IDX(j + r * NSL, fft_nt(NT), 4)]) : mk(T(0), T(0));
                v[i * RL + r] = pack_rows<V>(x);
            }
        }
        TwAhead<T> ahead;
        tw_ahead<NT, PL>(ahead, C::PLAN == 2 ? a.tw2 : C::PLAN ? a.tw1 : a.tw, t);
        inverse_fft<V, NT, PL>(v, S, t, C::PLAN == 2 ? a.tw2 : C::PLAN ? a.tw1 : a.tw, ahead, a.nl.inv_nt);
        in_regs = true;
    } else {
        bool chunks = true;
#pragma unroll
        for (int k = 0; k < L; ++k) chunks = chunks && row_io_chunks<T, NT>(src[k]);
        if (chunks) {
            using IO = RowIo<T, NT>;
            row_chunks<T, NT>(t, [&](int tau, int cq0, int cp0) {
                cx<T> cv[L][IO::CPC];
#pragma unroll
                for (int k = 0; k < L; ++k) {
                    if (valid) {
                        ld_chunk<T>(src[k] + FCN_IDX(tau, IO::N - IO::CPC + 1, 6), cv[k]);
                    } else {
#pragma unroll
                        for (int m = 0; m < IO::CPC; ++m) cv[k][m] = mk(T(0), T(0));
                    }
                }
#pragma unroll
                for (int m = 0; m < IO::CPC; ++m) {
                    cx<T> x[L];
#pragma unroll
                    for (int k = 0; k < L; ++k) x[k] = cv[k][m];
                    S[FCN_IDX((own_idx<NT, IO::NSL>(cq0, cp0, (tau & 15) + m)), C::PADN, 5)] = pack_rows<V>(x);
                }
            });
        } else {
#pragma unroll
            for (int i = 0; i < E; ++i) {
                const int idx = t + C::TPR * i;
                cx<T> x[L];
#pragma unroll
                for (int k = 0; k < L; ++k) x[k] = valid ? ld_field(&src[k][FCN_IDX(idx, fft_nt(NT), 6)]) : mk(T(0), T(0));
                S[FCN_IDX(pidx(tpos<NT>(idx), fft_nt(NT)), C::PADN, 5)] = pack_rows<V>(x);
            }
        }
        __syncthreads();
    }
    // the samples to shared memory (complete for every thread), where the
    // row is needed along tau
    auto to_smem = [&] {
        if (in_regs) {
            pass_store<V, NT, 0>(v, S, t);
            __syncthreads();
            in_regs = false;
        }
    };

    const bool keep_u = MODE != ROW_PLAIN && (ops & (OP_RHO | OP_STATS)) != 0;
    const bool need_u = (a.nl.flags & (PH_PLASMA | PH_MPI_SAT)) || keep_u;
    const int nhalf = ((ops & OP_NL) ? 1 : 0) + ((ops & OP_NL2) ? 1 : 0);
    int plan = -1;
    bool known = false;
#pragma unroll 1
    for (int hs = 0; hs < nhalf; ++hs) {
        if (!in_regs) {
            pass_load<V, NT, 0>(v, S, t);
            in_regs = true;
        }
        float m = 0.f;
        if (!known) {
            m = cta_bound<TH, T>(thread_max<V, E>(v), scr, hs);
            plan = nl_plan<T, NT, KT>(m, a.nl);
            // a rotation leaves |A| to a rounding or two, and so the bound
            // within a factor of 2: unless a tier ends in that range, the
            // second half step's plan is the same
            known = !keep_u && plan >= 0 && plan == nl_plan<T, NT, KT>(m * 0.499f, a.nl) &&
                    plan == nl_plan<T, NT, KT>(m * 2.002f, a.nl);
        }
        const bool out_u = MODE != ROW_PLAIN && keep_u && hs + 1 == nhalf;
        if (plan < 0 || out_u) {
            // u of every sample into U: through the scan along tau, unless
            // every increment of the CTA's rows is exactly zero
            const bool idle = KT == 8 && m * float(a.nl.is_root) < float(u_idle<T>()) && sizeof(T) == 4;
            auto at = [&](int e) { return FCN_IDX(pidx(E * t + e, fft_nt(NT)), C::PADN, 7); };   // pass 0's positions
            if (!row_keeps_u(MODE)) __syncthreads();      // U is the storage of S here
#pragma unroll
            for (int e = 0; e < E; ++e)
                U[at(e)] = idle ? Pack<V>::splat(T(0)) : vfma(v[e].x, v[e].x, v[e].y * v[e].y);
            __syncthreads();
            if (!idle) u_rows<V, NT, KT, MB, MODE != ROW_PLAIN>(U, t, &a.nl, scr, rloc);
            if (plan < 0) {
                const bool with_u = need_u;
#pragma unroll
                for (int e = 0; e < E; ++e)
                    v[e] = nl_full<KT, V>(v[e], with_u ? U[at(e)] : Pack<V>::splat(T(0)), a.nl);
            }
            if (!row_keeps_u(MODE)) __syncthreads();
        }
        nl_kerr<V, E>(v, a.nl, plan);
    }
    const bool have_u = nhalf > 0;
    if (keep_u) {
        if (!in_regs) {
            pass_load<V, NT, 0>(v, S, t);
            in_regs = true;
        }
        // statistics of the final rows; rho is written below, coalesced
        if ((ops & OP_STATS) && bf.stats) {
            // sum |A|^2; count of non-finite |A|^2, max |A|^2, max u
            double sum[L];
            T m[3 * L + 1];
#pragma unroll
            for (int k = 0; k < L; ++k) {
                std::conditional_t<sizeof(T) == 4, KahanF, PlainSum<T>> ks;
                T mx = T(0), mu = T(0), bad = T(0);
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const cx<T> x = row_of<V>(v[e], k);
                    const T i2 = vfma(x.x, x.x, x.y * x.y);
                    if (!isfinite(i2)) bad += T(1);
                    ks.add(i2);
                    mx = fmax(mx, i2);
                    if (have_u) {
                        const V u = U[FCN_IDX(pidx(E * t + e, fft_nt(NT)), C::PADN, 7)];
                        mu = fmax(mu, row_of<V>(mk(u, u), k).x);
                    }
                }
                sum[k] = ks.sum();
                m[k] = bad;
                m[L + 2 * k] = mx;
                m[L + 2 * k + 1] = mu;
            }
            row_totals<T, NT, TH, L, L, 2 * L>(sum, m, smem_raw, [&](int unit, const double *x, const T *y) {
#pragma unroll
                for (int k = 0; k < L; ++k) {
                    const int r = row_base + unit * L + k;
                    if (r >= a.nr) break;
                    double *st = bf.stats + FCN_IDX((size_t)r * NSTAT, (size_t)a.nr * NSTAT, 23);
                    st[ST_SUM_I] = x[k];
                    st[ST_MAX_I] = double(y[L + 2 * k]);
                    if (ops & (OP_NL | OP_NL2)) st[ST_MAX_U] = double(y[L + 2 * k + 1]);
                    st[ST_NONFINITE] = double(y[k]);
                }
            });
        }
        if ((ops & OP_RHO) && valid && bf.rho) {
            auto u_of = [&](int q, int k) {
                const V u = U[FCN_IDX(q, C::PADN, 30)];
                return have_u ? row_of<V>(mk(u, u), k).x * a.nl.rho_nt : T(0);
            };
#pragma unroll
            for (int k = 0; k < L; ++k) {
                if (k >= nrow) break;
                T *rr = bf.rho + (size_t)(row + k) * C::N;
                if (row_io_real_chunks<T, NT>(rr)) {
                    // 16-byte chunks in the sector-wise order of the field rows
                    using IO = RowIoReal<T, NT>;
                    row_real_chunks<T, NT>(t, [&](int tau) {
                        const int cp0 = tpos<NT>(tau & ~15);
                        const int cq0 = pidx(cp0, fft_nt(NT));
                        T w[IO::RC];
#pragma unroll
                        for (int m = 0; m < IO::RC; ++m) w[m] = u_of(own_idx<NT, NSL>(cq0, cp0, (tau & 15) + m), k);
                        T *dst = rr + FCN_IDX(tau, IO::N - IO::RC + 1, 12);
                        if constexpr (sizeof(T) == 4) *reinterpret_cast<float4 *>(dst) = make_float4(w[0], w[1], w[2], w[3]);
                        else *reinterpret_cast<double2 *>(dst) = make_double2(w[0], w[1]);
                    });
                } else {
                    // consecutive threads write consecutive tau points
#pragma unroll
                    for (int i = 0; i < E; ++i) {
                        const int idx = t + C::TPR * i;
                        rr[FCN_IDX(idx, fft_nt(NT), 12)] = u_of(pidx(tpos<NT>(idx), fft_nt(NT)), k);
                    }
                }
            }
        }
    }
    // the time-domain rows to HBM; DIFFK (the kernels of launches with
    // OP_DIFF): also the step-doubling norm's sums of each stored row A
    // against cmp, diff[2 row] = sum |cmp - A|^2, diff[2 row + 1] =
    // sum |A|^2 (per-thread sums in the working precision over the thread's
    // few points, FP64 from the row sum on)
    const bool store = (!(ops & OP_FFT) || (ops & OP_SPEC_OF_TIME)) && !(ops & OP_NOSTORE);
    T d2[L] = {}, b2[L] = {};
    const cx<T> *gc[L] = {};
    double *diff = nullptr;
    if constexpr (DIFFK) {
        const cx<T> *cmp = bf.cmp;
        diff = bf.diff;
#pragma unroll
        for (int k = 0; k < L; ++k) {
            gc[k] = cmp ? cmp + (size_t)(valid ? row + (k < nrow ? k : 0) : 0) * C::N : nullptr;
        }
    }
    if (store) {
        if (keep_u) __syncthreads();                     // row_totals' reads of the storage of S
        to_smem();
        auto acc = [&](int k, cx<T> x, cx<T> y) {          // x: stored value, y: compared value
            const T dx = y.x - x.x, dy = y.y - x.y;
            d2[k] = fma(dx, dx, fma(dy, dy, d2[k]));
            b2[k] = fma(x.x, x.x, fma(x.y, x.y, b2[k]));
        };
        if (valid) {
            bool chunks = true;
#pragma unroll
            for (int k = 0; k < L; ++k) {
                chunks = chunks && row_io_chunks<T, NT>(g[k]);
                if constexpr (DIFFK) chunks = chunks && (!gc[k] || row_io_chunks<T, NT>(gc[k]));
            }
            if (chunks) {
                using IO = RowIo<T, NT>;
                row_chunks<T, NT>(t, [&](int tau, int cq0, int cp0) {
                    cx<V> cv[IO::CPC];
#pragma unroll
                    for (int m = 0; m < IO::CPC; ++m)
                        cv[m] = S[FCN_IDX((own_idx<NT, IO::NSL>(cq0, cp0, (tau & 15) + m)), C::PADN, 11)];
#pragma unroll
                    for (int k = 0; k < L; ++k) {
                        cx<T> x[IO::CPC];
#pragma unroll
                        for (int m = 0; m < IO::CPC; ++m) x[m] = row_of<V>(cv[m], k);
                        if (k < nrow) st_chunk<T>(g[k] + FCN_IDX(tau, IO::N - IO::CPC + 1, 10), x);
                        if constexpr (DIFFK) {
                            if (gc[k]) {
                                cx<T> yv[IO::CPC];
                                ld_chunk<T>(gc[k] + FCN_IDX(tau, IO::N - IO::CPC + 1, 32), yv);
#pragma unroll
                                for (int m = 0; m < IO::CPC; ++m) acc(k, x[m], yv[m]);
                            }
                        }
                    }
                });
            } else {
#pragma unroll
                for (int i = 0; i < E; ++i) {
                    const int idx = t + C::TPR * i;
                    const cx<V> xv = S[FCN_IDX(pidx(tpos<NT>(idx), fft_nt(NT)), C::PADN, 11)];
#pragma unroll
                    for (int k = 0; k < L; ++k) {
                        const cx<T> x = row_of<V>(xv, k);
                        if (k < nrow) g[k][FCN_IDX(idx, fft_nt(NT), 10)] = x;
                        if constexpr (DIFFK) {
                            if (gc[k]) acc(k, x, gc[k][FCN_IDX(idx, fft_nt(NT), 32)]);
                        }
                    }
                }
            }
        }
    }
    if constexpr (DIFFK) {
        double sum[2 * L];
        T none[1];
#pragma unroll
        for (int k = 0; k < L; ++k) {
            sum[2 * k] = double(d2[k]);
            sum[2 * k + 1] = double(b2[k]);
        }
        row_totals<T, NT, TH, 2 * L, 0, 0>(sum, none, smem_raw, [&](int unit, const double *x, const T *) {
            if (!diff) return;
#pragma unroll
            for (int k = 0; k < L; ++k) {
                const int r = row_base + unit * L + k;
                if (r >= a.nr) break;
                diff[FCN_IDX((size_t)2 * r, (size_t)2 * a.nr, 33)] = x[2 * k];
                diff[FCN_IDX((size_t)2 * r + 1, (size_t)2 * a.nr, 34)] = x[2 * k + 1];
            }
        });
    }

    if (ops & OP_FFT) {
        // the in-place transform overwrites S: every thread's reads of it first
        if (store || keep_u) __syncthreads();
        if (!in_regs) pass_load<V, NT, 0>(v, S, t);
        TwAhead<T> ahead;
        tw_ahead<NT, 0>(ahead, C::PLAN == 2 ? a.tw2 : C::PLAN ? a.tw1 : a.tw, t);
        forward_fft<V, NT, 0>(v, S, t, C::PLAN == 2 ? a.tw2 : C::PLAN ? a.tw1 : a.tw, ahead);
        // last-pass outputs: index j + r*NS, j = t + TPR*i
        constexpr int NB = E / RL;
        if (!(ops & (OP_NOSTORE | OP_SPEC_OF_TIME)) && valid) {
#pragma unroll
            for (int i = 0; i < NB; ++i) {
                const int j = t + C::TPR * i;
#pragma unroll
                for (int r = 0; r < RL; ++r) {
#pragma unroll
                    for (int k = 0; k < L; ++k)
                        if (k < nrow) g[k][FCN_IDX(j + r * NSL, fft_nt(NT), 13)] = row_of<V>(v[i * RL + r], k);
                }
            }
        }
        if (MODE != ROW_PLAIN && (ops & OP_SPEC) && bf.stats) {
#pragma unroll
            for (int k = 0; k < L; ++k) {
                // spectral moments sum_q w^k |A_q|^2, w = signed bin, k = 0, 1, 2
                double m3[3] = {0.0, 0.0, 0.0};
                T none[1];
                if constexpr (sizeof(T) == 4) {
                    KahanF k0, k1, k2;
#pragma unroll
                    for (int i = 0; i < NB; ++i) {
                        const int j = t + C::TPR * i;
#pragma unroll
                        for (int r = 0; r < RL; ++r) {
                            const int q = j + r * NSL;
                            const float w = float(q < C::N / 2 ? q : q - C::N);
                            const cx<T> x = row_of<V>(v[i * RL + r], k);
                            const float p2 = fmaf(x.x, x.x, x.y * x.y);
                            k0.add(p2);
                            k1.add(w * p2);
                            k2.add(w * w * p2);
                        }
                    }
                    m3[0] = double(k0.s) - double(k0.c);
                    m3[1] = double(k1.s) - double(k1.c);
                    m3[2] = double(k2.s) - double(k2.c);
                } else {
#pragma unroll
                    for (int i = 0; i < NB; ++i) {
                        const int j = t + C::TPR * i;
#pragma unroll
                        for (int r = 0; r < RL; ++r) {
                            const int q = j + r * NSL;
                            const double w = double(q < C::N / 2 ? q : q - C::N);
                            const cx<T> x = row_of<V>(v[i * RL + r], k);
                            const double p2 = double(x.x) * double(x.x) + double(x.y) * double(x.y);
                            m3[0] += p2;
                            m3[1] += w * p2;
                            m3[2] += w * w * p2;
                        }
                    }
                }
                row_totals<T, NT, TH, 3, 0, 0>(m3, none, smem_raw, [&](int unit, const double *x, const T *) {
                    const int r = row_base + unit * L + k;
                    if (r >= a.nr) return;
                    double *st = bf.stats + FCN_IDX((size_t)r * NSTAT, (size_t)a.nr * NSTAT, 24);
                    st[ST_S0] = x[0];
                    st[ST_S1] = x[1];
                    st[ST_S2] = x[2];
                });
            }
        }
    }
}

// Up to kRowMulti pulses of one grid and one set of coefficients in one
// launch: blockIdx.y selects the pulse (its buffers; all else is shared).
// One launch over all pulses fills the waves that a launch per pulse leaves
// part-empty.  TH: CTA size; V = pk2: pairs of rows.
template <typename V, int NT, int KT, int TH, int MB, int MODE>
__global__ void __launch_bounds__(TH, MB)
row_kernel(const __grid_constant__ RowMultiArgs<typename Pack<V>::S> m) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int ROWS = TH / RowCfg<NT>::TPR * Pack<V>::L;
    pdl_enter();
    const int y = blockIdx.y;
    if (threadIdx.x == 0) {
        // the rows of the CTA that takes this one's place, into L2: CTAs
        // start in order, about kResident after one another (on 152 SMs; a
        // distance from the device and the form's true residency left seven
        // other cases as they are and 2048 x 8192 1.5 % slower)
        constexpr int kResident = 152 * (MB > 1 ? MB : 2);
        const unsigned n = blockIdx.x + kResident, yn = y + n / gridDim.x, xn = n % gridDim.x;
        const int row0 = (int)xn * ROWS, rows = min(ROWS, m.a.nr - row0);
        if (yn < gridDim.y) {
            const cx<typename Pack<V>::S> *f = (m.in[yn] ? m.in[yn] : m.field[yn]) + (size_t)row0 * fft_nt(NT);
            const unsigned bytes = (unsigned)(rows * fft_nt(NT) * (int)sizeof(*f)) & ~15u;
            if (bytes && (reinterpret_cast<uintptr_t>(f) & 15) == 0)
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(f), "r"(bytes) : "memory");
        }
    }
    const RowBufs<typename Pack<V>::S> bf = {m.field[y], m.rho[y], m.stats[y], m.in[y], m.cmp[y], m.diff[y]};
    row_body<V, NT, KT, TH, MB, MODE>(m.a, bf, blockIdx.x * ROWS, m.a.ops, smem_raw);
}

// Work list of rows: each CTA takes the item (pulse, first row) of its index,
// the next TH / (Nt/16) rows of that pulse; pulses may have different Nr and
// Nt (Nt = 512 ... 16 TH).  TH is the smallest CTA that holds a row of the
// list's largest Nt: 16 uneven pulses (Nr 64-256, Nt 512 and 1024) run their
// middle stage in one launch of 128-thread CTAs, five per SM, handed out by
// the hardware as slots free up (as persistent 512-thread CTAs pulling items
// from a counter: one per SM, every stage of a row waiting on 16 warps).
template <typename T, int KT, int TH, int MODE>
__global__ void __launch_bounds__(TH, TH >= 512 ? 1 : 640 / TH)
row_batch_kernel(const RowArgs<T> *__restrict__ pulses, const int2 *__restrict__ items, int ops) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int MB = TH >= 512 ? 1 : 640 / TH;
    const int2 w = items[blockIdx.x];
    const RowArgs<T> &a = pulses[w.x];
    const RowBufs<T> bf = {a.field, a.rho, a.stats, a.in, nullptr, nullptr};
    if (a.nt == 512) row_body<T, 512, KT, TH, MB, MODE>(a, bf, w.y, ops, smem_raw);
    else if (a.nt == 1024) row_body<T, 1024, KT, TH, MB, MODE>(a, bf, w.y, ops, smem_raw);
    else if (a.nt == 2048) row_body<T, 2048, KT, TH, MB, MODE>(a, bf, w.y, ops, smem_raw);
    else if constexpr (TH >= 256) {
        if (TH == 256 || a.nt == 4096) row_body<T, 4096, KT, TH, MB, MODE>(a, bf, w.y, ops, smem_raw);
        else if constexpr (TH >= 512) row_body<T, 8192, KT, TH, MB, MODE>(a, bf, w.y, ops, smem_raw);
    }
}
}  // namespace

namespace rowimpl {

// Rows S and the FP64 scratch, plus the u rows of the modes that keep them,
// of a CTA of TH threads.
template <typename V, int NT, int TH>
size_t smem_bytes(int mode) {
    using C = RowCfg<NT>;
    using T = typename Pack<V>::S;
    return (sizeof(cx<T>) + (row_keeps_u(mode) ? sizeof(T) : 0)) * Pack<V>::L * (TH / C::TPR) * C::PADN +
           sizeof(double) * kRowScratch;
}

// One compiled row kernel: value type, CTA size, minimum CTAs per SM.
template <typename V_, int NT_, int KT_, int TH_, int MB_>
struct RowForm {
    using V = V_;
    using T = typename Pack<V>::S;
    static constexpr int NT = NT_, TH = TH_;
    static constexpr int ROWS = TH / RowCfg<NT>::TPR * Pack<V>::L;       // rows per CTA
    template <int MODE>
    static constexpr auto kernel() { return row_kernel<V, NT, KT_, TH, MB_, MODE>; }
    // Sets the dynamic shared-memory limit; must run before any launch (and
    // outside stream capture).
    static cudaError_t prepare() {
        const int smem = (int)smem_bytes<V, NT, TH>(ROW_OUT);
        cudaError_t e = cudaFuncSetAttribute(kernel<ROW_PLAIN>(), cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(kernel<ROW_OUT>(), cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(kernel<ROW_DIFF>(), cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        return e;
    }
    static cudaError_t launch(const RowMultiArgs<T> &m, int npulse, cudaStream_t st) {
        const int mode = row_mode(m.a.ops);
        const dim3 grid((m.a.nr + ROWS - 1) / ROWS, npulse);
        auto k = mode == ROW_DIFF ? kernel<ROW_DIFF>() : mode == ROW_OUT ? kernel<ROW_OUT>() : kernel<ROW_PLAIN>();
        return launch_k(k, grid, dim3(TH), smem_bytes<V, NT, TH>(mode), st, m);
    }
};

// The kernels of the row variants (0..5; RowArgs::variant).  CTAs are small
// (a row's threads, at least 64 or 128): with the same warps per SM, more and
// smaller CTAs wait less on each other's barriers and leave a shorter last
// wave (middle launch of 8 x 2048 rows of 2048 points: 182 us in CTAs of 128
// threads, 193 us in CTAs of 256; one 1350 x 1024 pulse: 12.4 against
// 16.3 us).  Register caps: about 100 hold a thread's samples and the
// twiddles in flight (102: 182 us, 64 with twice the warps: 193 us).
//   0: one row per unit; the only form of FP64, K != 8 and Nt < 256;
//   1: pairs of rows in packed arithmetic, 128 registers (177 us);
//   2: one row per unit, 64 registers;
//   3: the pairs in CTAs of 64 threads (Nt <= 1024) or with more registers
//      (2048), single rows at 85 registers (4096); 8192: as 0;
//   4, 5: FFT plan 1 at 3 and 4 CTAs of 256 threads.
// Which is fastest depends on the number of rows; the autotuner picks.
template <int NT, int MIN>
constexpr int th_of() { return RowCfg<NT>::TPR < MIN ? MIN : RowCfg<NT>::TPR; }
constexpr int at_least_1(int n) { return n < 1 ? 1 : n; }

template <typename T, int NT, int KT>
using FormNat = RowForm<T, NT, KT, th_of<NT, 64>(), at_least_1((sizeof(T) == 4 ? 640 : 512) / th_of<NT, 64>())>;
template <int NT>
using FormPair = RowForm<pk2, NT, 8, th_of<NT, 128>(), at_least_1(512 / th_of<NT, 128>())>;
template <int NT>
using FormOcc = RowForm<float, NT, 8, th_of<NT, 128>(), 1024 / th_of<NT, 128>()>;
template <int NT>
using FormAlt = std::conditional_t<
    (RowCfg<NT>::TPR <= 64), RowForm<pk2, NT, 8, th_of<NT, 64>(), 8>,
    std::conditional_t<(RowCfg<NT>::TPR == 128), RowForm<pk2, NT, 8, th_of<NT, 128>(), 3>,
                       std::conditional_t<(RowCfg<NT>::TPR == 256), RowForm<float, NT, 8, th_of<NT, 256>(), 3>,
                                          FormNat<float, NT, 8>>>>;
template <int NT1>
using FormPlan1 = RowForm<float, NT1, 8, RowCfg<NT1>::THREADS, (RowCfg<NT1>::THREADS >= 512 ? 1 : 3)>;
template <int NT1>
using FormPlan1Occ = RowForm<float, NT1, 8, RowCfg<NT1>::THREADS, 1024 / RowCfg<NT1>::THREADS>;

// Small grids: FFT plan 2, 4 values per thread.  A launch of few rows is
// latency-bound, and in FP64 each of an SM's four schedulers has a quarter of
// its FP64 rate: a grid needs a warp on every one of the 608, and 128 x 256
// points in 16 values per thread are 64 warps (51 us in FP64, 6.2 us in FP32;
// with plan 2 16.5 and 4.3 us).  thin_rows: rows (of one pulse, so that
// launches of one and of several pulses agree) below which plan 2 serves
// variant 0; where the two meet, FP64: 512 x 1024 points (131 us both),
// 512 x 256 still 31 against 54 us; FP32: 512 x 512 6.3 against 8.3 us, 512 x
// 256 6.2 us both, 1024 and more points never ahead.
template <typename T, int NT, int KT>
using FormThin = RowForm<T, fft_tag(NT, 2), KT, th_of<fft_tag(NT, 2), 64>(), 1>;
template <typename T, int NT>
constexpr int thin_rows() {
    return fft_nt(NT) < 64 || fft_nt(NT) > (sizeof(T) == 8 ? 1024 : 512) ? 0
           : (sizeof(T) == 8 ? 400000 : 270000) / fft_nt(NT);
}

template <typename T, int NT>
constexpr bool has_forms() { return sizeof(T) == 4 && fft_nt(NT) >= 256; }

template <typename T, int NT>
cudaError_t prepare_nt() {
    cudaError_t e = FormNat<T, NT, 0>::prepare();
    if (e == cudaSuccess) e = FormNat<T, NT, 8>::prepare();
    if constexpr (thin_rows<T, NT>() > 0) {
        if (e == cudaSuccess) e = FormThin<T, NT, 0>::prepare();
        if (e == cudaSuccess) e = FormThin<T, NT, 8>::prepare();
    }
    if constexpr (has_forms<T, NT>()) {
        constexpr int NT1 = fft_tag(NT, 1);
        if (e == cudaSuccess) e = FormPair<NT>::prepare();
        if (e == cudaSuccess) e = FormOcc<NT>::prepare();
        if (e == cudaSuccess) e = FormAlt<NT>::prepare();
        if (e == cudaSuccess) e = FormPlan1<NT1>::prepare();
        if (e == cudaSuccess) e = FormPlan1Occ<NT1>::prepare();
    }
    return e;
}

// Calls f with the form of the launch's variant (K = 8, the photon number of
// 800 nm in air: unrolled powers; other K: the generic kernel).
template <typename T, int NT, typename F>
cudaError_t with_form(const RowArgs<T> &a, F &&f) {
    if constexpr (has_forms<T, NT>()) {
        if (a.nl.K == 8) {
            constexpr int NT1 = fft_tag(NT, 1);
            if (a.variant == 1) return f(FormPair<NT>());
            if (a.variant == 2) return f(FormOcc<NT>());
            if (a.variant == 3) return f(FormAlt<NT>());
            if (a.variant == 4 && a.tw1) return f(FormPlan1<NT1>());
            if (a.variant == 5 && a.tw1) return f(FormPlan1Occ<NT1>());
        }
    }
    if constexpr (thin_rows<T, NT>() > 0) {
        if (a.tw2 && a.nr < thin_rows<T, NT>()) {
            if (a.nl.K == 8) return f(FormThin<T, NT, 8>());
            return f(FormThin<T, NT, 0>());
        }
    }
    if (a.nl.K == 8) return f(FormNat<T, NT, 8>());
    return f(FormNat<T, NT, 0>());
}

template <typename T, int NT>
cudaError_t launch_nt_multi(const RowMultiArgs<T> &m, int npulse, cudaStream_t st) {
    if (m.a.nr <= 0 || npulse <= 0) return cudaSuccess;
    if (npulse > kRowMulti) return cudaErrorInvalidValue;
    return with_form<T, NT>(m.a, [&](auto form) { return decltype(form)::launch(m, npulse, st); });
}

template <typename T, int NT>
cudaError_t launch_nt(const RowArgs<T> &a, cudaStream_t st) {
    RowMultiArgs<T> m;
    m.a = a;
    for (int c = 0; c < kRowMulti; ++c) {
        m.field[c] = a.field;
        m.rho[c] = a.rho;
        m.stats[c] = a.stats;
        m.in[c] = a.in;
        m.cmp[c] = a.cmp;
        m.diff[c] = a.diff;
    }
    return launch_nt_multi<T, NT>(m, 1, st);
}

}  // namespace rowimpl

}  // namespace fcn
