// xy_kernel.cu -- transverse stage of the FCN z-step on a Cartesian grid
// (Ma & Lin, arXiv:1507.05988, Sec. 2: Delta_perp = d^2/dx^2 + d^2/dy^2 for
// beams without cylindrical symmetry).
//
// Each axis takes the Crank-Nicolson step of Eqs. (diff1)-(diff2) with the
// walls held at A = 0 (Eq. (bound) at r = max, on all four sides); the
// two-dimensional system is not tridiagonal, so the stage applies the x and
// the y factor one after the other (Peaceman-Rachford alternating
// directions; the factors commute, and the product differs from the unsplit
// two-dimensional step by O(dz^3) per step, the order of the Strang split).
// On a line of n nodes, spacing h, s = dz/(4 k0 h^2):
//   walls (j = 0, n-1) : b = 1, everything else 0
//   1..n-2             : a = c = -is, b = 1 + i(2s - delta_q)
//                        d = f =  is, e = 1 - i(2s - delta_q)
// with delta_q = k'' omega_q^2 dz/4 in the y factor and 0 in the x factor.
//
// Inside a line the coefficients do not depend on j, so both sweeps have the
// same factor alpha_j = i s / piv_j, and with the right-hand side divided by
// i s,
//   r_j = (x_{j-1} + x_{j+1}) - c x_j,   c = (2s - delta_q + i) / s,
// they read
//   y_j = alpha_j (y_{j-1} + r_j),   x_j = alpha_j x_{j+1} + y_j,
// alpha = 0 at the walls (and, by that, x = 0 there).  The matrix depends on
// (j, |q|, dz) only: alpha and its products over kXYProd nodes are computed
// once per dz in FP64 (xy_table_kernel).  The sweeps run as a chunked
// parallel scan of affine maps (colscan::block_scan): a thread owns L
// consecutive nodes of one line (FP64) or of two lines of the same frequency
// bin (FP32, in the halves of packed pairs; both share alpha), all in
// registers.  In FP32 alpha and c are two-float pairs (see xy_table_kernel).
// The lines of one launch are addressed as b * bstride + j * pitch + c (see
// XYLine), so the x lines (stride ny*nt) and the y lines (stride nt) use the
// same kernel, with C adjacent frequency columns per CTA for whole-sector row
// accesses.
//
// One FP32 launch on 255 x 255 x 256 points (133 MB) takes 70-72 us, 3.8 TB/s
// of field read and written (86-108 us when every thread formed the factors
// from the pivots four times, the chunk products and c in FP64); bound by
// issue and latency at two CTAs of 8 warps per SM.
#include "col_scan.cuh"

namespace fcn {
namespace {

using namespace colscan;

// One thread per |q| = 0..nt/2: piv_1 = b, piv_j = b - a c / piv_{j-1} =
// b + s^2 / piv_{j-1} (2 <= j <= n-2); the table holds alpha_j = i s / piv_j,
// 0 at the walls: in FP64 one complex double per entry, in FP32 a two-float
// pair (hi, lo).  Layout, rows of nt/2+1 entries: row 0 holds c of each bin,
// row 1 + j alpha_j, and row 1 + n + k the product of alpha over nodes
// k kXYProd .. (k + 1) kXYProd - 1.  On a
// line the coefficients do not depend on j, so the pivots settle to one value
// within a few nodes and the FP32 rounding of alpha is the same at almost
// every node: rounded once it made the discrete factor non-unitary coherently
// along the line, which showed as an energy drift of -2e-8 per line factor
// and step (an FP32 emulation of one line; -3e-10 with two-float factors).
// Without diffraction (s = 0, or too small to change anything: piv = b) the
// table holds 1/b instead, the factor of xy_point_kernel.
constexpr double kXYMinS = 1e-20;
template <typename T>
__global__ void xy_table_kernel(int n, int nt, double s, double dk, cx<T> *table) {
    const int nq = nt / 2 + 1;
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= nq) return;
    auto put = [&](size_t e, cx<double> v) {
        if constexpr (sizeof(T) == 4) {
            const float hx = float(v.x), hy = float(v.y);
            reinterpret_cast<float4 *>(table)[e] = make_float4(hx, hy, float(v.x - double(hx)), float(v.y - double(hy)));
        } else {
            table[e] = mk(T(v.x), T(v.y));
        }
    };
    const double delta = dk * double(q) * double(q);
    const cx<double> b = mk(1.0, 2.0 * s - delta);
    cx<double> inv = crecip(b), prod = mk(1.0, 0.0);
    if (s > kXYMinS) {
        // c of this bin, hi and lo parts: FP64 arithmetic in the line
        // kernel's threads would be a quarter of its time
        const cx<double> c = mk((2.0 * s - delta) / s, 1.0 / s);
        put(q, c);
    }
    table += (size_t)nq * (16 / sizeof(cx<T>));
    for (int j = 0; j < n; ++j) {
        const bool wall = j == 0 || j == n - 1;
        if (j >= 2) inv = crecip(b + mk(s * s * inv.x, s * s * inv.y));
        cx<double> al = s > kXYMinS ? cmul_i(inv, s) : inv;
        if (wall) al = mk(0.0, 0.0);
        put(FCN_IDX((size_t)j * nq + q, (size_t)n * nq, 70), al);
        prod = cmul(al, prod);
        if (j % kXYProd == kXYProd - 1 || j == n - 1) {
            put((size_t)(n + j / kXYProd) * nq + q, prod);
            prod = mk(1.0, 0.0);
        }
    }
}

// alpha as the sweeps use it: a two-float pair in FP32 (FP64: the lo part is
// zero and drops out at compile time).
template <typename T>
struct Piv2 {
    cx<T> h, l;
};
template <typename T>
__device__ __forceinline__ Piv2<T> load_piv(const cx<T> *tab, size_t e) {
    Piv2<T> p;
    if constexpr (sizeof(T) == 4) {
        const float4 w = __ldg(reinterpret_cast<const float4 *>(tab) + e);
        p.h = mk(w.x, w.y);
        p.l = mk(w.z, w.w);
    } else {
        p.h = ldg_cx(tab + e);
        p.l = czero<T>();
    }
    return p;
}
template <typename T>
__device__ __forceinline__ cx<T> load_prod(const cx<T> *tab, size_t e) {
    if constexpr (sizeof(T) == 4) {
        const float2 w = __ldg(reinterpret_cast<const float2 *>(reinterpret_cast<const float4 *>(tab) + e));
        return mk(w.x, w.y);
    } else {
        return ldg_cx(tab + e);
    }
}
// a x with a two-float: the lo product first, then the hi one fused.
template <typename V, typename T>
__device__ __forceinline__ cx<V> cmul2(const Piv2<T> &a, cx<V> x) {
    const auto K = [](T c) { return Pack<V>::splat(c); };
    if constexpr (sizeof(T) == 4) {
        const V tx = vfma(-x.y, K(a.l.y), x.x * K(a.l.x));
        const V ty = vfma(x.y, K(a.l.x), x.x * K(a.l.y));
        return mk(vfma(x.x, K(a.h.x), vfma(-x.y, K(a.h.y), tx)), vfma(x.x, K(a.h.y), vfma(x.y, K(a.h.x), ty)));
    } else {
        return mk(vfma(x.x, a.h.x, -(x.y * a.h.y)), vfma(x.x, a.h.y, x.y * a.h.x));
    }
}

// The thread's value: two lines in FP32 (batch items b = 2 blockIdx.y + i at
// the same column), one in FP64.
template <typename T>
struct LineV;
template <>
struct LineV<float> {
    using V = pk2;
};
template <>
struct LineV<double> {
    using V = double;
};

template <int L, int C>
__host__ __device__ constexpr int xy_threads(int n) { return (C * ((n + L - 1) / L) + 31) / 32 * 32; }

template <typename T, int L, int C, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB) xy_line_kernel(const __grid_constant__ XYLine<T> a) {
    using V = typename LineV<T>::V;
    constexpr int NP = Pack<V>::L;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    pdl_enter();                             // the row or line launch before this one stores the same field
    const int nw = blockDim.x >> 5;
    cx<V> *sB = reinterpret_cast<cx<V> *>(smem_raw);
    cx<V> *sC = sB + nw * C;
    cx<T> *sA = reinterpret_cast<cx<T> *>(sC + nw * C);

    const int c = blockIdx.x * C + (int)(threadIdx.x % C);       // < width (width % C == 0)
    const int chunk = threadIdx.x / C, j0 = chunk * L;
    const int nt = a.nt, n = a.n;
    const int q = c & (nt - 1);
    const int nq = nt / 2 + 1;
    const int qq = (q <= nt / 2) ? q : nt - q;
    const int b0 = blockIdx.y * NP;
    const bool two = NP == 2 && b0 + 1 < a.batch;                // an odd batch's last pair has one line
    cx<T> *l1 = a.field + (size_t)b0 * (size_t)a.bstride + c;
    cx<T> *l2 = l1 + (two ? a.bstride : 0);

    // alpha of the nodes (0 past the line's end) and r in place of y.  (Edge
    // chunks in a path of their own diverge from the other chunks of their
    // warp, and the CTA waits for them: 110 against 84 us.)
    const auto K = [](T c) { return Pack<V>::splat(c); };
    cx<V> y[L];
    Piv2<T> al[L];
    {
        cx<V> x[L + 2];
        const cx<T> *p1 = l1 + (long long)(j0 - 1) * a.pitch, *p2 = l2 + (long long)(j0 - 1) * a.pitch;
#pragma unroll
        for (int k = 0; k < L + 2; ++k, p1 += a.pitch, p2 += a.pitch) {
            x[k] = vzero<V>();
            if ((k > 0 || j0 > 0) && j0 - 1 + k < n) {
                const cx<T> u = *FCN_PTR(p1, a.field, a.total, 73);
                if constexpr (NP == 2) {
                    const cx<T> v = *FCN_PTR(p2, a.field, a.total, 74);
                    x[k] = mk(V{u.x, v.x}, V{u.y, v.y});
                } else {
                    x[k] = u;
                }
            }
        }
        unsigned e = (unsigned)((1 + j0) * nq + qq);
#pragma unroll
        for (int k = 0; k < L; ++k, e += nq) {
            if (j0 + k < n) {
                al[k] = load_piv(a.invden, FCN_IDX(e, (size_t)(n + 1) * nq, 72));
            } else {
                al[k].h = al[k].l = czero<T>();
            }
        }
        // c = (2s - delta_q + i) / s; in FP32 as two-float pairs (lo = rounding
        // error of the FP64 value), so that the rounding of the coefficients
        // does not perturb the discrete operator the same way at every step
        const Piv2<T> cc = load_piv(a.invden, qq);
#pragma unroll
        for (int k = 0; k < L; ++k) {
            V rx = x[k].x + x[k + 2].x, ry = x[k].y + x[k + 2].y;
            const V ux = x[k + 1].x, uy = x[k + 1].y;
            if constexpr (sizeof(T) == 4) {
                rx = vfma(-ux, K(cc.l.x), vfma(uy, K(cc.l.y), rx));
                ry = vfma(-uy, K(cc.l.x), vfma(-ux, K(cc.l.y), ry));
            }
            y[k] = mk(vfma(-ux, K(cc.h.x), vfma(uy, K(cc.h.y), rx)), vfma(-uy, K(cc.h.x), vfma(-ux, K(cc.h.y), ry)));
        }
    }
    // the chunk's product from those of its kXYProd-node parts
    cx<T> PA = czero<T>();
#pragma unroll
    for (int m = 0; m < L / kXYProd; ++m) {
        const int pc = chunk * (L / kXYProd) + m;
        if (pc * kXYProd < n) {
            const cx<T> f = load_prod(a.invden, (size_t)(1 + n + pc) * nq + qq);
            PA = m == 0 ? f : cfma(f, PA, czero<T>());
        } else {
            PA = czero<T>();
        }
    }
    // forward sweep: the chunk's map, then y from the value entering it
    cx<V> v = vzero<V>();
#pragma unroll
    for (int k = 0; k < L; ++k) v = cmul2(al[k], v + y[k]);
    v = block_scan<V, T, false, C, MAXT / 32>(PA, v, nw, sA, sB, sC);
#pragma unroll
    for (int k = 0; k < L; ++k) {
        v = cmul2(al[k], v + y[k]);
        y[k] = v;
    }
    // backward sweep: the same
    v = vzero<V>();
#pragma unroll
    for (int k = L - 1; k >= 0; --k) v = cmul2(al[k], v) + y[k];
    v = block_scan<V, T, true, C, MAXT / 32>(PA, v, nw, sA, sB, sC);
    cx<T> *p1 = l1 + (long long)(j0 + L - 1) * a.pitch, *p2 = l2 + (long long)(j0 + L - 1) * a.pitch;
    auto put = [&](cx<V> r) {
        if constexpr (NP == 2) {
            *FCN_PTR(p1, a.field, a.total, 75) = mk(r.x.a, r.y.a);
            if (two) *FCN_PTR(p2, a.field, a.total, 76) = mk(r.x.b, r.y.b);
        } else {
            *FCN_PTR(p1, a.field, a.total, 75) = r;
        }
    };
    if (a.disp == 0.0) {
#pragma unroll
        for (int k = L - 1; k >= 0; --k, p1 -= a.pitch, p2 -= a.pitch) {
            v = cmul2(al[k], v) + y[k];
            if (j0 + k < n) put(v);
        }
    } else {
        const DispPhase<T> ph = disp_phase<T>(a.disp, qq);
#pragma unroll
        for (int k = L - 1; k >= 0; --k, p1 -= a.pitch, p2 -= a.pitch) {
            v = cmul2(al[k], v) + y[k];
            cx<V> r = v;
            if constexpr (NP == 2) {
                const cx<T> u1 = disp_apply(mk(v.x.a, v.y.a), ph), u2 = disp_apply(mk(v.x.b, v.y.b), ph);
                r = mk(V{u1.x, u2.x}, V{u1.y, u2.y});
            } else {
                r = disp_apply(v, ph);
            }
            if (j0 + k < n) put(r);
        }
    }
}

// Without diffraction (s = 0) a line's factor is (1 + i delta_q) /
// (1 - i delta_q) at every inner node and 0 at the walls (the table holds
// 1/(1 - i delta_q)).  Pointwise, so bound by memory: a thread loads the
// kXYPoint rows of its column before it stores the first.  A step in FP32,
// us: 255 x 31 x 64 points 20, 255 x 255 x 256 221 (threads that walk the
// batch with one load in flight 83 and 331, the line kernel with factors
// alpha = 0 28 and 316; with diffraction 21 and 211).
constexpr int kXYPoint = 4;
constexpr int kXYPointTh = 256;
template <typename T>
__global__ void __launch_bounds__(kXYPointTh) xy_point_kernel(const __grid_constant__ XYLine<T> a) {
    const int cw = min(a.width, kXYPointTh);                     // columns of the CTA, a power of two
    const int c = blockIdx.y * cw + (int)(threadIdx.x & (cw - 1));
    const int rb = kXYPointTh / cw;                              // rows side by side
    const int q = c & (a.nt - 1), nq = a.nt / 2 + 1;
    const int qq = (q <= a.nt / 2) ? q : a.nt - q;
    const double delta = a.dk64 * double(qq) * double(qq);
    const T dh = T(delta), dl = T(delta - double(dh));
    const DispPhase<T> ph = disp_phase<T>(a.disp, qq);
    const Piv2<T> inner = load_piv(a.invden, (size_t)2 * nq + qq);
    // rows in the order in which they lie in memory
    const bool jmajor = a.pitch > a.bstride;
    const int fast = jmajor ? a.batch : a.n, rows = a.n * a.batch;
    const int r0 = blockIdx.x * (rb * kXYPoint) + (int)threadIdx.x / cw;
    cx<T> *p[kXYPoint];
    cx<T> x[kXYPoint];
    bool on[kXYPoint], wall[kXYPoint];
#pragma unroll
    for (int k = 0; k < kXYPoint; ++k) {
        const int r = r0 + k * rb;
        const int hi = r / fast, lo = r - hi * fast;
        const int j = jmajor ? hi : lo, b = jmajor ? lo : hi;
        on[k] = r < rows;
        wall[k] = j == 0 || j == a.n - 1;
        p[k] = a.field + ((size_t)b * (size_t)a.bstride + (size_t)j * (size_t)a.pitch + c);
        x[k] = on[k] ? *FCN_PTR(p[k], a.field, a.total, 77) : czero<T>();
    }
#pragma unroll
    for (int k = 0; k < kXYPoint; ++k) {
        const cx<T> r = mk(vfma(-dh, x[k].y, vfma(-dl, x[k].y, x[k].x)), vfma(dh, x[k].x, vfma(dl, x[k].x, x[k].y)));
        Piv2<T> f = inner;
        if (wall[k]) f.h = f.l = czero<T>();
        if (on[k]) *FCN_PTR(p[k], a.field, a.total, 78) = disp_apply(cmul2(f, r), ph);
    }
}

template <typename T, int L, int C, int MAXT, int MINB>
cudaError_t launch_form(const XYLine<T> &a, cudaStream_t st) {
    using V = typename LineV<T>::V;
    const int threads = xy_threads<L, C>(a.n);
    if (threads > MAXT || a.width % C != 0 || a.nt % C != 0) return cudaErrorInvalidConfiguration;
    const size_t smem = (2 * sizeof(cx<V>) + sizeof(cx<T>)) * (size_t)(threads / 32) * C;
    const dim3 grid(a.width / C, (a.batch + Pack<V>::L - 1) / Pack<V>::L);
    return launch_k(xy_line_kernel<T, L, C, MAXT, MINB>, grid, dim3(threads), smem, st, a);
}

}  // namespace

size_t xy_table_entries(int n, int nt) { return (size_t)(1 + n + (n + kXYProd - 1) / kXYProd) * (size_t)(nt / 2 + 1); }

template <typename T>
cudaError_t launch_xy_table(int n, int nt, double s, double dk, cx<T> *table, cudaStream_t st) {
    const int nq = nt / 2 + 1;
    // one warp per CTA: the recurrence is a serial FP64 chain per bin
    xy_table_kernel<T><<<(nq + 31) / 32, 32, 0, st>>>(n, nt, s, dk, table);
    return cudaGetLastError();
}

// Forms (chunk length L, columns C, CTA size, CTAs per SM asked for), FP32
// [FP64]; a form that does not fit the grid gives way to the longest chunks
// in 512 threads, with fewer columns on the smallest Nt.
//   0: 16, 4, 512 [8, 2]   1: 8, 8, 256 [4, 4]     2: 8, 8, 512 [8, 4]
//   3: 8, 4, 256 [4, 2]    4: 16, 8, 256 [8, 4]    5: 16, 16, 512 [8, 8]
//   6: 8, 16, 512 [4, 8]   7: 8, 4, 128 [4, 2]
template <typename T>
cudaError_t launch_xy_line(const XYLine<T> &a, cudaStream_t st) {
    if (a.n < 3 || a.nt < 1 || (a.nt & (a.nt - 1)) || a.width < 1 || (a.width % a.nt) || a.batch < 1)
        return cudaErrorInvalidValue;
    if (!(a.s64 > kXYMinS)) {
        const int cw = a.width < kXYPointTh ? a.width : kXYPointTh;
        const int per = kXYPointTh / cw * kXYPoint;              // rows per CTA
        xy_point_kernel<T><<<dim3((a.n * a.batch + per - 1) / per, a.width / cw), kXYPointTh, 0, st>>>(a);
        return cudaGetLastError();
    }
    constexpr bool F = sizeof(T) == 4;
    constexpr int LL = F ? 16 : 8, LS = F ? 8 : 4, CF = F ? 1 : 2;      // CF: FP64 columns are half as many
    cudaError_t e = cudaErrorInvalidConfiguration;
    switch (a.variant) {
        case 1: e = launch_form<T, LS, 8 / CF, 256, 2>(a, st); break;
        case 2: e = launch_form<T, 8, 8 / CF, 512, 1>(a, st); break;
        case 3: e = launch_form<T, LS, 4 / CF, 256, 2>(a, st); break;
        case 4: e = launch_form<T, LL, 8 / CF, 256, 1>(a, st); break;
        case 5: e = launch_form<T, LL, 16 / CF, 512, 1>(a, st); break;
        case 6: e = launch_form<T, LS, 16 / CF, 512, 1>(a, st); break;
        case 7: e = launch_form<T, LS, 4 / CF, 128, 4>(a, st); break;
        default: break;
    }
    if (e == cudaErrorInvalidConfiguration) e = launch_form<T, LL, 4 / CF, 512, 1>(a, st);
    if (e == cudaErrorInvalidConfiguration) e = launch_form<T, LL, 2, 512, 1>(a, st);     // Nt = 2
    return e;
}

template cudaError_t launch_xy_table<float>(int, int, double, double, cx<float> *, cudaStream_t);
template cudaError_t launch_xy_table<double>(int, int, double, double, cx<double> *, cudaStream_t);
template cudaError_t launch_xy_line<float>(const XYLine<float> &, cudaStream_t);
template cudaError_t launch_xy_line<double>(const XYLine<double> &, cudaStream_t);

}  // namespace fcn
