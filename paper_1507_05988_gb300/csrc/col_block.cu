// col_block.cu -- the column stage of the FCN z-step (Ma & Lin,
// arXiv:1507.05988, Sec. 3.1, Eqs. (matrix), (matrix1)) with a block of
// adjacent frequency columns per CTA, all rows in registers.
//
// As in col_kernel.cu the pivots are cached per dz and the two Thomas sweeps
//   y_j = alpha_j y_{j-1} + beta_j,   x_j = gamma_j x_{j+1} + y_j
// (alpha_j = i sl_j / piv_j, gamma_j = i sh_j / piv_j, beta_j = rhs_j / piv_j)
// run as chunked affine-map scans: a thread owns L consecutive rows of one
// column.  The products of alpha and of gamma over a chunk depend on the
// table only, so they are formed once per table (the table kernel, or
// launch_cn_prod) instead of in every launch; a chunk then composes its map
// with one multiply-add per row.  y and 1/piv stay in registers from the load
// to the store; alpha and gamma are formed from 1/piv where they are used.
// Shared memory holds the row coefficients (one broadcast load per row) and
// the warps' scan totals only.
//
// What bounds it: one 1024 x 4096 FP32 pulse takes 29-31 us with the field in
// L2 (45 us when x, alpha and gamma went through shared memory and every
// launch formed the chunk products).  Issue is 36 % of the cycles; half of a
// warp's time goes to global loads, which two CTAs of 8 warps per SM (128
// registers a thread) overlap in part.  At 33 us, column segments of 16, 32 or
// 64 bytes per row made no difference, two adjacent columns per thread in
// packed arithmetic took 39 us (the shuffles and shared-memory values double)
// and issuing the loads before the coefficients' 34.
#include <type_traits>

#include "col_scan.cuh"

namespace fcn {
namespace {

using namespace colscan;

// Row coefficients as the kernel reads them (shared memory): sl, sh and, in
// FP32, their low parts.
template <typename T>
struct CoRow;
template <>
struct alignas(16) CoRow<float> {
    float sl, sh, sll, shl;
};
template <>
struct alignas(16) CoRow<double> {
    double sl, sh;
};

// m y + b in a sweep: in FP32 the product first, then one
// rounding at the size of the sum.  (Folded into two FMAs the sum is rounded
// twice, and every later row inherits both.)
template <typename T>
__device__ __forceinline__ cx<T> sweep(cx<T> m, cx<T> y, cx<T> b) {
    if constexpr (sizeof(T) == 4)
        return mk(vfma(y.x, m.x, -(y.y * m.y)) + b.x, vfma(y.x, m.y, y.y * m.x) + b.y);
    else
        return cfma(m, y, b);
}
// Shared-memory index of row j's coefficients: one padding entry per chunk,
// so that the chunks of a warp read different banks.
template <int L>
__host__ __device__ __forceinline__ int co_idx(int j) { return j + j / L; }

// Right-hand sides over pivots, the rounded pivots for the sweep factors and
// the forward map's B of one chunk.  Chunks at the ends of the column run the
// same code with predicates (in a path of their own they would diverge from
// the other chunks of their warp, and the CTA wait for them).
template <typename T, int L>
__device__ __forceinline__ cx<T> block_load(const ColArgs<T> &a, int q, int qq, int j0, const CdCol<T> &cd,
                                            const PivLim<T> &lim, const CoRow<T> *co, cx<T> (&y)[L], cx<T> (&iv)[L]) {
    const int nr = a.nr, nt = a.nt;
    cx<T> x[L + 2];
    // element offsets in 32 bits (a field has at most 2^24 values) from the
    // uniform base pointers
    unsigned o = (unsigned)((j0 - 1) * nt + q);
#pragma unroll
    for (int k = 0; k < L + 2; ++k, o += nt) {
        x[k] = czero<T>();
        if ((k > 0 || j0 > 0) && j0 - 1 + k < nr) x[k] = a.field[FCN_IDX(o, (size_t)nr * nt, 66)];
    }
    o = (unsigned)(j0 * a.tp + qq);
#pragma unroll
    for (int k = 0; k < L; ++k, o += a.tp) {
        iv[k] = czero<T>();
        if (j0 + k < nr) iv[k] = ldg_cx(a.invden + FCN_IDX(o, (size_t)nr * a.tp, 67));
    }
    cx<T> B = czero<T>();
#pragma unroll
    for (int k = 0; k < L; ++k) {
        const CoRow<T> c = co[k];
        // rhs = x_j + i (sl x_{j-1} + sh x_{j+1} - (c0 - delta) x_j); the
        // axis row has its own c0, the last row (A = 0) and the rows past it
        // have none of it
        ExRow<T> e;
        e.sl = c.sl;
        e.sh = c.sh;
        e.d = T(1);
        e.cd = (k == 0 && j0 == 0) ? cd.ah : cd.ih;
        if constexpr (sizeof(T) == 4) {
            e.sll = c.sll;
            e.shl = c.shl;
            e.cdl = (k == 0 && j0 == 0) ? cd.al : cd.il;
        }
        const bool dead = j0 + k >= nr - 1;
        y[k] = piv_apply(ex_rhs(e, x[k], x[k + 1], x[k + 2]), iv[k], lim);
        iv[k] = piv_full(iv[k], lim);           // sl = sh = 0 in the dead rows: any finite value does
        if (dead) y[k] = czero<T>();
        B = cfma(cmul_i(iv[k], c.sl), B, y[k]);
    }
    return B;
}

// Threads of a CTA of C columns: C per chunk of L rows, whole warps.
template <int L, int C>
__host__ __device__ __forceinline__ int block_threads(int nr) { return (C * ((nr + L - 1) / L) + 31) / 32 * 32; }
template <typename T, int L, int C>
__host__ __device__ constexpr size_t block_smem(int threads) {
    return sizeof(CoRow<T>) * (threads / C * (L + 1)) + 3 * sizeof(cx<T>) * (threads / 32 * C);
}

// Columns [g C, g C + C) of one field.  Threads past block_threads(nr) return
// (whole warps, before any barrier); chunks past the last row hold zero maps.
template <typename T, int L, int C, int MAXT>
__device__ __forceinline__ void block_body(const ColArgs<T> &a, int g, unsigned char *smem_raw) {
    const int nr = a.nr, nt = a.nt, tp = a.tp;
    const int nthr = block_threads<L, C>(nr);
    if ((int)threadIdx.x >= nthr) return;
    const int nw = nthr >> 5, P = nthr / C;
    CoRow<T> *co = reinterpret_cast<CoRow<T> *>(smem_raw);
    cx<T> *sA = reinterpret_cast<cx<T> *>(co + P * (L + 1));
    cx<T> *sB = sA + nw * C, *sC = sB + nw * C;
    const int chunk = threadIdx.x / C;
    const int q = g * C + (int)(threadIdx.x % C);
    const int qq = q <= nt / 2 ? q : nt - q;
    const int j0 = chunk * L;
    for (int j = threadIdx.x; j < P * L; j += nthr) {
        CoRow<T> c = {};
        if (j < nr - 1) {
            const CnCoef<T> &f = a.coef[FCN_IDX(j, nr, 68)];
            c.sl = f.sl;
            c.sh = f.sh;
            if constexpr (sizeof(T) == 4) {
                c.sll = f.sll;
                c.shl = f.shl;
            }
        }
        co[FCN_IDX(co_idx<L>(j), P * (L + 1), 65)] = c;
    }
    CdCol<T> cd;
    PivLim<T> lim;
    col_consts<T>(a.cc, a.pivlim, a.s64, a.dk64, qq, &cd, &lim);
    // the chunk's products from those of its kProdRows-row parts
    constexpr int M = L / kProdRows<T>;
    const int NP = (nr + kProdRows<T> - 1) / kProdRows<T>;
    cx<T> PA = czero<T>(), QA = czero<T>();
#pragma unroll
    for (int m = 0; m < M; ++m) {
        const int c = chunk * M + m;
        if (c < NP) {
            const cx<T> f = ldg_cx(a.prod + FCN_IDX(c * tp + qq, 2 * NP * tp, 69));
            const cx<T> b = ldg_cx(a.prod + FCN_IDX((NP + c) * tp + qq, 2 * NP * tp, 70));
            PA = m == 0 ? f : cfma(f, PA, czero<T>());
            QA = m == 0 ? b : cfma(b, QA, czero<T>());
        } else {
            PA = QA = czero<T>();                // rows past nr: the zero map
        }
    }
    __syncthreads();
    const CoRow<T> *cr = co + co_idx<L>(j0);
    cx<T> y[L], iv[L];
    cx<T> B;
    B = block_load<T, L>(a, q, qq, j0, cd, lim, cr, y, iv);
    // exact y from the value entering the chunk
    cx<T> v = block_scan<T, T, false, C, MAXT / 32>(PA, B, nw, sA, sB, sC);
#pragma unroll
    for (int k = 0; k < L; ++k) {
        v = sweep(cmul_i(iv[k], cr[k].sl), v, y[k]);
        y[k] = v;
    }
    // backward sweep: the chunk's map, then x from the value entering it
    B = czero<T>();
#pragma unroll
    for (int k = L - 1; k >= 0; --k) B = cfma(cmul_i(iv[k], cr[k].sh), B, y[k]);
    v = block_scan<T, T, true, C, MAXT / 32>(QA, B, nw, sA, sB, sC);
    unsigned o = (unsigned)((j0 + L - 1) * nt + q);
    if (a.disp == 0.0) {
#pragma unroll
        for (int k = L - 1; k >= 0; --k, o -= nt) {
            v = sweep(cmul_i(iv[k], cr[k].sh), v, y[k]);
            if (j0 + k < nr) a.field[FCN_IDX(o, (size_t)nr * nt, 71)] = v;
        }
    } else {
        const DispPhase<T> ph = disp_phase<T>(a.disp, qq);
#pragma unroll
        for (int k = L - 1; k >= 0; --k, o -= nt) {
            v = sweep(cmul_i(iv[k], cr[k].sh), v, y[k]);
            if (j0 + k < nr) a.field[FCN_IDX(o, (size_t)nr * nt, 71)] = disp_apply(v, ph);
        }
    }
}

template <typename T, int L, int C, int MAXT, int MB>
__global__ void __launch_bounds__(MAXT, MB) cn_block_kernel(const __grid_constant__ ColArgs<T> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    pdl_enter();
    // groups g and ngroups - 1 - g share their pivot columns: adjacent CTAs
    const int ngroups = a.nt / C, b = blockIdx.x;
    block_body<T, L, C, MAXT>(a, (b & 1) ? (ngroups - 1 - (b >> 1)) : (b >> 1), smem_raw);
}

// Work list of columns: each CTA takes the item (pulse, column group) of its
// index; pulses may have different grids.
template <typename T, int L, int C, int MAXT, int MB>
__global__ void __launch_bounds__(MAXT, MB)
cn_block_list_kernel(const ColArgs<T> *__restrict__ pulses, const int2 *__restrict__ items) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int2 w = items[blockIdx.x];
    block_body<T, L, C, MAXT>(pulses[w.x], w.y, smem_raw);
}

// Products of alpha_j (first NP rows of prod) and gamma_j (next NP rows) over
// kProdRows rows, per |q|.
template <typename T>
__global__ void cn_prod_kernel(ColArgs<T> a, cx<T> *prod) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x, c = blockIdx.y;
    if (q > a.nt / 2) return;
    const int NP = gridDim.y;
    CdCol<T> cd;
    PivLim<T> lim;
    col_consts<T>(a.cc, a.pivlim, a.s64, a.dk64, q, &cd, &lim);
    cx<T> A = mk(T(1), T(0)), Q = mk(T(1), T(0));
    for (int j = c * kProdRows<T>; j < min(a.nr, (c + 1) * kProdRows<T>); ++j) {
        const cx<T> inv = piv_full(a.invden[FCN_IDX((size_t)j * a.tp + q, (size_t)a.nr * a.tp, 72)], lim);
        const CnCoef<T> f = a.coef[FCN_IDX(j, a.nr, 73)];
        A = cmul(cmul_i(inv, f.sl), A);
        Q = cmul(cmul_i(inv, f.sh), Q);
    }
    prod[FCN_IDX((size_t)c * a.tp + q, (size_t)2 * NP * a.tp, 74)] = A;
    prod[FCN_IDX((size_t)(NP + c) * a.tp + q, (size_t)2 * NP * a.tp, 75)] = Q;
}

template <typename T, int L, int C, int MAXT, int MB>
cudaError_t launch_form(const ColArgs<T> &a, cudaStream_t st) {
    if (!a.prod || !a.coef || a.nt % C || a.nt < 2 * C) return cudaErrorInvalidConfiguration;
    const int threads = block_threads<L, C>(a.nr);
    if (threads > MAXT) return cudaErrorInvalidConfiguration;
    return launch_k(cn_block_kernel<T, L, C, MAXT, MB>, dim3(a.nt / C), dim3(threads), block_smem<T, L, C>(threads), st,
                    a);
}

}  // namespace

// FP32 forms (chunk rows L, columns C), FP64 in brackets:
//   0: L 16, C 4 in CTAs of up to 256 threads, 128 registers [8, 2]; taller
//      grids as 2 (1024 x 4096: 29-32 us, 45 before; 1350 x 1024: 14.5-17 us,
//      28.5 before);
//   1: L 8, C 4, 512 threads at 64 registers [8, 4 at 128] (1024 x 4096: 35 us,
//      but 128 x 256: 6.3 against 8.2 us);
//   2: L 16, C 8, up to 512 threads at 128 registers, C 4 when taller
//      [8, 4, then 8, 2] (1024 x 4096: 31 us; 2048 x 8192: 140 us, 219 us in
//      one sequential sweep per column);
//   3: small grids: L 8, C 2 [4, 1], CTAs of up to 256 threads (FP64 128 x
//      256: 12.4-15 us against 20 us for 0, 28.8 us before).
template <typename T>
cudaError_t launch_cn_block(const ColArgs<T> &a, int form, cudaStream_t st) {
    constexpr bool F = sizeof(T) == 4;
    cudaError_t e = cudaErrorInvalidConfiguration;
    if (form == 0) e = launch_form<T, F ? 16 : 8, F ? 4 : 2, 256, 2>(a, st);
    else if (form == 1) e = launch_form<T, 8, 4, 512, F ? 2 : 1>(a, st);
    else if (form == 3) e = launch_form<T, F ? 8 : 4, F ? 2 : 1, 256, F ? 4 : 2>(a, st);
    if (e == cudaErrorInvalidConfiguration && form == 2) e = launch_form<T, F ? 16 : 8, F ? 8 : 4, 512, 1>(a, st);
    if (e == cudaErrorInvalidConfiguration) e = launch_form<T, F ? 16 : 8, F ? 4 : 2, 512, 1>(a, st);
    return e;
}

// The batched column launch: L 8, C 8 for grids of up to 512 rows, L 16, C 4
// for taller ones (of up to 2048).
int cn_batch_columns(int max_nr) { return max_nr <= 512 ? 8 : 4; }

template <>
cudaError_t launch_cn_batch<float>(const ColArgs<float> *pulses, const int2 *items, int nitems, int max_nr,
                                   cudaStream_t st) {
    if (max_nr <= 256) {
        const int t = block_threads<8, 8>(max_nr);
        cn_block_list_kernel<float, 8, 8, 256, 3><<<nitems, t, block_smem<float, 8, 8>(t), st>>>(pulses, items);
    } else if (max_nr <= 512) {
        const int t = block_threads<8, 8>(max_nr);
        cn_block_list_kernel<float, 8, 8, 512, 1><<<nitems, t, block_smem<float, 8, 8>(t), st>>>(pulses, items);
    } else {
        const int t = block_threads<16, 4>(max_nr);
        cn_block_list_kernel<float, 16, 4, 512, 1><<<nitems, t, block_smem<float, 16, 4>(t), st>>>(pulses, items);
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_cn_prod(const ColArgs<T> &a, cx<T> *prod, cudaStream_t st) {
    const dim3 grid((a.nt / 2 + 1 + 63) / 64, (a.nr + kProdRows<T> - 1) / kProdRows<T>);
    cn_prod_kernel<T><<<grid, 64, 0, st>>>(a, prod);
    return cudaGetLastError();
}

template cudaError_t launch_cn_block<float>(const ColArgs<float> &, int, cudaStream_t);
template cudaError_t launch_cn_block<double>(const ColArgs<double> &, int, cudaStream_t);
template cudaError_t launch_cn_prod<float>(const ColArgs<float> &, cx<float> *, cudaStream_t);
template cudaError_t launch_cn_prod<double>(const ColArgs<double> &, cx<double> *, cudaStream_t);

}  // namespace fcn
