// row_batch.cu -- the batched (work-list) row stage: pulses of uneven grids
// (Nt = 512 ... 8192) in one launch per stage.  FP32 with K = 8, the form the
// batched path runs in (see row_kernel.cuh for the row body).
#include "row_kernel.cuh"

namespace fcn {

int row_batch_threads(int max_nt) { return max_nt <= 2048 ? 128 : max_nt <= 4096 ? 256 : 512; }

namespace {
// A CTA of th threads holds 16 th samples and one padding value per 16,
// whatever its rows' Nt, and as many u values in the modes that keep them.
size_t batch_smem(int th, int mode) {
    return (size_t)17 * th * (row_keeps_u(mode) ? 12 : 8) + sizeof(double) * kRowScratch;
}

template <typename F>
cudaError_t with_threads(int th, F &&f) {
    if (th == 128) return f(std::integral_constant<int, 128>());
    if (th == 256) return f(std::integral_constant<int, 256>());
    return f(std::integral_constant<int, 512>());
}
}  // namespace

template <>
cudaError_t prepare_rows_batch<float>(int th) {
    return with_threads(th, [&](auto n) {
        constexpr int TH = decltype(n)::value;
        cudaError_t e = cudaFuncSetAttribute(row_batch_kernel<float, 8, TH, ROW_PLAIN>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)batch_smem(TH, ROW_PLAIN));
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(row_batch_kernel<float, 8, TH, ROW_OUT>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)batch_smem(TH, ROW_OUT));
        return e;
    });
}

template <>
cudaError_t launch_rows_batch<float>(const RowArgs<float> *pulses, const int2 *items, int nitems, int ops, int th,
                                     cudaStream_t st) {
    return with_threads(th, [&](auto n) {
        constexpr int TH = decltype(n)::value;
        const int mode = row_mode(ops) == ROW_PLAIN ? ROW_PLAIN : ROW_OUT;
        auto k = mode == ROW_OUT ? row_batch_kernel<float, 8, TH, ROW_OUT> : row_batch_kernel<float, 8, TH, ROW_PLAIN>;
        k<<<nitems, TH, batch_smem(TH, mode), st>>>(pulses, items, ops);
        return cudaGetLastError();
    });
}

}  // namespace fcn
