// Host-side dump of the row launches' shared memory for
// tests/test_host_plans.py: per form and set of operations, the bytes the
// launch asks for, the rows and the scratch, and the u rows behind them that
// the kernel of that launch writes when a half step runs.  Compiled for the
// host only; no GPU call.
#include <cstdio>

#include "../paper_1507_05988_gb300/csrc/row_kernel.cuh"

using namespace fcn;

template <typename V, int NT, int TH>
static void dump(const char *name) {
    using C = RowCfg<NT>;
    using T = typename Pack<V>::S;
    const size_t vals = (size_t)(TH / C::TPR) * C::PADN;
    for (int ops = 0; ops < 1024; ++ops) {
        const int mode = row_mode(ops);
        std::printf("%s %d %d %d %d %zu %zu %zu\n", name, fft_nt(NT), TH, ops, mode, rowimpl::smem_bytes<V, NT, TH>(mode),
                    vals * sizeof(cx<V>) + sizeof(double) * kRowScratch, row_keeps_u(mode) ? vals * sizeof(V) : (size_t)0);
        static_assert(sizeof(V) == Pack<V>::L * sizeof(T), "packed");
    }
}

int main() {
    dump<float, 64, 64>("f32");
    dump<float, 4096, 256>("f32");
    dump<double, 4096, 256>("f64");
    dump<pk2, 1024, 64>("pair");
    dump<pk2, 8192, 512>("pair");
    return 0;
}
