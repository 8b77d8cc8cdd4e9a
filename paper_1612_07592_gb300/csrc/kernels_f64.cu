// kernels_f64.cu -- the FP64 step: the instantiations of the persistent kernel for double.
//
// This translation unit is compiled with -fmad=false: no multiply and add is
// contracted into a fused multiply-add unless the source asks for one, so each
// FP64 operation of the step is one IEEE-rounded multiply or add whatever kernel
// (single run or batch, any launch shape) it is inlined into.  The FP64 oracle is built
// with the same rule (no contraction).
#include "kernels.cuh"

namespace pe {

// ---------------------------------------------------------------------------
// persistent kernel for double
// ---------------------------------------------------------------------------
void launch_step_persistent_f64(const TablesDev& t, const BatchDevT<double>& b, int steps, int grid, int block,
                                cudaStream_t s) {
    // all runs of b share one field kind (the caller groups a batch by kind)
    with_field_kind(b.runs[0].fk, [&](auto g) {
        constexpr int G = decltype(g)::value;
        if (b.n_runs == 1) k_step_persistent<double, true, G><<<grid, block, 0, s>>>(t, b, steps);
        else k_step_persistent<double, false, G><<<grid, block, 0, s>>>(t, b, steps);
    });
}

// the kernel a launch of these runs uses (for graph nodes)
const void* persistent_kernel_f64(const BatchDevT<double>& b) {
    const void* f = nullptr;
    with_field_kind(b.runs[0].fk, [&](auto g) {
        constexpr int G = decltype(g)::value;
        f = b.n_runs == 1 ? (const void*)k_step_persistent<double, true, G> : (const void*)k_step_persistent<double, false, G>;
    });
    return f;
}

// Electrons per tile when the caller sets none.  The step is bound by the FP64 pipe, which takes a warp instruction in
// some 64 clocks on each scheduler, full or not: one warp to a scheduler fills it.  Tiles of one warp spread a small
// run over all schedulers (us per step, tiles of 16 / 32 / 64 / 256 electrons: 1e4 electrons 8.8 / 6.5 / 7.0 / 13.3,
// 3e4 22 / 11.7 / 13.3 / 13.3); from about 1e5 on the tile makes no difference (1e5 38.0 / 37.7 with 32 / 256) and the
// larger one flushes its sums less often (3e5 100.6 / 94.5).  One launch per step, tiles of 256 and the rates
// formed for every brems test took 23 us a step on 1e4 electrons (the 2000-step job 46.5 ms, now 12.9).
int default_tile_f64(int64_t n, int sms) { return n <= (int64_t)sms * 512 ? 32 : 256; }

int persistent_occupancy_f64(int block) {
    int occ = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_step_persistent<double, false, FK_PLANE_LP>, block, 0);
    return e == cudaSuccess ? occ : 1;
}

}  // namespace pe
