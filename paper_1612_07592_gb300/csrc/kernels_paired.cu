// kernels_paired.cu -- the FP32 step: instantiations and dispatch of the paired kernels (two
// electrons per thread) for every prescribed-field kind (the 1D plane wave, its reflection, the 2D
// focus, constant fields), and the plane wave's one-step streaming form.
// This translation unit is built without multiply-add contraction and with IEEE division and
// square root: its kernels (single run, batch, streaming) inline the same emission branches, and
// with every rounding written in the source they agree bit for bit (the approximate forms the
// step needs are explicit instructions in pair_f32.cuh).
#include "kernels.cuh"
#include "pair_f32.cuh"

namespace pe {

// Launches of at most this many steps (the state round-trips memory) on a single run
// of a plane-wave kind use the streaming form of the paired kernel.
constexpr int kStreamMaxSteps = 4;

// The rows of sigma_Z in shared memory: all of them up to 8 KB, where they cost no resident CTA; above that the run's own.
int pair_sig_stride(const TablesDev& t) { return t.n_Z * t.n_E <= 2048 ? t.n_E : 0; }
int pair_smem_bytes(const TablesDev& t) {                            // 54 KB at most (tables of up to 4096 rows)
    return kPairFixedBytes + 4 * (t.n_eta + (pair_sig_stride(t) ? t.n_Z * t.n_E : t.n_E));
}

static bool plane_kind(int fk) { return fk == FK_PLANE_LP || fk == FK_PLANE_CP; }
// tables, then 16-byte alignment slack and the stage buffers
template <int F, bool kOne>
static int stream_smem_bytes(int base) { return base + 16 + StreamShape<F, kOne>::kStages * kStageBytes<F>; }
static bool use_stream(const BatchDevT<float>& b, int steps, int block) {
    return b.n_runs == 1 && plane_kind(b.runs[0].fk) && steps <= kStreamMaxSteps && block == kStreamTile;
}
// beside the static shared memory of a kernel (below 6 KB) a launch may use 48 KB without being told so
static void allow_smem(const void* f, int smem) {
    if (smem > 40 * 1024) cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}

// Whether the lanes of a warp wait for one another's emissions: where these are frequent, in the reflected wave (5 %
// of the particle-steps) and in constant fields when a run's largest bremsstrahlung probability per step P reaches 1e-3;
// not in the plane wave and the 2D focus (below 1e-3).  1 GeV bunch, 2e5 electrons x 1500 steps, us waiting / not: in Au
// at P = 5e-4 1558 / 1395, 1.1e-3 1679 / 1528, 1.6e-3 1765 / 1659, 2.7e-3 1889 / 1876, 5.4e-3 2166 / 2390; by null
// collisions (one candidate in P of the steps) 5e-4 1156 / 1024, 1.1e-3 1284 / 1483, 5.4e-3 2001 / 4424; in Al at 2e-4 1469 /
// 1312 and 1016 / 798.  The direct method alone breaks even at 3e-3 and loses a tenth at most below that; null collisions
// gain from 1e-3 on, and so do runs that emit by NCS as well (a field of 10, P = 1.1e-3: 2075 / 4443 for 1e5 electrons x 800).
template <int G>
static bool hold_of(const BatchDevT<float>& b) {
    if constexpr (G == FK_CONST) {
        for (int k = 0; k < b.n_runs; ++k)
            if (!b.runs[k].enable_brems || b.runs[k].c.P_hat < 1e-3f) return false;
        return true;
    } else {
        return G == FK_REFL_LP || G == FK_REFL_CP;
    }
}

// the flags that every run of a launch has (pair_f32.cuh)
static int flags_of(const BatchDevT<float>& b) {
    bool paper = true, brems = true;
    for (int k = 0; k < b.n_runs; ++k) {
        const RunDevT<float>& r = b.runs[k];
        const bool direct = r.enable_brems && r.brems_method == PE_BREMS_DIRECT && !r.box_enable;
        paper = paper && direct && r.enable_ncs;
        brems = brems && direct && !r.enable_ncs;
    }
    return paper ? kFlagsPaper : brems ? kFlagsBrems : kFlagsRun;
}

// The kernel of a launch, its threads per CTA (block/2: two electrons per thread) and dynamic
// shared memory: the resident paired kernel, or for the plane wave its streaming form.
using StepKernel = void (*)(TablesDev, BatchDevT<float>, int);
template <bool kSingle, int G>
static StepKernel kernel_of(const BatchDevT<float>& b, int steps, int block, int base_smem, int& threads, int& smem) {
    smem = base_smem;
    threads = block / 2;
    const int flags = flags_of(b);
    if constexpr (G == FK_PLANE_LP || G == FK_PLANE_CP) {
        if (kSingle && use_stream(b, steps, block)) {
            auto shape = [&](auto f, auto one) -> StepKernel {
                smem = stream_smem_bytes<decltype(f)::value, decltype(one)::value>(base_smem);
                return k_step_pair_stream<G, decltype(f)::value, decltype(one)::value>;
            };
            using Paper = std::integral_constant<int, kFlagsPaper>;
            using Run = std::integral_constant<int, kFlagsRun>;
            if (flags == kFlagsPaper) return steps == 1 ? shape(Paper{}, std::true_type{}) : shape(Paper{}, std::false_type{});
            return steps == 1 ? shape(Run{}, std::true_type{}) : shape(Run{}, std::false_type{});
        }
    }
    constexpr bool kMayHold = G == FK_REFL_LP || G == FK_REFL_CP || G == FK_CONST;
    constexpr bool kMayNot = G != FK_REFL_LP && G != FK_REFL_CP;
    const bool hold = hold_of<G>(b);
    if constexpr (G == FK_CONST)
        if (flags == kFlagsBrems)
            return hold ? k_step_pair<kSingle, G, kFlagsBrems, true> : k_step_pair<kSingle, G, kFlagsBrems, false>;
    if (flags == kFlagsPaper)
        return hold ? k_step_pair<kSingle, G, kFlagsPaper, kMayHold> : k_step_pair<kSingle, G, kFlagsPaper, !kMayNot>;
    return hold ? k_step_pair<kSingle, G, kFlagsRun, kMayHold> : k_step_pair<kSingle, G, kFlagsRun, !kMayNot>;
}

template <bool kSingle, int G>
static void launch_one(const TablesDev& t, const BatchDevT<float>& b, int steps, int grid, int block, cudaStream_t s,
                       int base_smem) {
    int threads, smem;
    const StepKernel f = kernel_of<kSingle, G>(b, steps, block, base_smem, threads, smem);
    allow_smem((const void*)f, smem);
    // the streaming form is launched once per step or few: the next launch's CTAs start as this one's leave, clear their
    // sums, copy the tables and wait there for its last (griddepcontrol)
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = kSingle && use_stream(b, steps, block) ? 1 : 0;
    cudaLaunchKernelEx(&cfg, f, t, b, steps);
}

template <typename F>
static void with_paired_kind(int fk, F&& f) {
    switch (fk) {
        case FK_PLANE_LP: f(std::integral_constant<int, FK_PLANE_LP>{}); break;
        case FK_PLANE_CP: f(std::integral_constant<int, FK_PLANE_CP>{}); break;
        case FK_GAUSS_LP: f(std::integral_constant<int, FK_GAUSS_LP>{}); break;
        case FK_GAUSS_CP: f(std::integral_constant<int, FK_GAUSS_CP>{}); break;
        case FK_REFL_LP: f(std::integral_constant<int, FK_REFL_LP>{}); break;
        case FK_REFL_CP: f(std::integral_constant<int, FK_REFL_CP>{}); break;
        default: f(std::integral_constant<int, FK_CONST>{}); break;
    }
}

void launch_step_persistent_f32(const TablesDev& t, const BatchDevT<float>& b, int steps, int grid, int block,
                                cudaStream_t s) {
    const int smem = pair_smem_bytes(t);
    with_paired_kind(b.runs[0].fk, [&](auto g) {
        if (b.n_runs == 1) launch_one<true, decltype(g)::value>(t, b, steps, grid, block, s, smem);
        else launch_one<false, decltype(g)::value>(t, b, steps, grid, block, s, smem);
    });
}

// the kernel a launch of these runs uses, its threads per CTA and dynamic shared memory
// (for graph nodes); sets the shared-memory attribute
const void* persistent_kernel_f32(const BatchDevT<float>& b, int steps, int base_smem, int block, int* threads,
                                  int* smem_out) {
    const void* f = nullptr;
    int th = block, smem = base_smem;
    with_paired_kind(b.runs[0].fk, [&](auto g) {
        f = (const void*)(b.n_runs == 1 ? kernel_of<true, decltype(g)::value>(b, steps, block, base_smem, th, smem)
                                        : kernel_of<false, decltype(g)::value>(b, steps, block, base_smem, th, smem));
    });
    allow_smem(f, smem);
    *threads = th;
    *smem_out = smem;
    return f;
}

// Default CTAs per SM of the grid: three resident waves of the resident paired kernel (tiles differ in
// cost with their emission histories, and a CTA per one or two tiles lets the block scheduler balance
// them: measured +6 % over one wave, +2.5 % over two, on 1e6 electrons); one wave for the streaming
// form (each CTA streams many tiles of equal cost).
int default_ctas_per_sm_f32(const BatchDevT<float>& b, int steps, int block, int base_smem) {
    int threads, smem, occ = 0;
    const void* f = persistent_kernel_f32(b, steps, base_smem, block, &threads, &smem);
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, f, threads, smem);
    return (use_stream(b, steps, block) ? 1 : 3) * (e == cudaSuccess && occ > 0 ? occ : 1);
}

}  // namespace pe
