// kernels_pic.cu -- the 1D electromagnetic PIC around the emission step.
//
//  k_pic_particles  one thread per electron: fields gathered from the grid at
//                   x^n (linear weights), the emission step of Sec. 2.2 (push,
//                   NCS, brems, position), then the electron's current J^{n+1/2}
//                   by charge-conserving linear weighting, summed per CTA in
//                   shared memory and once per CTA into the run's accumulator;
//                   an electron that left [0, L] is removed after its deposit.
//                   The last CTA to finish (a count after the sums) then advances
//                   the grid: E_x -= dt J_x at the half nodes; the wave variants
//                   F+- = E_y +- B_z and G+- = E_z -+ B_y carried one cell along
//                   +-x with the current at the path's midpoint; the laser enters
//                   at x = 0; the sums and the count are cleared for the next step.
//                   One launch per step.
//  k_pic_rho        ion charge of the neutral start (the electrons' initial
//                   charge with the opposite sign), a diagnostic of Gauss's law.
//
// Currents are summed as dimensionless 2^-36 fixed-point integers, one rounding
// per contribution: exact and independent of the order of the atomic adds.
#include "kernels.cuh"

namespace pe {

namespace {

__device__ __forceinline__ long long fxq(double v) { return __double2ll_rn(v * 68719476736.0); }
__device__ __forceinline__ long long fxq(float v) { return __float2ll_rn(v * 68719476736.0f); }

// weight of grid point k (node, or half node with off = 1/2) for a particle at s = x/dx
template <typename R>
__device__ __forceinline__ R lin_w(R s, int k, R off) {
    R d = fabs(s - ((R)k + off));
    return d < (R)1 ? (R)1 - d : (R)0;
}

__device__ __forceinline__ void acc_add(unsigned long long* a, long long v) {
    if (v) atomicAdd(a, (unsigned long long)v);
}

// Shared-memory current sums as two 32-bit words per grid word (32-bit shared atomics are native, 64-bit ones a
// compare-and-swap loop): a contribution V = rn(v 2^36) (|v| <= 1) adds h = rint(v 2^20) to the high word and
// l = V - 2^16 h, |l| <= 2^15, to the low word, both signed.  In FP32 h and l come from two magic-number roundings:
// t = v 2^20 and its remainder r = t - h are exact, and since 2^16 h is even, rn(r 2^16) rounds as V does.  A
// float-to-64-bit conversion runs on the FP64 pipe (64 clocks of a scheduler for a warp, eight of them an
// electron: a fifth of the step).  Up to kFlushTiles tiles of 256 electrons (each adds at most once per word per
// electron) both sums stay below 2^31 in magnitude; the CTA then moves them into the run's 64-bit sums.
constexpr int kFlushTiles = 7;
struct SplitSums {
    int* hi;   // [3 n_cells]
    int* lo;   // [3 n_cells]
};
__device__ __forceinline__ void acc_add(const SplitSums& a, int k, float v) {
    const float t = v * 0x1.0p20f;
    const float hb = t + 0x1.8p23f;
    const float lb = (t - (hb - 0x1.8p23f)) * 0x1.0p16f + 0x1.8p23f;
    const int h = __float_as_int(hb) - 0x4B400000, l = __float_as_int(lb) - 0x4B400000;
    if ((h | l) && fabsf(v) < 2.0f) {                   // nothing for a NaN (an electron removed at the next step)
        atomicAdd(a.hi + k, h);
        atomicAdd(a.lo + k, l);
    }
}
__device__ __forceinline__ void acc_add(const SplitSums& a, int k, double v) {
    const long long q = fxq(v);
    if (q) {
        atomicAdd(a.hi + k, (int)(q >> 16));
        atomicAdd(a.lo + k, (int)(q & 0xffff));
    }
}
__device__ __forceinline__ void flush_split(const SplitSums& a, int nj, unsigned long long* acc) {
    for (int k = threadIdx.x; k < nj; k += blockDim.x) {
        const long long v = (long long)a.hi[k] * 65536 + (long long)a.lo[k];
        if (v) atomicAdd(acc + k, (unsigned long long)v);
        a.hi[k] = 0;
        a.lo[k] = 0;
    }
}

// current of one electron moving from x_old to x_new (|x_new - x_old| < dx) with
// velocity (vy, vz): J_x at half nodes from the change of its node weights
// (cumulative, charge conserving); J_y, J_z at half nodes with the mean of its
// half-node weights at the two positions.  Dimensionless sums; the field kernel
// applies the weight and the charge sign.
template <typename R>
__device__ __forceinline__ void pic_deposit(R dx, int n, R x_old, R x_new, R vy, R vz, const SplitSums& sj) {
    const R so = x_old / dx, sn = x_new / dx;
    const int ia = (int)floor(so < sn ? so : sn);
    R cum = 0;
#pragma unroll
    for (int k = ia; k <= ia + 1; ++k) {
        cum += lin_w<R>(sn, k, (R)0) - lin_w<R>(so, k, (R)0);
        if (k >= 0 && k < n) acc_add(sj, k, cum);
    }
#pragma unroll
    for (int k = ia - 1; k <= ia + 1; ++k) {
        const R sbar = (R)0.5 * (lin_w<R>(so, k, (R)0.5) + lin_w<R>(sn, k, (R)0.5));
        if (sbar > (R)0 && k >= 0 && k < n) {
            acc_add(sj, n + k, vy * sbar);
            acc_add(sj, 2 * n + k, vz * sbar);
        }
    }
}

// The field update of one step by one CTA of any size: E_x -= dt J_x at the half nodes;
// F+ and G+ carried one cell along +x, F- and G- along -x, each with the current at the
// midpoint of its path; the laser enters at x = 0; the current sums are cleared.  In place, by blocks of kNodes
// nodes a thread: a block's values are formed in registers, all its loads in flight together, and stored after
// a barrier; the +x variants go through the blocks from the right and the -x ones from the left, so no block reads
// what another has written.  The update is the serial end of a step, bound by the latency of its loads (with one
// node after the other a thread, 1000 cells took some 4 us).  The sums are read at L2 (they were built there by atomics).
template <typename R, bool kCP>
__device__ void pic_fields_block(const RunDevT<R>& r) {
    const int n = r.n_cells;
    const StepC<R>& c = r.c;
    R* ex = static_cast<R*>(r.grid);
    R* fp = ex + n;
    R* fm = fp + n + 1;
    R* gp = fm + n + 1;
    R* gm = gp + n + 1;
    unsigned long long* jx = r.jacc;
    unsigned long long* jy = jx + n;
    unsigned long long* jz = jy + n;
    const R dt = c.dt;
    const R kx = c.pic_kx, kyz = c.pic_kyz;   // J_x = kx sum, J_y,z = kyz sum (charge sign included)
    auto J = [](const unsigned long long* a, int i) { return (R)(long long)__ldcg(a + i); };
    constexpr int kNodes = sizeof(R) == 4 ? 4 : 2;
    const int block = kNodes * blockDim.x;
    const int blocks = (n + block) / block;                            // of the n + 1 nodes
    for (int b = 0; b < blocks; ++b) {
        const int right = (blocks - 1 - b) * block + threadIdx.x;      // this thread's nodes: every blockDim-th
        const int left = b * block + threadIdx.x;
        R vp[kNodes], wp[kNodes], vm[kNodes], wm[kNodes], e[kNodes];
#pragma unroll
        for (int k = 0; k < kNodes; ++k) {
            const int i = right + k * blockDim.x, m = left + k * blockDim.x;
            const bool in = i > 0 && i <= n, im = m < n;
            vp[k] = in ? fp[i - 1] - dt * kyz * J(jy, i - 1) : (R)0;   // along +x through half node i - 1
            wp[k] = in ? gp[i - 1] - dt * kyz * J(jz, i - 1) : (R)0;
            vm[k] = im ? fm[m + 1] - dt * kyz * J(jy, m) : (R)0;       // along -x through half node m
            wm[k] = im ? gm[m + 1] - dt * kyz * J(jz, m) : (R)0;
            e[k] = im ? ex[m] - dt * kx * J(jx, m) : (R)0;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kNodes; ++k) {
            const int i = right + k * blockDim.x, m = left + k * blockDim.x;
            if (i <= n) { fp[i] = vp[k]; gp[i] = wp[k]; }
            if (m <= n) { fm[m] = vm[k]; gm[m] = wm[k]; }
            if (m < n) ex[m] = e[k];
        }
        __syncthreads();
    }
    for (int i = threadIdx.x; i < 3 * n; i += blockDim.x) jx[i] = 0;
    if (threadIdx.x == 0) {
        // the laser enters at x = 0: F+ = 2 g_y, G+ = 2 g_z at t^{n+1}
        R gy, gz;
        const R nf1 = (R)(r.step0 + 1);
        plane_e<R, kCP>(c, phase(c, nf1, (R)0, (R)0), gy, gz);
        fp[0] = (R)2 * gy;
        gp[0] = (R)2 * gz;
    }
}

// Resident CTAs of 256 threads per SM the registers are sized for.  FP32, 1e6 electrons, 500 steps: 4 24.6 ms, 2 26.8, 3
// 26.3, 5 27.6 (each CTA adds one flush of its current sums).  FP64 (us a step, 1000 cells): 4 (64 registers, spilled) 451
// at 5e5 electrons and 760 at 1e6, 3 434 / 794, 2 409 / 755.  FP64 with at most a tile a warp takes the emissions in
// place (a queue would send the few electrons of a warp through the rest of the step a second time, at the FP64 price of
// a full warp) and fits 3 CTAs: 1e5 electrons 117, with the queue 173 at 4 CTAs and 147 at 2; 1e3 electrons 44 and 51.
#ifndef PE_PIC_MIN_CTAS
#define PE_PIC_MIN_CTAS 4
#endif
template <typename R, bool kInPlace>
constexpr int pic_ctas() { return sizeof(R) == 4 ? PE_PIC_MIN_CTAS : kInPlace ? 3 : 2; }
constexpr int kPicThreads = 256;
// emissions of a warp that wait (fewer than 32 left by the last round and at most 32 more): electron, eta, gamma
template <typename R>
struct PicQueue {
    uint32_t i[64];
    R eta[64], gamma[64];
};

// kCommon: NCS on and direct brems (a PIC run has no absorbing box), known at compile time.  The rate tables are read
// from shared memory if `staged`.
//
// An emission is several times as long as the rest of the step and falls to a few per cent of the electrons, so more
// than half of the warps would issue all of it for one or two lanes.  An electron whose optical depth crosses is
// (unless kInPlace) stored as it is after the push and queued by its warp; the warp takes the queue 32 emissions at a
// time, or what there is when its electrons of the round are done, and goes through the rest of the step with them.  1e6
// electrons, 1000 cells, steps 0 to 500 (us per step): 59 with the emissions where they fell, 64-bit shared sums and a kernel that waits
// for the one before; 58.6 with the currents' 64-bit conversions off the FP64 pipe; 49 with the queue, native sums and
// overlapped launches; 48 with the test of Eq. 4 from the draw's high word; 45 with the field update below.  5000
// electrons: 19, now 14, the length of the chain from one step's loads to the next's.  What is left is issue (0.6 a
// cycle, some 900 instructions for 32 electrons, a quarter of them the deposit).
template <typename R, bool kCommon, bool kInPlace>
__global__ void __launch_bounds__(kPicThreads, (pic_ctas<R, kInPlace>()))
    k_pic_particles(TablesDev t, RunDevT<R> r, int staged) {
    extern __shared__ __align__(16) unsigned char smem[];
    PicQueue<R>* s_queue = reinterpret_cast<PicQueue<R>*>(smem);
    int* s_j = reinterpret_cast<int*>(s_queue + kPicThreads / 32);              // 3 n_cells current sums (split)
    const int nj = 3 * r.n_cells;
    uint32_t* s_hist = reinterpret_cast<uint32_t*>(s_j + 2 * nj);
    R* s_h = reinterpret_cast<R*>(s_hist + PE_HIST_WORDS + PE_T_E_NCS_STORED + 8 * kEnergySums);
    R* s_sig = s_h + t.n_eta;
    const SplitSums sj{s_j, s_j + nj};
    const SumsDigits acc{s_hist, s_hist + PE_HIST_WORDS, s_hist + PE_HIST_WORDS + PE_T_E_NCS_STORED};
    const R* g_h = (sizeof(R) == 4) ? (const R*)t.h32 : (const R*)t.h64;
    const R* g_sig = (sizeof(R) == 4) ? (const R*)t.sig32 : (const R*)t.sig64;
    constexpr int kWords = PE_HIST_WORDS + PE_T_E_NCS_STORED + 8 * kEnergySums;
    static_assert(kWords % 2 == 0, "cleared in 8-byte words");
    for (int k = threadIdx.x; k < nj + kWords / 2; k += blockDim.x) reinterpret_cast<int2*>(s_j)[k] = make_int2(0, 0);
    if (staged) {
        for (int k = threadIdx.x; k < t.n_eta; k += blockDim.x) s_h[k] = g_h[k];
        for (int k = threadIdx.x; k < t.n_Z * t.n_E; k += blockDim.x) s_sig[k] = g_sig[k];
    }
    // what follows reads what the previous step wrote: the launch of this kernel may overlap its end
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __syncthreads();

    const R* h_tab = staged ? s_h : g_h;
    const R* sig_z = (staged ? s_sig : g_sig) + (size_t)r.iz * t.n_E;
    const uint32_t step = (uint32_t)r.step0;
    const R nf = (R)step;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    PicQueue<R>& Q = s_queue[warp];
    // groups of kFlushTiles tiles: the split sums and the digits stay in range
    for (int64_t group = (int64_t)blockIdx.x * blockDim.x; group < r.n; group += kFlushTiles * stride) {
        int64_t base = group + 32 * warp;
        int tiles = 0, queued = 0;
        while (true) {
            const bool more = tiles < kFlushTiles && base < r.n;
            const int emitting = queued >= 32 ? 32 : (more ? 0 : queued);     // of the warp, this round
            if (!more && !emitting) break;
            int64_t i = 0;
            bool on = false;
            Particle<R> P;
            R gamma, inv_g, x_old;
            if (emitting) {
                if (lane < emitting) {
                    const int at = queued - emitting + lane;
                    i = Q.i[at];
                    gamma = Q.gamma[at];
                    load_particle<R>(r, i, P);
                    x_old = P.x + P.x_lo;
                    emit_one<R>(t, r, r.id0 + (uint32_t)i, step, P, gamma, inv_g, Q.eta[at], acc);
                    on = true;
                }
                queued -= emitting;
            } else {
                i = base + lane;
                bool active = i < r.n;
                if (active) {
                    load_particle<R>(r, i, P);
                    active = live_or_kill<R>(r, i, P, step, r.tally);
                }
                bool crossed = false;
                R eta;
                if (active) {
                    x_old = P.x + P.x_lo;
                    crossed = push_one<R, FK_PIC, kCommon>(t, r, h_tab, nf, P, gamma, inv_g, eta, acc);
                    if (kInPlace && crossed) {
                        emit_one<R>(t, r, r.id0 + (uint32_t)i, step, P, gamma, inv_g, eta, acc);
                        crossed = false;
                    }
                }
                if constexpr (!kInPlace) {
                    const unsigned mask = __ballot_sync(0xffffffffu, crossed);
                    if (crossed) {
                        const int at = queued + __popc(mask & ((1u << lane) - 1u));
                        Q.i[at] = (uint32_t)i;
                        Q.eta[at] = eta;
                        Q.gamma[at] = gamma;
                        store_particle<R>(r, i, P);
                    }
                    queued += __popc(mask);
                }
                on = active && !crossed;
                base += stride;
                ++tiles;
            }
            __syncwarp();
            if (on) {
                rest_one<R, FK_PIC, kCommon>(t, r, sig_z, r.id0 + (uint32_t)i, step, P, gamma, inv_g, acc);
                const R g = m_sqrt((R)1 + P.u[0] * P.u[0] + P.u[1] * P.u[1] + P.u[2] * P.u[2]);
                const R x_new = P.x + P.x_lo;
                pic_deposit<R>(r.c.dt, r.n_cells, x_old, x_new, P.u[1] / g, P.u[2] / g, sj);
                if (x_new < (R)0 || x_new > r.c.box1) {   // it left through a boundary face, carrying its charge out
                    P.x = (R)NAN;
                    atomicAdd(r.tally + PE_T_N_KILLED, 1ull);
                    atomicAdd(r.tally + PE_T_KILLED_STEPS, (unsigned long long)step + 1ull);
                }
                store_particle<R>(r, i, P);
            }
            __syncwarp();
        }
        __syncthreads();
        flush_split(sj, nj, r.jacc);
        acc.flush_energies(r.tally);
        __syncthreads();
    }
    acc.flush_counts(r.hist, r.tally);
    // the last CTA to finish (its sums and every other CTA's are in the run's sums) advances
    // the fields; the count word after the sums goes back to zero for the next step
    __shared__ bool s_last;
    __threadfence();
    __syncthreads();
    unsigned int* done = reinterpret_cast<unsigned int*>(r.jacc + 3 * r.n_cells);
    if (threadIdx.x == 0) s_last = atomicAdd(done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (s_last) {
        __threadfence();
        if (r.polarisation == PE_CP) pic_fields_block<R, true>(r);
        else pic_fields_block<R, false>(r);
        if (threadIdx.x == 0) *done = 0;
    }
}

constexpr int kFieldThreads = 1024;

template <typename R>
__global__ void __launch_bounds__(256) k_pic_rho_deposit(RunDevT<R> r) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= r.n) return;
    Particle<R> P;
    load_pos(r, i, P);
    const R x = P.x + P.x_lo;
    if (isnan(x)) return;
    const R s = x / r.c.dt;
    const int i0 = (int)floor(s);
    for (int k = i0; k <= i0 + 1; ++k)
        if (k >= 0 && k <= r.n_cells) acc_add(r.jacc + k, fxq(lin_w<R>(s, k, (R)0)));
}

template <typename R>
__global__ void __launch_bounds__(kFieldThreads) k_pic_rho_store(RunDevT<R> r) {
    const int n = r.n_cells;
    R* rho = static_cast<R*>(r.grid) + n + 4 * (n + 1);
    for (int i = threadIdx.x; i <= n; i += blockDim.x) {
        rho[i] = -r.c.pic_kyz * (R)(long long)r.jacc[i];   // + (w/dx) sum of node weights
        r.jacc[i] = 0;
    }
}

}  // namespace

// Dynamic shared memory of the particle kernel and whether the rate tables are in it.  Tables that leave no room for the
// queues are read in global memory; a grid and tables beyond kPicSharedMost together are refused (the launch
// fails), as they are without the queues.
constexpr size_t kPicSharedMost = 232448 - 16;
static size_t pic_smem_bytes(const TablesDev& t, int n_cells, int precision, int& staged) {
    const size_t rs = precision == PE_F32 ? 4 : 8;
    const size_t queues = kPicThreads / 32 * (precision == PE_F32 ? sizeof(PicQueue<float>) : sizeof(PicQueue<double>));
    const size_t sums = 4 * (6 * (size_t)n_cells + PE_HIST_WORDS + PE_T_E_NCS_STORED + 8 * kEnergySums);
    const size_t tables = rs * (t.n_eta + (size_t)t.n_Z * t.n_E);
    const size_t grid_and_tables = 8 * (PE_HIST_WORDS + PE_TALLY_WORDS) + 24 * (size_t)n_cells + tables;
    staged = queues + sums + tables <= kPicSharedMost;
    if (grid_and_tables > kPicSharedMost) return grid_and_tables;
    return queues + sums + (staged ? tables : 0);
}

template <typename R>
static void pic_step(const TablesDev& t, const RunDevT<R>& r, int sms, cudaStream_t s) {
    int staged = 1;
    const size_t smem = pic_smem_bytes(t, r.n_cells, sizeof(R) == 4 ? PE_F32 : PE_F64, staged);
    const bool common = r.enable_ncs && r.enable_brems && r.brems_method == PE_BREMS_DIRECT;
    const int64_t blocks = (r.n + kPicThreads - 1) / kPicThreads;
    const bool in_place = sizeof(R) == 8 && blocks <= (int64_t)pic_ctas<R, true>() * sms;
    auto* f = common ? k_pic_particles<R, true, false> : k_pic_particles<R, false, false>;
    if constexpr (sizeof(R) == 8)
        if (in_place) f = common ? k_pic_particles<R, true, true> : k_pic_particles<R, false, true>;
    cudaFuncSetAttribute((const void*)f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    const int64_t most = (int64_t)(in_place ? pic_ctas<R, true>() : pic_ctas<R, false>()) * sms;
    const int grid = (int)(blocks < most ? (blocks > 0 ? blocks : 1) : most);
    // the next step's CTAs start as this step's leave, clear their sums and wait there for its last (griddepcontrol)
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kPicThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, f, t, r, staged);
}

void launch_pic_step(const TablesDev& t, const RunDev& r, int precision, int sms, cudaStream_t s) {
    if (precision == PE_F32) pic_step<float>(t, to_float(r), sms, s);
    else pic_step<double>(t, r, sms, s);
}

void launch_pic_rho(const RunDev& r, int precision, cudaStream_t s) {
    const int grid = (int)((r.n + 255) / 256);
    if (precision == PE_F32) {
        const RunDevT<float> f = to_float(r);
        if (grid > 0) k_pic_rho_deposit<float><<<grid, 256, 0, s>>>(f);
        k_pic_rho_store<float><<<1, kFieldThreads, 0, s>>>(f);
    } else {
        if (grid > 0) k_pic_rho_deposit<double><<<grid, 256, 0, s>>>(r);
        k_pic_rho_store<double><<<1, kFieldThreads, 0, s>>>(r);
    }
}

}  // namespace pe
