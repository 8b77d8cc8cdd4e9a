// kernels_pair.cu -- Bethe-Heitler conversion of photon records in the target.
//
// Sec. 2.2 implements pair production by photons in the field of the nuclei like the
// bremsstrahlung: a direct MC collision of Eq. (4), here with the pair cross section
// sigma_BH(k) of the photon energy k.  A photon moves at c along its direction from its
// emission point; at every step inside the target it takes the test, and on a conversion
// the positron fraction x is drawn from the tabulated CDF of Tsai's pair DCS.
//
// Two methods of the same law: the per-step tests of Eq. 4 (the paper's direct collision),
// and the free path (the trials of one crossing share P, so the first success is geometric:
// one draw per photon, the random-free-path sampling Sec. 2.2 mentions).
//
// Rounds of 32 photons per warp.  Each lane first finds its photon's run of consecutive
// steps inside the target, on the FP64 position computed exactly as the definition computes it at each step
// (GB300's FP64 pipe is narrow: the literal per-step position kept it 84 % busy).  Then the warp takes the tests of the
// round's photons one photon at a time, 64 steps at once (the draws are counter-based, so the first passing
// step is found from a ballot): the per-step work is a Philox word and a compare on every lane, whatever the spread
// of path lengths.  Conversions are queued and sampled 32 at a time.
#include "kernels.cuh"

namespace pe {
namespace {

constexpr uint32_t kPurBH = 0x40000000u;      // per-step tests: counter word 3 = kPurBH + emission step
constexpr uint32_t kPurBHFree = 0x50000000u;  // free path: counter word 3 = kPurBHFree + emission step


// sigma_BH(k) by row interpolation in log k over [2, gamma_max] (0 for k <= 2); the row
// position (i, w) is kept for the sampling of x
__device__ __forceinline__ double bh_sigma_of(const TablesDev& t, const double* sig, double k, bool& above, int& i,
                                              double& w) {
    const TabC<double>& c = t.cd;
    above = false;
    if (!(k > 2.0)) return 0.0;
    int fl;
    row_pos<double>(k, c.ln_k_min, c.inv_dln_k, c.g_last, t.n_E, i, w, fl);
    i = dbg_idx(t.dbg, i, t.n_E - 1);
    above = (fl == 1);
    return (1.0 - w) * sig[i] + w * sig[i + 1];
}

// positron fraction x in [1/k, 1 - 1/k] from the CDF interpolated at row position (i, w) of k,
// at uniform Rv (2/k is formed as 2 (1/k), the same double)
__device__ __forceinline__ double bh_sample_x(const TablesDev& t, const double* cdf_z, double k, int i, double w,
                                              double Rv) {
    const double* ra = cdf_z + (size_t)i * t.n_s;
    const double* rb = ra + t.n_s;
    int j;
    const double fr = invert_rows<double>(ra, rb, w, t.n_s, Rv, j);
    double s;
    if (j < 0) s = 0.0;
    else if (j >= t.n_s - 1) s = 1.0;
    else s = ((double)j + fr) / (double)(t.n_s - 1);
    const double ik = 1.0 / k;
    return ik + s * (1.0 - 2.0 * ik);
}


#ifndef PE_PAIR_MIN_CTAS_SM
#define PE_PAIR_MIN_CTAS_SM 3      // resident CTAs of 256 threads per SM the registers are sized for
#endif
constexpr int kPairThreads = 256;
// conversions of a warp that wait for their sampling: photon, step and the two words of the positron's share (fewer
// than 32 left by the last round and at most 32 more)
struct PairQueue {
    uint32_t j[64], step[64], z[64], w[64];
};

// The first step m of [a + 1, b] with past(m), which is false at a and true from some step up to b on: from the crossing
// time in float (`guess` steps after ne), then the exact test on either side of it.  A binary search took some dozen of
// these tests (four FP64-pipe instructions each); the float time is off by less than a step (2e-7 of it).
template <typename P>
__device__ __forceinline__ int64_t first_past(int64_t a, int64_t b, int64_t ne, float guess, P past) {
    int64_t m = ne + (guess > 0.0f && guess < 4.0e9f ? (int64_t)__float2uint_rz(guess) : 0);
    m = m <= a ? a + 1 : m > b ? b : m;
    while (m > a + 1 && past(m - 1)) --m;
    while (!past(m)) ++m;
    return m;
}

// kFree: the free-path method (one geometric draw per photon) instead of the per-step tests.
//
// The tests: integer issue.  A passing draw is below the threshold, so its high word is at most the threshold's; that
// word alone is formed for every test (eight of Philox's twenty products fewer, with the first rounds' on the
// photon's own words, the same for all its tests), the whole draw for the few that low.  What is FP64 -- the
// bounds of a photon's run of steps, its threshold, the sampling of a conversion -- runs on 32 photons or 32 queued
// conversions at a time: the FP64 pipe takes the same time for one lane.  3e5 photons, 2.8e8 tests through 1.5 mm of Au:
// 1.21 ms with whole draws, binary searches and each conversion sampled by its own lane, now 0.78 (47 instructions for 32
// tests, from 86; bound by the integer multiplies, four clocks of a scheduler each); the free path, 3e6 photons, 2.34
// and 1.71 ms.
template <bool kFree>
__global__ void __launch_bounds__(kPairThreads, PE_PAIR_MIN_CTAS_SM) k_pair_transport(
    TablesDev t, RunDev r, const Photon* ph, int64_t n_ph, int64_t step_end, int per_round, PairRec* out, int64_t cap,
    unsigned long long* tally) {
    __shared__ PairQueue s_queue[kPairThreads / 32];
    const StepC<double>& c = r.c;
    const double* sig = t.bhsig64 + (size_t)r.iz * t.n_E;
    const double* cdf = t.bhcdf64 + (size_t)r.iz * t.n_E * t.n_s;
    const bool two_d = r.geometry == PE_GAUSS_2D;
    const uint32_t lane = threadIdx.x & 31;
    PairQueue& Q = s_queue[threadIdx.x >> 5];
    int queued = 0;                                 // conversions in Q (the same on every lane)
    unsigned long long n_entered = 0, n_above = 0, tests = 0;      // of the warp (the same on every lane); of the lane
    ulonglong2 e_pairs = make_ulonglong2(0, 0), e_pos = make_ulonglong2(0, 0);   // of the lane
    // the last `count` queued conversions, one to a lane: the positron's share and the pair record
    auto sample = [&](int count) {
        const bool on = lane < (uint32_t)count;
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(tally + PE_PT_N_PAIRS, (unsigned long long)count);
        base = __shfl_sync(0xffffffffu, base, 0);
        if (on) {
            const int at = queued - count + lane;
            const uint32_t jq = Q.j[at];
            const int64_t hit = Q.step[at];
            const Photon p = ph[jq];
            const double k = (double)p.e;
            bool above;
            int ik;
            double wk;
            bh_sigma_of(t, sig, k, above, ik, wk);
            const double x = bh_sample_x(t, cdf, k, ik, wk, uni53(w64(Q.z[at], Q.w[at])));
            const double ep = x * k;
            PairRec q;
            q.x = (float)photon_pos(c, p.kx, p.x, p.step, hit);
            q.y = (float)(two_d ? photon_pos(c, p.ky, p.y, p.step, hit) : 0.0);
            q.e_minus = (float)(k - ep);
            q.e_plus = (float)ep;
            q.kx = p.kx; q.ky = p.ky; q.kz = p.kz;
            q.step = (uint32_t)hit;
            q.photon = jq;
            q.id_mech = p.id_mech;
            fx_acc(e_pairs, fx_of(k));
            fx_acc(e_pos, fx_of(ep));
            if (base + lane < (unsigned long long)cap) out[base + lane] = q;
        }
        queued -= count;
        __syncwarp();
    };
    const int64_t stride = (int64_t)gridDim.x * (kPairThreads / 32) * per_round;
    // warp-uniform rounds of per_round <= 32 photons, so that every lane reaches the votes
    for (int64_t base = ((int64_t)blockIdx.x * (kPairThreads / 32) + (threadIdx.x >> 5)) * per_round; base < n_ph;
         base += stride) {
        const int64_t j = base + lane;
        // lane's photon: the run [a, b] of steps inside the target and the threshold of the test
        Photon p{};
        int64_t a = 1, b = 0;
        uint64_t thr = 0;
        double lam = 0.0;                          // n_i sigma_BH c dt = -ln(1 - P)
        bool above = false;
        if (lane < (uint32_t)per_round && j < n_ph) {
            p = ph[j];
            const double k = (double)p.e;
            if (k > 2.0) {
                const double kx = p.kx, ky = p.ky, xe = p.x, ye = p.y;
                const int64_t ne = p.step;
                int ik;
                double wk;
                lam = c.K_br * bh_sigma_of(t, sig, k, above, ik, wk);
                if constexpr (!kFree) {
                    const double P = -expm1(-lam);
                    thr = P >= 1.0 ? 0xFFFFFFFFFFFFFFFFull : __double2ull_rz(P * 0x1.0p64);
                }
                // The steps with the photon inside the target form one run [a, b] (its position
                // is monotone in the step and the target convex): bound it with each face by the
                // position exactly as the step computes it, so the tests run on integers only.
                a = ne + 1;
                b = step_end - 1;
                auto clip = [&](double d, double e, double lo, double hi) {
                    if (a > b) return;
                    if (d == 0.0) {
                        const double v = photon_pos(c, d, e, ne, a);
                        if (!(v >= lo && v <= hi)) b = a - 1;
                        return;
                    }
                    const double in_face = d > 0.0 ? lo : hi, out_face = d > 0.0 ? hi : lo;
                    const float per_step = 1.0f / ((float)d * (float)c.dt);
                    // the entry face is reached (d > 0: pos >= lo; d < 0: pos <= hi) ...
                    auto entered = [&](int64_t m) {
                        const double v = photon_pos(c, d, e, ne, m);
                        return d > 0.0 ? v >= in_face : v <= in_face;
                    };
                    // ... and the exit face passed
                    auto gone = [&](int64_t m) {
                        const double v = photon_pos(c, d, e, ne, m);
                        return !(d > 0.0 ? v <= out_face : v >= out_face);
                    };
                    if (!entered(b)) { b = a - 1; return; }
                    if (!entered(a)) a = first_past(a, b, ne, ceilf((float)(in_face - e) * per_step), entered);
                    if (gone(a)) { b = a - 1; return; }
                    if (gone(b)) b = first_past(a, b, ne, floorf((float)(out_face - e) * per_step) + 1.0f, gone) - 1;
                };
                clip(kx, xe, c.x0, c.x1);
                if (two_d) clip(ky, ye, -c.yh, c.yh);
            }
        }
        const unsigned entered_mask = __ballot_sync(0xffffffffu, a <= b);
        n_entered += __popc(entered_mask);
        n_above += __popc(__ballot_sync(0xffffffffu, a <= b && above));
        bool conv = false;                          // the lane's photon converts: at step `hit`, share from (hz, hw)
        uint32_t hit = 0, hz = 0, hw = 0;
        if constexpr (kFree) {
            // the trials of the crossing all have probability P = 1 - exp(-lam): the number of
            // failures before the first success is geometric, floor(-ln U / lam); one draw per photon
            if (a <= b && lam > 0.0) {
                const uint4 w = philox4x32_10(make_uint4(p.id_mech, r.run_id, (uint32_t)a, kPurBHFree + p.step),
                                              r.seed_lo, r.seed_hi);
                ++tests;
                const double jf = floor(-log(uni53(w64(w.x, w.y))) / lam);
                conv = jf <= (double)(b - a);
                if (conv) {
                    hit = (uint32_t)(a + (int64_t)jf);
                    hz = w.z;
                    hw = w.w;
                }
            }
        } else {
            // The warp takes the tests of each photon of the round in turn, 64 steps at a time
            // (lane l tests steps m0 + l and m0 + 32 + l); the conversion is at the first step whose draw passes.
            for (unsigned left = entered_mask; left; left &= left - 1u) {
                const int src = __ffs(left) - 1;
                const uint32_t as = __shfl_sync(0xffffffffu, (uint32_t)a, src);
                const uint32_t last = __shfl_sync(0xffffffffu, (uint32_t)(b - a), src);   // the run's last step - as
                const uint32_t idm = __shfl_sync(0xffffffffu, p.id_mech, src);
                const uint32_t pur = kPurBH + __shfl_sync(0xffffffffu, p.step, src);
                const uint64_t th = __shfl_sync(0xffffffffu, thr, src);
                const uint32_t th_hi = (uint32_t)(th >> 32);
                bool found = false;
                uint32_t at = last;
                for (uint32_t o = 0;; o += 64) {
                    const uint32_t o1 = o + lane, o2 = o1 + 32, rest = last - o;      // steps after as + o
                    const uint32_t y1 = philox4x32_10(make_uint4(idm, r.run_id, as + o1, pur), r.seed_lo, r.seed_hi).y;
                    const uint32_t y2 = philox4x32_10(make_uint4(idm, r.run_id, as + o2, pur), r.seed_lo, r.seed_hi).y;
                    const bool c1 = lane <= rest && y1 <= th_hi, c2 = lane + 32 <= rest && y2 <= th_hi;
                    if (__any_sync(0xffffffffu, c1 || c2)) {
                        uint32_t id2 = idm;
                        asm volatile("" : "+r"(id2));   // the whole draws are formed here, not carried from above
#pragma unroll
                        for (int half = 0; half < 2; ++half) {
                            if (found) continue;
                            const uint32_t oh = half ? o2 : o1;
                            const uint4 w = philox4x32_10(make_uint4(id2, r.run_id, as + oh, pur), r.seed_lo, r.seed_hi);
                            const unsigned bal = __ballot_sync(0xffffffffu, (half ? c2 : c1) && w64(w.x, w.y) < th);
                            if (bal) {
                                const int first = __ffs(bal) - 1;
                                at = o + 32 * half + first;
                                const uint32_t z = __shfl_sync(0xffffffffu, w.z, first);
                                const uint32_t v = __shfl_sync(0xffffffffu, w.w, first);
                                if (lane == (uint32_t)src) { hz = z; hw = v; }
                                found = true;
                            }
                        }
                    }
                    if (found || rest < 64) break;
                }
                if (lane == (uint32_t)src) {
                    tests += (unsigned long long)at + 1;
                    conv = found;
                    hit = as + at;
                }
            }
        }
        const unsigned mask = __ballot_sync(0xffffffffu, conv);
        if (mask) {
            if (conv) {
                const int at = queued + __popc(mask & ((1u << lane) - 1u));
                Q.j[at] = (uint32_t)j;
                Q.step[at] = hit;
                Q.z[at] = hz;
                Q.w[at] = hw;
            }
            queued += __popc(mask);
            __syncwarp();
            if (queued >= 32) sample(32);
        }
    }
    if (queued) sample(queued);
    for (int o = 16; o > 0; o >>= 1) tests += __shfl_xor_sync(0xffffffffu, tests, o);
    e_pairs = warp_sum(e_pairs);
    e_pos = warp_sum(e_pos);
    if (lane == 0) {
        if (n_entered) atomicAdd(tally + PE_PT_N_ENTERED, n_entered);
        if (n_above) atomicAdd(tally + PE_PT_N_K_ABOVE, n_above);
        if (tests) atomicAdd(tally + PE_PT_N_TESTS, tests);
        fx_add_words(tally + PE_PT_E_PAIRS, e_pairs);
        fx_add_words(tally + PE_PT_E_POSITRONS, e_pos);
    }
}

}  // namespace

void launch_pair_transport(const TablesDev& t, const RunDev& r, const void* photons, int64_t n_photons,
                           int64_t step_end, void* pairs, int64_t capacity, unsigned long long* tally, int method,
                           cudaStream_t s) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    constexpr int kWarps = kPairThreads / 32;
    if (method == PE_PAIR_FREE_PATH) {
        // one draw a photon, FP64 work at a price per warp: full warps
        const int64_t blocks = (n_photons + kPairThreads - 1) / kPairThreads;
        const int grid = (int)(blocks < (int64_t)sms * 8 ? (blocks > 0 ? blocks : 1) : (int64_t)sms * 8);
        k_pair_transport<true><<<grid, kPairThreads, 0, s>>>(t, r, static_cast<const Photon*>(photons), n_photons,
                                                             step_end, 32, static_cast<PairRec*>(pairs), capacity, tally);
    } else {
        // a warp goes through its photons' tests one photon after the other: few photons are spread over the resident
        // warps (3000 took 214 us as 94 warps of 32, now 185), many go in rounds of 32 (16 or 8 cost more FP64 set-up
        // than they even out: 3e6 in 7.0, 7.1 and 7.4 ms)
        const int64_t warps = (int64_t)sms * PE_PAIR_MIN_CTAS_SM * kWarps;
        const int64_t spread = (n_photons + warps - 1) / warps;
        const int per_round = (int)(spread < 32 ? spread : 32);
        const int64_t need = ((n_photons + per_round - 1) / per_round + kWarps - 1) / kWarps;
        const int grid = (int)(need < (int64_t)sms * 256 ? need : (int64_t)sms * 256);
        k_pair_transport<false><<<grid, kPairThreads, 0, s>>>(t, r, static_cast<const Photon*>(photons), n_photons,
                                                              step_end, per_round, static_cast<PairRec*>(pairs),
                                                              capacity, tally);
    }
}

}  // namespace pe
