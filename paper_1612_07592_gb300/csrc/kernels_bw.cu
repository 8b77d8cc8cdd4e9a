// kernels_bw.cu -- Breit-Wheeler conversion of photon records in the run's prescribed fields.
//
// Sec. 1 names pair production by a photon in the laser field; its rate is taken, like the
// NCS module's (Sec. 2.2), as that of a locally constant crossed field: a photon of energy k
// (m c^2) with quantum parameter chi makes pairs at W = alpha E_S T(chi) / k per unit time
// (1/omega_L).  Each photon record moves at c along its direction from its emission point;
// at step m (n_e < m < step_end) it is at x_e + k^ (m - n_e) c dt, the run's fields there at
// t = m dt give chi, and an optical depth tau_0 = -ln U falls by W dt per step; at the first
// step with tau <= 0 the photon converts, the positron's share x from the tabulated CDF.
//
// One thread per photon, with the step loop flattened: every pass of the loop takes one
// step of each lane's current photon, and a lane whose photon is done (converted, at
// step_end, or out of reach of every pulse for good) takes its next photon, so the lanes of
// a warp stay busy whatever the spread of path lengths.  The steps before the first pulse reaches a photon are
// counted in one go.  A pulse is out of reach of a photon
// when it is behind it -- its fields vanish identically once its phase t - x (for the
// reflected wave t + x - 2 x_m) is past the pulse's end, and both phases only grow along a
// photon's path -- or when it can never give chi above the table: a plane wave gives
// chi = (k -+ k_x) |E| / E_S exactly (- for the incident pulse, + for its mirror image) with
// |E| <= r a0 sqrt(1 + k_env^2) (Cauchy-Schwarz on g' sin + g cos), so with a factor 2 of
// margin the bound below chi_min means T = 0 at every step (photons co-moving with the
// incident pulse, for instance).  From then on chi < chi_min, T = 0 and the
// optical depth stays, so the photon stops with its remaining steps counted as taken (the
// tally equals stepping them).
//
// FP64 runs step in double (parity with the oracle: the same pair list).  FP32 runs step in
// float -- positions, fields, chi and T -- with the optical depth as a compensated float
// pair, tau_0 drawn in float-pair arithmetic; the once-per-conversion sampling of x runs in
// double in both.
#include "kernels.cuh"

namespace pe {
namespace {

constexpr uint32_t kPurBWTau = 0x60000000u;   // tau_0: counter (id_mech, run id, n_e, kPurBWTau + n_e)
constexpr uint32_t kPurBWX = 0x70000000u;     // x at conversion step m: (id_mech, run id, m, kPurBWX + n_e)

// T(chi): 0 below the table (flag -1), the last node above (flag 1), else L linear in ln chi
__device__ __forceinline__ double bw_T(const BwDev& b, double chi, int& flag) {
    if (!(chi >= b.chi_min)) { flag = -1; return 0.0; }
    double tp = (log(chi) - b.ln_chi_min) * b.inv_dln_chi;
    if (tp >= (double)(b.n_chi - 1)) { flag = 1; return b.T_last; }
    flag = 0;
    if (tp < 0.0) tp = 0.0;
    int i = (int)floor(tp);
    if (i > b.n_chi - 2) i = b.n_chi - 2;
    const double w = tp - (double)i;
    i = dbg_idx(b.dbg, i, b.n_chi - 1);
    return exp((1.0 - w) * b.L64[i] + w * b.L64[i + 1] - 8.0 / (3.0 * chi));
}
__device__ __forceinline__ float bw_T(const BwDev& b, float chi, int& flag) {
    if (!(chi >= b.fchi_min)) { flag = -1; return 0.0f; }
    const float tp = (__logf(chi) - b.fln_chi_min) * b.finv_dln_chi;
    if (tp >= b.f_last) { flag = 1; return b.fT_last; }
    flag = 0;
    // row by the magic-number split (no int/float conversion: GB300 runs those on its FP64 pipe)
    int i;
    float w;
    split_pos(fmaxf(tp, 0.0f), i, w);
    i = dbg_idx(b.dbg, i, b.n_chi - 1);
    // T below ~1e-38 (chi below ~0.03) underflows to 0: a rate 1e-36 times the unit
    return __expf((1.0f - w) * b.L32[i] + w * b.L32[i + 1] - 8.0f / (3.0f * chi));
}

// positron share x at uniform R: the CDF rows interpolated in ln chi (chi clamped to the
// table), inverted linearly in s between the nodes, x = (1 - cos(pi s)) / 2
__device__ __forceinline__ double bw_sample_x(const BwDev& b, double chi, double R) {
    if (!(chi >= b.chi_min)) chi = b.chi_min;
    const double tp = (log(chi) - b.ln_chi_min) * b.inv_dln_chi;
    int i;
    double w;
    if (tp >= (double)(b.n_chi - 1)) { i = b.n_chi - 2; w = 1.0; }
    else if (!(tp >= 0.0)) { i = 0; w = 0.0; }
    else { i = min((int)floor(tp), b.n_chi - 2); w = tp - (double)i; }
    i = dbg_idx(b.dbg, i, b.n_chi - 1);
    const double* ra = b.cdf64 + (size_t)i * b.n_x;
    int j;
    const double fr = invert_rows<double>(ra, ra + b.n_x, w, b.n_x, R, j);
    double s;
    if (j < 0) s = 0.0;
    else if (j >= b.n_x - 1) s = 1.0;
    else s = ((double)j + fr) / (double)(b.n_x - 1);
    return 0.5 * (1.0 - cos(kPi * s));
}

// the photon's chi: the electron's eta with u -> kvec and gamma -> |kvec|, in the same
// cancellation-safe arrangement (|kvec| - k_x = k_perp^2 / (|kvec| + k_x) for k_x > 0);
// kk = |kvec| and gm depend on the photon only
template <typename R>
__device__ __forceinline__ R chi_photon(const R kv[3], R gm, const R E[3], const R B[3], R inv_ES) {
    const R d0 = B[0], d1 = B[1] + E[2], d2 = B[2] - E[1];
    const R V0 = gm * E[0] + (kv[1] * d2 - kv[2] * d1);
    const R V1 = gm * E[1] + (kv[2] * d0 - kv[0] * d2);
    const R V2 = gm * E[2] + (kv[0] * d1 - kv[1] * d0);
    const R kE = kv[0] * E[0] + kv[1] * E[1] + kv[2] * E[2];
    const R q = V0 * V0 + V1 * V1 + V2 * V2 + (R)2 * V0 * kE;
    return q > (R)0 ? m_sqrt(q) * inv_ES : (R)0;
}

// optical depth: double, or a compensated float pair
template <typename R> struct Depth;
template <> struct Depth<double> {
    double v;
    __device__ void set(double t) { v = t; }
    __device__ void sub(double d) { v -= d; }
    __device__ bool crossed() const { return v <= 0.0; }
};
template <> struct Depth<float> {
    float v, lo;
    __device__ void set(double t) { v = (float)t; lo = (float)(t - (double)v); }
    __device__ void set(float t) { v = t; lo = 0.0f; }
    __device__ void sub(float d) {       // TwoSum: v + lo stays exact to ~2^-48
        const float s = v - d, bb = s - v;
        lo += (v - (s - bb)) + (-d - bb);
        v = s;
    }
    __device__ bool crossed() const { return v + lo <= 0.0f; }
};

// position at step m: e + d ((m - n_e) dt) with sf = m - n_e held as a floating-point counter
// (advanced by exact + 1, so no integer-to-float conversion per step: GB300 runs conversions on
// its narrow FP64 pipe); one rounding for the product and one for the FMA
__device__ __forceinline__ double bw_pos(const StepC<double>& c, double d, double e, double sf) {
    return __fma_rn(d, __dmul_rn(sf, c.dt), e);
}
__device__ __forceinline__ float bw_pos(const StepC<float>& c, float d, float e, float sf) {
    return fmaf(d, sf * c.dt, e);
}

// Resident CTAs of 256 threads per SM the registers are sized for (FP32 reflected kind, 4e5 / 3e6 photons of 2000
// steps, two thirds converted): 2 CTAs 2.6 / 14.3 ms, 3 2.57 / 13.2, 4 2.66 / 14.0, 5 3.05, 6 3.42
#ifndef PE_BW_MIN_CTAS
#define PE_BW_MIN_CTAS 3
#endif

constexpr int kBwThreads = 256;
// conversions of a warp that wait for their sampling: photon, step, chi and position (fewer than 32 left by the last
// pass and at most 32 more)
template <typename R>
struct Conversions {
    uint32_t j[64], m[64];
    R chi[64], x[64], y[64];
    ulonglong2 e_pairs, e_pos;          // the warp's energy sums, its lane 0's
};

// steps a photon can be advanced at once before a pulse whose phase is `phi` at its present step and grows by `rate`
// a step: the fields vanish identically while the phase is <= 0 (0.05 of margin covers the rounding of the FP32 phase),
// so chi and T are 0 there
template <typename R>
__device__ __forceinline__ R free_steps(R phi, R rate) {
    const R d = ((R)-0.05 - phi) / rate - (R)1;
    return rate > (R)1e-6 && d > (R)0 ? m_floor(d) : (R)0;
}

// One warp-wide loop: each pass, the lanes without a photon take their next one from the CTA's share (a counter in
// shared memory: lanes whose photons end early take more of them), and every lane with one takes a step of it.  The
// votes hold the lanes of a warp together; without them the lanes that had left one another in the search for a
// photon never met again, and each pass ran for 10 of 32 lanes.  A conversion's sampling is FP64, on GB300's narrow
// pipe, and was done by the one lane that had it: 35 of 35 M FP64 warp instructions, half of the time; queued and done
// 32 at a time it is 2.4 M.  Measured, 4e5 photons x 2000 steps in the reflected a0 = 400 pulse, two thirds of them
// converted: 5.5 ms; 4.0 with the votes and the steps ahead of the pulse counted in one go; 2.57 with the queue.
// Records lie in order of emission, so the shares are interleaved: 9.6e6 photons of a reflected job 46.9 ms at the start,
// 41.8 with shares in one piece, 34.1 so. What is left is issue (0.8 a cycle), a third of it at 4e5 photons for lanes
// that wait for the last photons of a CTA's share.
template <typename R, int G>
__global__ void __launch_bounds__(kBwThreads, PE_BW_MIN_CTAS) k_bw_transport(BwDev bw, RunDevT<R> r, const Photon* ph,
                                                                     int64_t n_ph, int64_t step_end,
                                                                     PairRec* out, int64_t cap,
                                                                     unsigned long long* tally) {
    const StepC<R>& c = r.c;
    const bool two_d = r.geometry == PE_GAUSS_2D;
    constexpr bool kLeave = G != FK_CONST;                 // a prescribed pulse: fields vanish before and behind it
    constexpr bool kRefl = G == FK_REFL_LP || G == FK_REFL_CP;
    constexpr bool kPlane = G == FK_PLANE_LP || G == FK_PLANE_CP || kRefl;   // chi bounded as for a plane wave
    // 2 E_max / E_S of the incident pulse: twice the bound on chi / (k - k_x)
    const R reach = (R)2 * c.a0 * m_sqrt((R)1 + c.k_env * c.k_env) * c.inv_ES;
    const R chi_min = sizeof(R) == 8 ? (R)bw.chi_min : (R)bw.fchi_min;
    const R L_end = (R)2 * c.phi_r + c.phi_f + (sizeof(R) == 8 ? (R)1e-6 : (R)1e-3);   // pulse end + margin
    const int lane = threadIdx.x & 31;
    __shared__ unsigned int s_taken;                       // photons of the CTA's share handed out
    __shared__ Conversions<R> s_conv[kBwThreads / 32];
    if (threadIdx.x == 0) s_taken = 0;
    __syncthreads();
    Conversions<R>& Q = s_conv[threadIdx.x >> 5];
    int queued = 0;                                        // conversions in Q (the same on every lane)
    if (lane == 0) Q.e_pairs = Q.e_pos = make_ulonglong2(0, 0);
    // the last `count` queued conversions, one to a lane: the positron's share of k, the pair record and the sums
    auto sample = [&](int count) {
        const bool on = lane < count;
        PairRec q;
        double kd = 0.0, ep = 0.0;
        if (on) {
            const int at = queued - count + lane;
            const uint32_t jq = Q.j[at], mq = Q.m[at];
            const Photon p = ph[jq];
            const uint4 w = philox4x32_10(make_uint4(p.id_mech, r.run_id, mq, kPurBWX + p.step), r.seed_lo, r.seed_hi);
            kd = (double)p.e;
            const double x = bw_sample_x(bw, (double)Q.chi[at], uni53(w64(w.x, w.y)));
            ep = x * kd;
            q.x = (float)Q.x[at];
            q.y = (float)(two_d ? Q.y[at] : (R)0);
            q.e_minus = (float)(kd - ep);
            q.e_plus = (float)ep;
            q.kx = p.kx; q.ky = p.ky; q.kz = p.kz;
            q.step = mq;
            q.photon = jq;
            q.id_mech = p.id_mech;
        }
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(tally + PE_PT_N_PAIRS, (unsigned long long)count);
        base = __shfl_sync(0xffffffffu, base, 0);
        if (on && base + lane < (unsigned long long)cap) out[base + lane] = q;
        const ulonglong2 a = warp_sum(fx_of(kd)), b = warp_sum(fx_of(ep));
        if (lane == 0) {
            fx_acc(Q.e_pairs, a);
            fx_acc(Q.e_pos, b);
        }
        queued -= count;
        __syncwarp();
    };
    unsigned long long n_followed = 0, n_tests = 0, n_above = 0;
    int64_t j = 0;
    bool have = false, more = true;                // a photon in hand; the share may hold another
    Photon p{};
    R k = 0, kv[3] = {0, 0, 0}, gm = 0, kx = 0, ky = 0, xe = 0, ye = 0, kdt = 0;
    int64_t ne = 0, m = 0;
    R sf = 0, mf = 0;                              // m - n_e and m as exact floating-point counters
    bool inc_never = false, ref_never = true;     // a pulse can never raise chi above the table
    Depth<R> tau;
    tau.set(1.0);
    while (true) {
        const unsigned need = __ballot_sync(0xffffffffu, !have && more);
        if (need) {
            unsigned int first = 0;
            if (lane == __ffs(need) - 1) first = atomicAdd(&s_taken, (unsigned int)__popc(need));
            first = __shfl_sync(0xffffffffu, first, __ffs(need) - 1);
            if (!have && more) {
                // a photon to step has k > 2 m c^2, a step left before step_end, and a pulse that can raise its
                // chi into the table; the others are only counted (no draw)
                const unsigned int q = first + __popc(need & ((1u << lane) - 1u));
                // photon q of the CTA: blocks of 32, every gridDim.x-th (records are in order of emission)
                j = ((int64_t)(q >> 5) * gridDim.x + blockIdx.x) * 32 + (q & 31u);
                more = j < n_ph;
                if (more) p = ph[j];
                if (more && p.e > 2.0f) {                  // the same decision as (double) k > 2
                    ++n_followed;
                    ne = (int64_t)p.step;
                    m = ne + 1;
                    k = (R)p.e;
                    kx = (R)p.kx; ky = (R)p.ky; xe = (R)p.x; ye = (R)p.y;
                    kv[0] = k * kx; kv[1] = k * ky; kv[2] = k * (R)p.kz;
                    const R kk = m_sqrt(kv[0] * kv[0] + kv[1] * kv[1] + kv[2] * kv[2]);
                    gm = (kv[0] > (R)0) ? (kv[1] * kv[1] + kv[2] * kv[2]) / (kk + kv[0]) : kk - kv[0];
                    if (kPlane) {
                        // k - k_x is gm (formed without cancellation); k + k_x likewise for backward photons
                        const R gp = (kv[0] < (R)0) ? (kv[1] * kv[1] + kv[2] * kv[2]) / (kk - kv[0]) : kk + kv[0];
                        inc_never = gm * reach < chi_min;
                        ref_never = !kRefl || gp * c.refl_r * reach < chi_min;
                    }
                    have = m < step_end;
                    if (kPlane && inc_never && ref_never) {  // no pulse can convert it: every step counted, none taken
                        n_tests += (unsigned long long)(have ? step_end - m : 0);
                        have = false;
                    }
                }
                if (have) {
                    const uint4 w = philox4x32_10(make_uint4(p.id_mech, r.run_id, (uint32_t)ne, kPurBWTau + p.step),
                                                  r.seed_lo, r.seed_hi);
                    kdt = c.bw_coef / k;
                    sf = (R)1;
                    if constexpr (sizeof(R) == 8) {
                        tau.set(-log(uni53(w64(w.x, w.y))));
                        mf = (R)m;
                    } else {
                        // -ln U from the same 53 bits in float-pair arithmetic, and the step as a float
                        // without a conversion instruction (m < 8192): no FP64-pipe work per photon
                        tau.set(tau_draw_f32(w.x, w.y));
                        mf = int_to_float_small((int)m);
                    }
                    if constexpr (kLeave) {
                        // the steps before the first pulse that matters reaches it are counted, not taken
                        const R px = bw_pos(c, kx, xe, sf);
                        R skip = inc_never && kPlane ? (R)(step_end - m)
                                                     : free_steps<R>(phase(c, mf, px, (R)0), c.dt * ((R)1 - kx));
                        if (kRefl && !ref_never) {
                            const R s2 = free_steps<R>(phase_refl(c, mf, px, (R)0), c.dt * ((R)1 + kx));
                            skip = s2 < skip ? s2 : skip;
                        }
                        if (skip >= (R)(step_end - m)) {
                            n_tests += (unsigned long long)(step_end - m);
                            have = false;
                        } else {
                            n_tests += (unsigned long long)skip;
                            m += (int64_t)skip;
                            sf += skip;
                            mf += skip;
                        }
                    }
                }
            }
        }
        if (!__any_sync(0xffffffffu, have)) {
            if (!__any_sync(0xffffffffu, more)) break;
            continue;
        }
        bool conv = false;
        R chi = 0, px = 0, py = 0;
        if (have) {
            // step m of the lane's photon
            px = bw_pos(c, kx, xe, sf);
            py = bw_pos(c, ky, ye, sf);
            R E[3], B[3];
            fields<R, G>(r, px, (R)0, py, mf, E, B);
            chi = chi_photon<R>(kv, gm, E, B, c.inv_ES);
            int fl;
            const R T = bw_T(bw, chi, fl);
            ++n_tests;
            n_above += fl == 1;
            if constexpr (sizeof(R) == 8) tau.sub(c.bw_coef * T / k);    // (alpha E_S dt) T / k, the oracle's order
            else tau.sub(kdt * T);
            if (tau.crossed()) {
                conv = true;
                have = false;
            } else {
                ++m;
                if (m >= step_end) {
                    have = false;
                } else if (kLeave) {
                    // every pulse behind the photon for good, or never strong enough for it: the
                    // remaining steps see chi below the table
                    bool gone = inc_never || phase(c, mf, px, (R)0) > L_end;
                    if (kRefl) gone = gone && (ref_never || phase_refl(c, mf, px, (R)0) > L_end);
                    if (gone) {
                        n_tests += (unsigned long long)(step_end - m);
                        have = false;
                    }
                }
                sf += (R)1;
                mf += (R)1;
            }
        }
        // A conversion ends its photon, so nothing of this pass waits for it: its sampling (FP64, a binary search)
        // is queued and done 32 at a time, on full warps
        const unsigned mask = __ballot_sync(0xffffffffu, conv);
        if (mask) {
            if (conv) {
                const int at = queued + __popc(mask & ((1u << lane) - 1u));
                Q.j[at] = (uint32_t)j;
                Q.m[at] = (uint32_t)m;
                Q.chi[at] = chi;
                Q.x[at] = px;
                Q.y[at] = py;
            }
            queued += __popc(mask);
            __syncwarp();
            if (queued >= 32) sample(32);
        }
    }
    if (queued) sample(queued);
    if (lane == 0) {
        fx_add_words(tally + PE_PT_E_PAIRS, Q.e_pairs);
        fx_add_words(tally + PE_PT_E_POSITRONS, Q.e_pos);
    }
    // counters: one warp sum each
    for (int o = 16; o > 0; o >>= 1) {
        n_followed += __shfl_xor_sync(0xffffffffu, n_followed, o);
        n_tests += __shfl_xor_sync(0xffffffffu, n_tests, o);
        n_above += __shfl_xor_sync(0xffffffffu, n_above, o);
    }
    if (lane == 0) {
        if (n_followed) atomicAdd(tally + PE_PT_N_ENTERED, n_followed);
        if (n_tests) atomicAdd(tally + PE_PT_N_TESTS, n_tests);
        if (n_above) atomicAdd(tally + PE_PT_N_K_ABOVE, n_above);
    }
}

template <typename R, int G>
void launch_kind(const BwDev& b, const RunDevT<R>& r, const void* photons, int64_t n, int64_t step_end, void* pairs,
                 int64_t cap, unsigned long long* tally, cudaStream_t s) {
    int dev = 0, sms = 0, occ = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_bw_transport<R, G>, kBwThreads, 0) != cudaSuccess || occ < 1)
        occ = 1;
    // the resident CTAs share the photons by blocks of 32; a few photons are spread a block to a CTA
    const int64_t blocks = (n + 31) / 32;
    const int grid = (int)(blocks < (int64_t)sms * occ ? (blocks > 0 ? blocks : 1) : (int64_t)sms * occ);
    k_bw_transport<R, G><<<grid, kBwThreads, 0, s>>>(b, r, static_cast<const Photon*>(photons), n, step_end,
                                              static_cast<PairRec*>(pairs), cap, tally);
}

}  // namespace

void launch_bw_transport(const BwDev& b, const RunDev& r, int precision, const void* photons, int64_t n_photons,
                         int64_t step_end, void* pairs, int64_t capacity, unsigned long long* tally, cudaStream_t s) {
    with_field_kind(r.fk, [&](auto g) {
        constexpr int G = decltype(g)::value;
        if (precision == PE_F32)
            launch_kind<float, G>(b, to_float(r), photons, n_photons, step_end, pairs, capacity, tally, s);
        else
            launch_kind<double, G>(b, r, photons, n_photons, step_end, pairs, capacity, tally, s);
    });
}

}  // namespace pe
