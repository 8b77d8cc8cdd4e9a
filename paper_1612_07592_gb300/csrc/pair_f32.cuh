// pair_f32.cuh -- the FP32 step of every prescribed-field kind (the 1D plane wave, its
// reflection, the 2D focus, constant fields) with two electrons per thread.  Blackwell issues paired single-precision arithmetic
// (FFMA2/FADD2/FMUL2: two FP32 results per instruction), so the common path of
// the step -- fields, Boris push, eta, rate lookup, optical depth, the
// bremsstrahlung probability of Eq. 4, position -- runs on float2 values holding
// the two electrons, with the operations of the one-electron float step in the
// same order (where a form differs -- a Newton-refined reciprocal for a
// division, a series for 1 - e^{-x} at small x, Fast2Sum for the optical depth
// -- the comment at the spot says why it holds).  The draws of the
// bremsstrahlung test, emissions and the absorbing boundary leave the packed
// path and run per electron.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "kernels.cuh"

namespace pe {

// ---- paired arithmetic -----------------------------------------------------------
__device__ __forceinline__ float2 P2(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// a - b with one paired instruction: (-1) b + a
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, P2(-1.0f), a); }
__device__ __forceinline__ float2 neg2(float2 a) { return __fmul2_rn(a, P2(-1.0f)); }
// per-electron operations (no paired form)
// the hardware's approximate square root, written out (the translation unit that instantiates the
// paired kernels rounds its own divisions and square roots as IEEE operations)
__device__ __forceinline__ float2 sqrt2(float2 a) {
    float2 r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(a.x));
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(a.y));
    return r;
}
// Reciprocal square root of a >= 1 (every use: 1 + u^2, 1 + a^2), square root (above) and base-2 logarithm in their
// flush-to-zero forms: the same results for normal operands without the scaling that subnormal ones need, some three
// instructions each (an eta, or its square, below 2^-126 counts as 0).  1D job 19.5 -> 18.4 ms, 2D focus 16.3 -> 15.4,
// bunch 8.2 -> 7.7; same bits.
__device__ __forceinline__ float2 rsqrt2(float2 a) {
    float2 r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(a.x));
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(a.y));
    return r;
}
// -1/d for d >= 1 (both uses below): the hardware reciprocal estimate of -d refined by one
// Newton-Raphson step, r' = r + r (1 + d r), which squares its relative error (about 1 ulp after
// it); it replaces an IEEE division, whose special-case check and branch cost more than the
// estimate and two FMAs.  The sign is taken by the estimate's operand (free) rather than by a
// paired multiply by -1 (a whole instruction: paired arithmetic has no negated operands), and the
// callers absorb it into a constant factor.
__device__ __forceinline__ float2 nrcp2(float2 d) {
    float2 r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(-d.x));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(-d.y));
    const float2 e = fma2(d, r, P2(1.0f));
    return fma2(r, e, r);
}
__device__ __forceinline__ float2 log2v(float2 a) {
    float2 r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(a.x));
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(a.y));
    return r;
}
__device__ __forceinline__ float2 sel2(bool cx, bool cy, float2 a, float2 b) {
    return make_float2(cx ? a.x : b.x, cy ? a.y : b.y);
}
__device__ __forceinline__ float2 clamp2(float2 a, float lo, float hi) {
    return make_float2(fminf(fmaxf(a.x, lo), hi), fminf(fmaxf(a.y, lo), hi));
}
__device__ __forceinline__ float comp(float2 a, int k) { return k ? a.y : a.x; }
__device__ __forceinline__ void set_comp(float2& a, int k, float v) { if (k) a.y = v; else a.x = v; }

// TwoSum on pairs: (s, e) with s + e = a + b exactly
__device__ __forceinline__ void two_sum2(float2 a, float2 b, float2& s, float2& e) {
    s = add2(a, b);
    float2 bb = sub2(s, a);
    e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
}

// 1 - e^{-x} by the Taylor series x (1 - x/2 + x^2/6 - x^3/24) (for x < 2^-5), paired; the
// same operations in the same order as one_minus_exp_neg_f32
__device__ __forceinline__ float2 brems_series2(float2 x) {
    return mul2(x, fma2(x, fma2(x, fma2(x, P2(-1.0f / 24.0f), P2(1.0f / 6.0f)), P2(-0.5f)), P2(1.0f)));
}

// ramp sine/cosine of the envelope (0 <= v <= pi/2), paired: the hardware units
__device__ __forceinline__ void ramp_sincos2(float2 v, float2& s_out, float2& c_out) {
    s_out = make_float2(__sinf(v.x), __sinf(v.y));
    c_out = make_float2(__cosf(v.x), __cosf(v.y));
}

// sine and cosine of the carrier phase, paired: Cody-Waite reduction (1980) by 2 pi with a
// two-part constant to |r| <= pi, then the hardware sine and cosine (absolute error below
// 2^-21.4 on [-pi, pi]; 20 instructions per pair fewer than the polynomial form)
__device__ __forceinline__ void sincos2(float2 v, float2& s_out, float2& c_out) {
    const float kMagic = 0x1.8p23f;
    const float2 t = fma2(v, P2(0.159154943091895336f), P2(kMagic));    // 2 pi k + ..., k = rint(v / 2 pi)
    const float2 nk = sub2(P2(kMagic), t);                              // -k, exact
    float2 r = fma2(nk, P2(6.28318548202514648f), v);                   // 2 pi, nearest float
    r = fma2(nk, P2(-1.74845553e-7f), r);                               // 2 pi - its nearest float
    s_out = make_float2(__sinf(r.x), __sinf(r.y));
    c_out = make_float2(__cosf(r.x), __cosf(r.y));
}

// e^{-v} for v >= 0, paired: the hardware base-2 exponential of -v log2(e) (relative error a few
// ulp; underflows to 0)
__device__ __forceinline__ float2 exp_neg2(float2 v) {
    const float2 a = mul2(v, P2(-1.44269504088896341f));
    float2 r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(a.x));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(a.y));
    return r;
}

// Amplitude and Gouy phase of the 2D paraxial focus at a = (x - x_f) / z_R, without an
// arctangent: sqrt(w0 / w) e^{i atan(a) / 2} = (1 + i a)^{1/2} / |1 + i a|, and with
// n = |1 + i a| = sqrt(1 + a^2) the square root of 1 + i a is R + i I, R = sqrt((n + 1) / 2),
// I = a / (2 R) (the half-angle formulas; I written without the cancelling n - 1).  Returns
// Rn = R / n and In = I / n, and 1 / n^2 = w0^2 / w^2.
__device__ __forceinline__ void gouy2(float2 a, float2& Rn, float2& In, float2& inv_n2) {
    const float2 q1 = fma2(a, a, P2(1.0f));                    // n^2
    const float2 inv_n = rsqrt2(q1);
    inv_n2 = mul2(inv_n, inv_n);
    const float2 hh = fma2(mul2(q1, inv_n), P2(0.5f), P2(0.5f));   // (n + 1) / 2
    const float2 inv_r = rsqrt2(hh);
    Rn = mul2(mul2(hh, inv_r), inv_n);
    In = mul2(mul2(P2(0.5f), a), mul2(inv_r, inv_n));
}

// envelope g = sin^2(k psi) of a pulse at phase phi, psi the phase distance to the nearer end of
// the pulse, k psi clamped to [0, pi/2] (0 outside the pulse, pi/2 on the flat top); dg/dphi =
// +-k sin(2 k psi), + before the middle of the pulse and - after it (it vanishes on the flat top
// and outside).  envelope_arg2: k psi and the distance to the pulse's end.
__device__ __forceinline__ float2 envelope_arg2(const StepC<float>& c, float2 phi, float2& rem) {
    rem = sub2(P2(2.0f * c.phi_r + c.phi_f), phi);
    const float2 psi = make_float2(fminf(phi.x, rem.x), fminf(phi.y, rem.y));
    return clamp2(mul2(P2(c.k_env), psi), 0.0f, 1.57079632679489662f);
}
__device__ __forceinline__ void envelope2(const StepC<float>& c, float2 phi, float2 arg, float2 rem, float2& g,
                                          float2& dg) {
    float2 rs, rc;
    ramp_sincos2(arg, rs, rc);
    g = mul2(rs, rs);
    const float2 kts = mul2(P2(2.0f * c.k_env), mul2(rs, rc));
    const float2 side = sub2(rem, phi);
    dg = make_float2(copysignf(kts.x, side.x), copysignf(kts.y, side.y));
}

// What the run's flags are at compile time: nothing (read from the run), the paper's setup (NCS on, direct brems, no
// absorbing box), or brems alone (direct, no NCS, no box: the Sec. 2.2 bunch), so that the step carries no test of them
// and no code of a process that is off (the bunch, 5e5 electrons x 2000 steps: 7.7 ms with the flags read in each step
// and the push of zero fields, 5.7 without either).
enum { kFlagsRun = 0, kFlagsPaper = 1, kFlagsBrems = 2 };
template <int F>
__device__ __forceinline__ bool ncs_on(const RunDevT<float>& r) {
    return F == kFlagsPaper ? true : F == kFlagsBrems ? false : r.enable_ncs != 0;
}
template <int F>
__device__ __forceinline__ bool brems_on(const RunDevT<float>& r) { return F != kFlagsRun || r.enable_brems; }
template <int F>
__device__ __forceinline__ bool null_on(const RunDevT<float>& r) {
    return F == kFlagsRun && r.brems_method == PE_BREMS_NULL;
}
template <int F>
__device__ __forceinline__ bool box_on(const RunDevT<float>& r) { return F == kFlagsRun && r.box_enable; }

// two electrons; per-electron activity and optical-depth pairs.  The event fingerprints stay in memory: an
// emission adds to its electron's word there (add_events).
struct Pair {
    float2 x, x_lo, u0, u1, u2, tau, tau_lo;
    float2 y, y_lo;                     // 2D focus only (zero and unused in 1D)
    uint32_t wait[2];
    bool act[2];
};

__device__ __forceinline__ Particle<float> unpack(const Pair& Q, int k) {
    Particle<float> P;
    P.x = comp(Q.x, k); P.x_lo = comp(Q.x_lo, k);
    P.y = comp(Q.y, k); P.y_lo = comp(Q.y_lo, k);
    P.u[0] = comp(Q.u0, k); P.u[1] = comp(Q.u1, k); P.u[2] = comp(Q.u2, k);
    P.tau = comp(Q.tau, k); P.tau_lo = comp(Q.tau_lo, k);
    P.ev_cnt = P.ev_hash = 0;
    // a select, not Q.wait[k]: an index unknown at compile time (the emission loops) would move the
    // array to local memory
    P.wait = k ? Q.wait[1] : Q.wait[0];
    return P;
}
__device__ __forceinline__ void repack(Pair& Q, int k, const Particle<float>& P) {
    set_comp(Q.x, k, P.x); set_comp(Q.x_lo, k, P.x_lo);
    set_comp(Q.y, k, P.y); set_comp(Q.y_lo, k, P.y_lo);
    set_comp(Q.u0, k, P.u[0]); set_comp(Q.u1, k, P.u[1]); set_comp(Q.u2, k, P.u[2]);
    set_comp(Q.tau, k, P.tau); set_comp(Q.tau_lo, k, P.tau_lo);
    if (k) Q.wait[1] = P.wait; else Q.wait[0] = P.wait;
}
// The inactive halves of a pair take no further part (see push_pair); in registers only, after what is stored of them.
template <int G>
__device__ __forceinline__ void retire(Pair& Q) {
    if constexpr (G == FK_CONST) {
        if (!Q.act[0]) Q.u0.x = __int_as_float(0x7fc00000);
        if (!Q.act[1]) Q.u0.y = __int_as_float(0x7fc00000);
    }
}
// an emission's fingerprint into electron id's word (its thread alone has the electron)
__device__ __forceinline__ void add_events(const RunDevT<float>& r, uint32_t id, const Particle<float>& P) {
    if (!r.events) return;
    unsigned long long* w = r.events + (uint32_t)(id - r.id0);
    const unsigned long long e = *w;
    *w = ((unsigned long long)((uint32_t)(e >> 32) + P.ev_hash) << 32) | ((uint32_t)e + P.ev_cnt);
}
// state back to memory without the event word
__device__ __forceinline__ void store_one(const RunDevT<float>& r, int64_t i, const Particle<float>& P) {
    store_pos(r, i, P);
    ((float*)r.ux)[i] = P.u[0];
    ((float*)r.uy)[i] = P.u[1];
    ((float*)r.uz)[i] = P.u[2];
    store_tau(r, i, P);
    if (r.wait) r.wait[i] = P.wait;
}

// phase t^n - x of the pulse and t^n + x - 2 x_m of its mirror image at the pair's positions
__device__ __forceinline__ float2 phase2(const StepC<float>& c, float2 nf2, const Pair& Q) {
    return sub2(fma2(nf2, P2(c.dt_lo), sub2(mul2(nf2, P2(c.dt_hi)), Q.x)), Q.x_lo);
}
__device__ __forceinline__ float2 phase_refl2(const StepC<float>& c, float2 nf2, const Pair& Q) {
    return add2(add2(fma2(nf2, P2(c.dt_hi), P2(-c.xm2_hi)), Q.x), fma2(nf2, P2(c.dt_lo), sub2(Q.x_lo, P2(c.xm2_lo))));
}
// gamma and 1/gamma from one reciprocal square root
__device__ __forceinline__ void gamma_pair(const Pair& Q, float2& gamma, float2& inv_g) {
    const float2 g2 = fma2(Q.u2, Q.u2, fma2(Q.u1, Q.u1, fma2(Q.u0, Q.u0, P2(1.0f))));
    inv_g = rsqrt2(g2);
    gamma = mul2(g2, inv_g);
}
// no pulse at either electron (its envelope's argument is zero, or the electron is not there) and nothing to emit
template <int G>
__device__ __forceinline__ bool no_pulse(const StepC<float>& c, float nf, const Pair& Q) {
    float2 rem;
    float2 arg = envelope_arg2(c, phase2(c, P2(nf), Q), rem);
    if constexpr (G == FK_REFL_LP || G == FK_REFL_CP)
        arg = add2(arg, envelope_arg2(c, phase_refl2(c, P2(nf), Q), rem));
    const float2 tsum = add2(Q.tau, Q.tau_lo);
    return arg.x + arg.y == 0.0f && !(tsum.x <= 0.0f || tsum.y <= 0.0f);
}

// The first half of a step of two electrons: fields at (x^n, t^n), Boris push, gamma, and with NCS on eta, the
// rate and the optical depth.  Returns a bit per electron whose optical depth crossed zero (it emits).
// G = FK_PLANE_LP, FK_PLANE_CP: the 1D plane wave; FK_REFL_LP, FK_REFL_CP: the plane wave and its mirror
// image; FK_GAUSS_LP, FK_GAUSS_CP: the 2D paraxial focus; FK_CONST: constant fields.  An inactive half of
// the pair (a removed electron, or an empty slot past the end of the run) has x = NaN -- and u_x = NaN (retire) in
// constant fields, which do not depend on x -- so its momenta, gamma and optical depth are NaN from its first step on
// and its eta NaN or (where a maximum with 0 is taken) 0: the eta count, the optical depth's crossing and the target
// test are false for it without reading the activity flags.  Nothing of an inactive half is stored.
template <int G, int F>
__device__ __forceinline__ unsigned push_pair(const TablesDev& t, const RunDevT<float>& r, const float* h_tab,
                                              float nf, Pair& Q, float2& gamma, float2& inv_g, float2& eta,
                                              float2& n_above) {
    const StepC<float>& c = r.c;
    const TabC<float>& tc = t.cf;
    const float2 h = P2(0.5f * c.dt);
    // fields at (x^n, t^n): phase, envelope, carrier
    const float2 nf2 = P2(nf);
    const float2 phi = phase2(c, nf2, Q);
    constexpr bool kPlane = G == FK_PLANE_LP || G == FK_PLANE_CP;
    constexpr bool kRefl = G == FK_REFL_LP || G == FK_REFL_CP;
    constexpr bool kConst = G == FK_CONST;
    constexpr bool kCP = G == FK_PLANE_CP || G == FK_GAUSS_CP || G == FK_REFL_CP;
    if constexpr (kConst) {
        // the run's constant fields are zero: the push is the identity and eta is 0, so the optical depth stays (if it
        // is positive, as an emission leaves it); only gamma is formed
        if (r.no_field) {
            const float2 tsum = add2(Q.tau, Q.tau_lo);
            if (!(tsum.x <= 0.0f || tsum.y <= 0.0f)) {
                gamma_pair(Q, gamma, inv_g);
                return 0;
            }
        }
    }
    float2 g = P2(0.0f), dg = P2(0.0f), rem;
    if constexpr (!kConst) {
        const float2 arg = envelope_arg2(c, phi, rem);
        envelope2(c, phi, arg, rem, g, dg);
    }
    float2 by = P2(0.0f), bz = P2(0.0f);                // B_y, B_z of the reflected kinds
    const float2 ma0 = P2(-c.a0);
    float2 ey, ez = P2(0.0f), ex = P2(0.0f), bx = P2(0.0f);
    if constexpr (kPlane) {
    float2 st, ct;
    sincos2(phi, st, ct);
    ey = mul2(ma0, fma2(dg, st, mul2(g, ct)));                 // -a0 (g' sin + g cos)
    if (G == FK_PLANE_CP) ez = mul2(P2(c.a0), sub2(mul2(dg, ct), mul2(g, st)));   // a0 (g' cos - g sin)
    // Boris push with E = (0, ey, ez), B = (0, -ez, ey)
    const float2 mhey = mul2(P2(-0.5f * c.dt), ey);                    // -h E_y (the sign is exact)
    float2 um0 = Q.u0;
    float2 um1 = add2(Q.u1, mhey);
    float2 um2 = (G == FK_PLANE_CP) ? sub2(Q.u2, mul2(h, ez)) : Q.u2;
    float2 q = fma2(um2, um2, fma2(um1, um1, fma2(um0, um0, P2(1.0f))));
    float2 ig = rsqrt2(q);
    float2 t2 = mul2(mhey, ig);                                        // -h B_z / gamma
    if constexpr (G == FK_PLANE_CP) {
        float2 t1 = mul2(mul2(h, ez), ig);                             // -h B_y / gamma
        float2 f = mul2(P2(-2.0f), nrcp2(fma2(t2, t2, fma2(t1, t1, P2(1.0f)))));
        float2 s1 = mul2(f, t1), s2 = mul2(f, t2);
        float2 p0 = add2(um0, sub2(mul2(um1, t2), mul2(um2, t1)));
        float2 p1 = sub2(um1, mul2(um0, t2));
        float2 p2 = add2(um2, mul2(um0, t1));
        Q.u0 = add2(um0, sub2(mul2(p1, s2), mul2(p2, s1)));
        Q.u1 = add2(sub2(um1, mul2(p0, s2)), mhey);
        Q.u2 = sub2(add2(um2, mul2(p0, s1)), mul2(h, ez));
    } else {
        // LP: B = (0, 0, E_y), so t and s lie along z and the rotation leaves u_z alone; the
        // terms with t_y (exact zeros) are left out, which changes no rounding
        float2 f = mul2(P2(-2.0f), nrcp2(fma2(t2, t2, P2(1.0f))));
        float2 s2 = mul2(f, t2);
        float2 p0 = add2(um0, mul2(um1, t2));
        float2 p1 = sub2(um1, mul2(um0, t2));
        Q.u0 = add2(um0, mul2(p1, s2));
        Q.u1 = add2(sub2(um1, mul2(p0, s2)), mhey);
    }
    } else if constexpr (kConst) {
        // constant fields (the Sec. 2.2 bunch: fields off), the general Boris push
        ex = P2(c.E_const[0]);
        ey = P2(c.E_const[1]);
        ez = P2(c.E_const[2]);
        bx = P2(c.B_const[0]);
        by = P2(c.B_const[1]);
        bz = P2(c.B_const[2]);
        const float2 mh = P2(-0.5f * c.dt);
        const float2 um0 = fma2(mh, ex, Q.u0), um1 = fma2(mh, ey, Q.u1), um2 = fma2(mh, ez, Q.u2);
        const float2 ig = rsqrt2(fma2(um2, um2, fma2(um1, um1, fma2(um0, um0, P2(1.0f)))));
        const float2 mhig = mul2(mh, ig);
        const float2 t0 = mul2(bx, mhig), t1 = mul2(by, mhig), t2 = mul2(bz, mhig);   // -h B / gamma
        const float2 f = mul2(P2(-2.0f), nrcp2(fma2(t2, t2, fma2(t1, t1, fma2(t0, t0, P2(1.0f))))));
        const float2 s0_ = mul2(f, t0), s1 = mul2(f, t1), s2 = mul2(f, t2);
        const float2 p0 = add2(um0, sub2(mul2(um1, t2), mul2(um2, t1)));
        const float2 p1 = add2(um1, sub2(mul2(um2, t0), mul2(um0, t2)));
        const float2 p2 = add2(um2, sub2(mul2(um0, t1), mul2(um1, t0)));
        Q.u0 = fma2(mh, ex, add2(um0, sub2(mul2(p1, s2), mul2(p2, s1))));
        Q.u1 = fma2(mh, ey, add2(um1, sub2(mul2(p2, s0_), mul2(p0, s2))));
        Q.u2 = fma2(mh, ez, add2(um2, sub2(mul2(p0, s1), mul2(p1, s0_))));
    } else if constexpr (kRefl) {
        // incident pulse (B = x^ x E) plus the mirror image -r e(psi) at the reflected phase
        // t + x - 2 x_m, moving along -x (B = -x^ x E): E = (0, e_y + r_y, e_z + r_z),
        // B = (0, r_z - e_z, e_y - r_y)
        float2 st, ct;
        sincos2(phi, st, ct);
        const float2 eiy = mul2(ma0, fma2(dg, st, mul2(g, ct)));
        const float2 eiz = kCP ? mul2(P2(c.a0), sub2(mul2(dg, ct), mul2(g, st))) : P2(0.0f);
        const float2 pr = phase_refl2(c, nf2, Q);
        float2 gr, dgr, sr, cr, rem_r;
        const float2 arg_r = envelope_arg2(c, pr, rem_r);
        envelope2(c, pr, arg_r, rem_r, gr, dgr);
        sincos2(pr, sr, cr);
        const float2 ry = mul2(P2(c.refl_r * c.a0), fma2(dgr, sr, mul2(gr, cr)));    // -r (-a0 (...))
        ey = add2(eiy, ry);
        bz = sub2(eiy, ry);
        if constexpr (kCP) {
            const float2 rz = mul2(P2(-c.refl_r * c.a0), sub2(mul2(dgr, cr), mul2(gr, sr)));
            ez = add2(eiz, rz);
            by = sub2(rz, eiz);
        }
        // Boris push with E = (0, E_y, E_z), B = (0, B_y, B_z)
        const float2 mh = P2(-0.5f * c.dt);
        const float2 um0 = Q.u0;
        const float2 um1 = fma2(mh, ey, Q.u1);
        const float2 um2 = kCP ? fma2(mh, ez, Q.u2) : Q.u2;
        const float2 ig = rsqrt2(fma2(um2, um2, fma2(um1, um1, fma2(um0, um0, P2(1.0f)))));
        const float2 mhig = mul2(mh, ig);
        const float2 t2 = mul2(bz, mhig);                              // -h B_z / gamma
        if constexpr (kCP) {
            const float2 t1 = mul2(by, mhig);                          // -h B_y / gamma
            const float2 f = mul2(P2(-2.0f), nrcp2(fma2(t2, t2, fma2(t1, t1, P2(1.0f)))));
            const float2 s1 = mul2(f, t1), s2 = mul2(f, t2);
            const float2 p0 = add2(um0, sub2(mul2(um1, t2), mul2(um2, t1)));
            const float2 p1 = sub2(um1, mul2(um0, t2));
            const float2 p2 = fma2(um0, t1, um2);
            Q.u0 = add2(um0, sub2(mul2(p1, s2), mul2(p2, s1)));
            Q.u1 = fma2(mh, ey, sub2(um1, mul2(p0, s2)));
            Q.u2 = fma2(mh, ez, fma2(p0, s1, um2));
        } else {
            const float2 f = mul2(P2(-2.0f), nrcp2(fma2(t2, t2, P2(1.0f))));
            const float2 s2 = mul2(f, t2);
            const float2 p0 = fma2(um1, t2, um0);
            const float2 p1 = sub2(um1, mul2(um0, t2));
            Q.u0 = fma2(p1, s2, um0);
            Q.u1 = fma2(mh, ey, sub2(um1, mul2(p0, s2)));
        }
    } else {
        // 2D paraxial focus (fields() in physics.cuh), amplitude and Gouy phase by gouy2: with
        // S = sqrt(w0 / w) e^{-y^2 / w^2} and theta = phi - y^2 / (2 R_c) + atan(a) / 2,
        // E_y = -a0 S (g' sin + g cos), E_x = a0 g S (y / R_c cos + 2 y / w^2 sin), for CP
        // E_z = a0 S (g' cos - g sin) and B_x = a0 g S (2 y / w^2 cos - y / R_c sin); B = (B_x, -E_z, E_y)
        const float2 a = mul2(sub2(Q.x, P2(c.xf)), P2(c.inv_zr));
        float2 Rn, In, inv_n2;
        gouy2(a, Rn, In, inv_n2);
        const float2 yy = mul2(Q.y, Q.y);
        const float2 inv_w2 = mul2(inv_n2, P2(c.inv_w0sq));
        const float2 inv_R = mul2(mul2(a, inv_n2), P2(c.inv_zr));
        const float2 G_ = exp_neg2(mul2(yy, inv_w2));
        float2 s0, c0;
        sincos2(fma2(mul2(yy, inv_R), P2(-0.5f), phi), s0, c0);
        const float2 Sc = mul2(G_, sub2(mul2(Rn, c0), mul2(In, s0)));    // S cos(theta)
        const float2 Ss = mul2(G_, fma2(Rn, s0, mul2(In, c0)));          // S sin(theta)
        ey = mul2(ma0, fma2(dg, Ss, mul2(g, Sc)));
        const float2 yR = mul2(Q.y, inv_R), y2w = mul2(mul2(P2(2.0f), Q.y), inv_w2);
        const float2 a0g = mul2(P2(c.a0), g);
        ex = mul2(a0g, fma2(yR, Sc, mul2(y2w, Ss)));
        if constexpr (kCP) {
            ez = mul2(P2(c.a0), sub2(mul2(dg, Sc), mul2(g, Ss)));
            bx = mul2(a0g, sub2(mul2(y2w, Sc), mul2(yR, Ss)));
        }
        // Boris push, u^- = u - h E, rotation by t = -h B / gamma^-, u^+ = u^- + (u^- + u^- x t) x s
        // - h E (terms of the exact zeros left out: B_y = B_x = E_z = 0 for LP)
        const float2 mh = P2(-0.5f * c.dt);
        const float2 um0 = fma2(mh, ex, Q.u0);
        const float2 um1 = fma2(mh, ey, Q.u1);
        const float2 um2 = kCP ? fma2(mh, ez, Q.u2) : Q.u2;
        const float2 ig = rsqrt2(fma2(um2, um2, fma2(um1, um1, fma2(um0, um0, P2(1.0f)))));
        const float2 mhig = mul2(mh, ig);
        const float2 t2 = mul2(ey, mhig);                              // -h B_z / gamma
        if constexpr (kCP) {
            const float2 t0 = mul2(bx, mhig);                          // -h B_x / gamma
            const float2 t1 = mul2(ez, mul2(P2(0.5f * c.dt), ig));     // -h B_y / gamma, B_y = -E_z
            const float2 f = mul2(P2(-2.0f), nrcp2(fma2(t2, t2, fma2(t1, t1, fma2(t0, t0, P2(1.0f))))));
            const float2 s0_ = mul2(f, t0), s1 = mul2(f, t1), s2 = mul2(f, t2);
            const float2 p0 = add2(um0, sub2(mul2(um1, t2), mul2(um2, t1)));
            const float2 p1 = add2(um1, sub2(mul2(um2, t0), mul2(um0, t2)));
            const float2 p2 = add2(um2, sub2(mul2(um0, t1), mul2(um1, t0)));
            Q.u0 = fma2(mh, ex, add2(um0, sub2(mul2(p1, s2), mul2(p2, s1))));
            Q.u1 = fma2(mh, ey, add2(um1, sub2(mul2(p2, s0_), mul2(p0, s2))));
            Q.u2 = fma2(mh, ez, add2(um2, sub2(mul2(p0, s1), mul2(p1, s0_))));
        } else {
            const float2 f = mul2(P2(-2.0f), nrcp2(fma2(t2, t2, P2(1.0f))));
            const float2 s2 = mul2(f, t2);
            const float2 p0 = fma2(um1, t2, um0);
            const float2 p1 = sub2(um1, mul2(um0, t2));
            Q.u0 = fma2(mh, ex, fma2(p1, s2, um0));
            Q.u1 = fma2(mh, ey, sub2(um1, mul2(p0, s2)));
        }
    }
    // gamma and 1/gamma from one reciprocal square root (1/gamma serves the rate and the
    // position update; emitting lanes refresh it from their new gamma)
    gamma_pair(Q, gamma, inv_g);
    unsigned crossed = 0;
    if (ncs_on<F>(r)) {
        // eta = (gamma - u_x) |E| / E_S for the plane wave; ngm = u_x - gamma, for u_x > 0 as
        // -(1 + u_y^2 + u_z^2) / (gamma + u_x) (no cancellation), its sign taken by the last factor
        float2 up = fma2(Q.u2, Q.u2, fma2(Q.u1, Q.u1, P2(1.0f)));
        float2 ngm = sel2(Q.u0.x > 0.0f, Q.u0.y > 0.0f, mul2(up, nrcp2(add2(gamma, Q.u0))), sub2(Q.u0, gamma));
        if constexpr (kPlane) {
            float2 Emag = (G == FK_PLANE_CP) ? sqrt2(fma2(ez, ez, mul2(ey, ey))) : make_float2(fabsf(ey.x), fabsf(ey.y));
            eta = mul2(mul2(ngm, Emag), P2(-c.inv_ES));
        } else if constexpr (kConst) {
            // eta = |V^2 + 2 V_x (u.E)|^{1/2} / E_S with V = (gamma - u_x) E + u x d, d = B - x^ x E =
            // (B_x, B_y + E_z, B_z - E_y); nV = -V
            const float2 d1 = add2(by, ez), d2 = sub2(bz, ey);
            const float2 nV0 = sub2(mul2(ngm, ex), sub2(mul2(Q.u1, d2), mul2(Q.u2, d1)));
            const float2 nV1 = sub2(mul2(ngm, ey), sub2(mul2(Q.u2, bx), mul2(Q.u0, d2)));
            const float2 nV2 = sub2(mul2(ngm, ez), sub2(mul2(Q.u0, d1), mul2(Q.u1, bx)));
            const float2 uE = fma2(Q.u2, ez, fma2(Q.u1, ey, mul2(Q.u0, ex)));
            const float2 qv = sub2(fma2(nV2, nV2, fma2(nV1, nV1, mul2(nV0, nV0))), mul2(mul2(P2(2.0f), nV0), uE));
            const float2 rq = sqrt2(make_float2(fmaxf(qv.x, 0.0f), fmaxf(qv.y, 0.0f)));
            eta = mul2(rq, P2(c.inv_ES));
        } else if constexpr (kRefl) {
            // eta = |V^2 + 2 V_x (u.E)|^{1/2} / E_S with V = (gamma - u_x) E + u x d, d = B - x^ x E =
            // (0, B_y + E_z, B_z - E_y); nV1, nV2 = -V_y, -V_z
            const float2 d2 = sub2(bz, ey);
            const float2 d1 = kCP ? add2(by, ez) : P2(0.0f);
            const float2 V0 = kCP ? sub2(mul2(Q.u1, d2), mul2(Q.u2, d1)) : mul2(Q.u1, d2);
            const float2 nV1 = fma2(ngm, ey, mul2(Q.u0, d2));
            const float2 nV2 = kCP ? sub2(mul2(ngm, ez), mul2(Q.u0, d1)) : P2(0.0f);
            const float2 uE = kCP ? fma2(Q.u2, ez, mul2(Q.u1, ey)) : mul2(Q.u1, ey);
            const float2 qv = fma2(mul2(P2(2.0f), V0), uE, fma2(nV2, nV2, fma2(nV1, nV1, mul2(V0, V0))));
            const float2 rq = sqrt2(make_float2(fmaxf(qv.x, 0.0f), fmaxf(qv.y, 0.0f)));
            eta = mul2(rq, P2(c.inv_ES));
        } else {
            // eta = |V^2 + 2 V_x (u.E)|^{1/2} / E_S with V = (gamma - u_x) E + u x (B - x^ x E): here
            // B_y + E_z = B_z - E_y = 0, so u x (...) = (0, u_z B_x, -u_y B_x); nV = -V except in y
            const float2 nV0 = mul2(ngm, ex);
            const float2 uE = fma2(Q.u1, ey, fma2(Q.u0, ex, kCP ? mul2(Q.u2, ez) : P2(0.0f)));
            float2 V1 = mul2(ngm, ey), V2 = P2(0.0f);
            if constexpr (kCP) {
                V1 = sub2(mul2(Q.u2, bx), V1);                         // u_z B_x + (gamma - u_x) E_y
                V2 = fma2(Q.u1, bx, mul2(ngm, ez));                    // -(V_z)
            }
            const float2 qv = sub2(fma2(V2, V2, fma2(V1, V1, mul2(nV0, nV0))), mul2(mul2(P2(2.0f), nV0), uE));
            const float2 rq = sqrt2(make_float2(fmaxf(qv.x, 0.0f), fmaxf(qv.y, 0.0f)));
            eta = mul2(rq, P2(c.inv_ES));
        }
        // h(eta): row interpolation in log eta (log2 scaled to the row position by one FMA), the
        // classical limit below the table; above it the last row, counted (the position is clamped
        // just below the top node, so the split needs no correction there)
        const float2 tp = fma2(log2v(eta), P2(tc.inv_dln_eta * 0.693147180559945309f),
                               P2(-tc.ln_eta_min * tc.inv_dln_eta));
        n_above = add2(n_above, make_float2(tp.x >= tc.eta_last ? 1.0f : 0.0f, tp.y >= tc.eta_last ? 1.0f : 0.0f));
        const float2 tpc = clamp2(tp, 0.0f, tc.eta_last - 0x1.0p-10f);
        const float2 tt = add2(sub2(tpc, P2(0.5f)), P2(0x1.8p23f));
        const int ix = dbg_idx(t.dbg, __float_as_int(tt.x) - 0x4B400000, t.n_eta - 1);
        const int iy = dbg_idx(t.dbg, __float_as_int(tt.y) - 0x4B400000, t.n_eta - 1);
        const float2 w = sub2(tpc, sub2(tt, P2(0x1.8p23f)));
        const float2 h0 = make_float2(h_tab[ix], h_tab[iy]), h1 = make_float2(h_tab[ix + 1], h_tab[iy + 1]);
        float2 hv = fma2(w, sub2(h1, h0), h0);
        hv = sel2(eta.x >= tc.eta_min, eta.y >= tc.eta_min, hv, P2(tc.h_classical));
        // tau -= ncs_coef (eta / gamma) h(eta), compensated by Dekker's Fast2Sum (exact for
        // |tau| >= |dtau|, which holds on every step but the one where tau crosses zero, and
        // that step emits and resets tau)
        const float2 ndtau = mul2(mul2(P2(-c.ncs_coef), mul2(eta, inv_g)), hv);
        const float2 s = add2(Q.tau, ndtau);
        const float2 e = sub2(ndtau, sub2(s, Q.tau));
        Q.tau = s;
        Q.tau_lo = add2(Q.tau_lo, e);
        float2 tsum = add2(Q.tau, Q.tau_lo);
        crossed = (unsigned)(tsum.x <= 0.0f) | ((unsigned)(tsum.y <= 0.0f) << 1);
    }
    return crossed;
}

// The bremsstrahlung test of Eq. 4 of the pair after its NCS emissions (or the null-collision waits): a bit per
// electron with a collision to sample (a candidate, for null collisions).
template <int G, int F>
__device__ __forceinline__ unsigned brems_pair(const TablesDev& t, const RunDevT<float>& r, const float* sig_tab,
                                               const uint32_t id[2], uint32_t n, Pair& Q, float2 gamma, float2 inv_g,
                                               const SumsCta& acc) {
    constexpr bool kOneD = G != FK_GAUSS_LP && G != FK_GAUSS_CP;
    const StepC<float>& c = r.c;
    const TabC<float>& tc = t.cf;
    unsigned hit = 0;
    if (null_on<F>(r)) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            if (!Q.act[k]) continue;
            if (Q.wait[k] == 0u) hit |= 1u << k;
            else if (Q.wait[k] != PE_WAIT_NEVER) --Q.wait[k];
        }
        return hit;
    }
    // Almost every test fails, and the draw alone shows it: a passing draw has its high word at most the
    // run's largest probability (br_cap), so the first thing formed is that one word of the draw, and the
    // rate, the probability and the rest of the draw only for an electron whose word is that low (or whose
    // gamma may be above the table, which is counted).  Philox bounds the test in the target; with the rate
    // and the probability formed for every electron there, 6e6 electrons one step per call took 120 us a
    // step and then 92, the 1 GeV Au bunch (5e5 electrons, 2000 steps) 10.9 ms and then 9.9, the 1e6 x 4000
    // job, in the target for a tenth of its steps, 19.6 and then 19.1 ms.
    bool in[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const float x = comp(Q.x, k);
        in[k] = x >= c.x0 && x <= c.x1 && (kOneD || fabsf(comp(Q.y, k)) <= c.yh) &&
                comp(gamma, k) > 1.0f + tc.photon_min;
    }
    if (in[0] || in[1]) {
        const uint32_t hi0 = draw(r, id[0], n, PUR_BREMS).y, hi1 = draw(r, id[1], n, PUR_BREMS).y;
        in[0] = in[0] && (hi0 <= r.br_cap || gamma.x >= tc.g_safe);
        in[1] = in[1] && (hi1 <= r.br_cap || gamma.y >= tc.g_safe);
    }
    if (in[0] || in[1]) {
        // x_b = K sigma_Z(gamma) beta on the paired instructions (row position in log gamma from log2 by
        // one FMA, clamped below the top node as for h(eta); beta = |u| / gamma), then per electron the
        // whole draw and the integer test
        const float2 tg = fma2(log2v(gamma), P2(tc.inv_dln_g * 0.693147180559945309f),
                               P2(-tc.ln_g_min * tc.inv_dln_g));
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (in[k] && comp(tg, k) >= tc.g_last) acc.count(PE_T_N_GAMMA_ABOVE);
        const float2 tgc = clamp2(tg, 0.0f, tc.g_last - 0x1.0p-10f);
        const float2 tt = add2(sub2(tgc, P2(0.5f)), P2(0x1.8p23f));
        const int gx = dbg_idx(t.dbg, __float_as_int(tt.x) - 0x4B400000, t.n_E - 1);
        const int gy = dbg_idx(t.dbg, __float_as_int(tt.y) - 0x4B400000, t.n_E - 1);
        const float2 w = sub2(tgc, sub2(tt, P2(0x1.8p23f)));
        const float2 s0 = make_float2(sig_tab[gx], sig_tab[gy]);
        const float2 s1 = make_float2(sig_tab[gx + 1], sig_tab[gy + 1]);
        const float2 sig = fma2(w, sub2(s1, s0), s0);
        const float2 um = sqrt2(fma2(Q.u2, Q.u2, fma2(Q.u1, Q.u1, mul2(Q.u0, Q.u0))));
        const float2 xb = mul2(mul2(P2(c.K_br), sig), mul2(um, inv_g));
        // 1 - e^{-x_b} by its Taylor series below 2^-5 (truncation under 2^-26 relative), the
        // library expm1f above: one_minus_exp_neg_f32 on the paired instructions
        const float2 ser = brems_series2(xb);
        float pb_[2] = {ser.x, ser.y};
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            if (!in[k]) continue;
            if (!(comp(xb, k) < 0x1.0p-5f)) pb_[k] = -expm1f(-comp(xb, k));
            uint32_t idk = id[k];
            asm volatile("" : "+r"(idk));               // formed again here, not carried from the test above
            const uint4 wd = draw(r, idk, n, PUR_BREMS);
            if (brems_event(pb_[k], wd)) hit |= 1u << k;
        }
    }
    return hit;
}

// A thread's emission state while it waits (see pair_loop), in shared memory: eta and gamma of its step and 1/gamma
struct Held {
    float2 *eta, *gamma, *inv_g;
};
// its NCS emissions.  One inlined branch that takes the crossings of a lane one at a time, so lanes whose crossing is
// in different halves of their pairs take it together; or one for each half (kTwoSites), which spares the
// selects: the single-run kernels of the kinds with rare emissions (2D focus job 16.2 against 16.6 ms; in the
// batch instances, whose registers spill, 24.9 against 24.5).
template <int G, bool kTwoSites>
__device__ __forceinline__ void emit_ncs_pair(const TablesDev& t, const RunDevT<float>& r, const uint32_t id[2],
                                              uint32_t n, unsigned m, Pair& Q, float2& gamma, float2& inv_g, float2 eta,
                                              const SumsCta& acc) {
    auto emit = [&](int k) {
        Particle<float> P = unpack(Q, k);
        float gk = comp(gamma, k);
        const uint32_t idk = k ? id[1] : id[0];
        bool st;
        Photon ph;
        take(ncs_emit_body<float>(t, r, idk, n, P, gk, comp(eta, k), comp(Q.x, k), comp(Q.y, k), acc), P, gk, st, ph);
        if (st) append_now(r, ph);
        add_events(r, idk, P);
        repack(Q, k, P);
        // 1/gamma by the correctly rounded reciprocal: with the branch inlined, a plain division of its sqrt
        // result is open to per-kernel rewriting (1/sqrt as rsqrt), and every paired kernel must round it alike
        set_comp(inv_g, k, __frcp_rn(gk));
        set_comp(gamma, k, gk);
    };
    if constexpr (kTwoSites) {
        if (m & 1u) emit(0);
        if (m & 2u) emit(1);
    } else {
        while (m) {
            emit((m & 1u) ? 0 : 1);
            m &= m - 1u;
        }
    }
}
// its bremsstrahlung photons, or null-collision candidates
template <int G, int F>
__device__ __forceinline__ void emit_brems_pair(const TablesDev& t, const RunDevT<float>& r, const float* sig_tab,
                                                const uint32_t id[2], uint32_t n, unsigned m, Pair& Q, float2 gamma,
                                                float2& inv_g, const SumsCta& acc) {
    constexpr bool kOneD = G != FK_GAUSS_LP && G != FK_GAUSS_CP;
    const StepC<float>& c = r.c;
    while (m) {
        const int k = (m & 1u) ? 0 : 1;
        m &= m - 1u;
        Particle<float> P = unpack(Q, k);
        float gk = comp(gamma, k);
        const uint32_t idk = k ? id[1] : id[0];
        const float x = comp(Q.x, k), y = comp(Q.y, k);
        bool st;
        Photon ph;
        if (null_on<F>(r)) {
            const bool in_slab = x >= c.x0 && x <= c.x1 && (kOneD || fabsf(y) <= c.yh);
            take(brems_candidate<float>(t, r, sig_tab, idk, n, P, gk, in_slab, x, y, acc), P, gk, st, ph);
        } else {
            take(brems_emit_body<float>(t, r, idk, n, P, gk, x, y, draw(r, idk, n, PUR_BREMS), acc), P, gk, st, ph);
        }
        if (st) append_now(r, ph);
        add_events(r, idk, P);
        repack(Q, k, P);
        set_comp(inv_g, k, __frcp_rn(gk));
    }
}
// x^{n+1} = x^n + dt u_x / gamma (and y), compensated
template <int G>
__device__ __forceinline__ void move_pair(const StepC<float>& c, Pair& Q, float2 inv_g) {
    const float2 dt = P2(c.dt);
    float2 s, e;
    two_sum2(Q.x, mul2(mul2(dt, Q.u0), inv_g), s, e);
    Q.x = s;
    Q.x_lo = add2(Q.x_lo, e);
    if constexpr (G == FK_GAUSS_LP || G == FK_GAUSS_CP) {
        two_sum2(Q.y, mul2(mul2(dt, Q.u1), inv_g), s, e);
        Q.y = s;
        Q.y_lo = add2(Q.y_lo, e);
    }
}

__device__ __forceinline__ void load_one(const RunDevT<float>& r, int64_t i, Pair& Q, int k,
                                         unsigned long long* tally) {
    Particle<float> P;
    load_particle<float>(r, i, P);
    Q.act[k] = live_or_kill<float>(r, i, P, (uint32_t)r.step0, tally);
    repack(Q, k, P);
}

// absorbing box (Sec. 3) after a step: a removed electron is stored at once
template <int G>
__device__ __forceinline__ void box_pair(const RunDevT<float>& r, int64_t i0, int64_t i1, uint32_t n, Pair& Q,
                                         unsigned long long* s_tally) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        if (!Q.act[k]) continue;
        Particle<float> P = unpack(Q, k);
        box_check<float>(r, P, n, s_tally);
        set_comp(Q.x, k, P.x);
        if (isnan(P.x)) {
            Q.act[k] = false;
            store_one(r, k ? i1 : i0, P);
        }
    }
    retire<G>(Q);
}

// The steps of a warp's electrons before the pulse is at any of them: without a field the push is the identity and eta is
// 0, so the optical depth stays, and a step is gamma, the bremsstrahlung test and the move.  Returns the steps done.
// A job spends 5 to 30 % of its steps so.  In a loop of its own because a branch around the push in every step costs
// the paired instructions their order: 1D job 18.4 ms without either, 19.2 with such a branch, 18.1 with the loop; 2D
// focus (1000 steps) 15.4, 13.6 and 13.0; reflected 15.4, 15.6 and 14.9; batch of 64 23.0, 22.0 and 20.8.
template <int G, int F>
__device__ __forceinline__ int steps_before_pulse(const TablesDev& t, const RunDevT<float>& r, const float* sig_z,
                                                  const uint32_t id[2], int64_t i0, int64_t i1, Pair& Q, int steps,
                                                  const SumsCta& acc, unsigned long long* s_tally) {
    const uint32_t n0 = (uint32_t)r.step0;
    float nf = (float)n0;
    int s = 0;
    for (; s < steps; ++s, nf += 1.0f) {
        const bool act = Q.act[0] || Q.act[1];
        if (!__all_sync(0xffffffffu, !act || no_pulse<G>(r.c, nf, Q))) break;
        if (act) {
            const uint32_t n = n0 + (uint32_t)s;
            float2 gamma, inv_g;
            gamma_pair(Q, gamma, inv_g);
            if (brems_on<F>(r)) {
                const unsigned hit = brems_pair<G, F>(t, r, sig_z, id, n, Q, gamma, inv_g, acc);
                if (hit) emit_brems_pair<G, F>(t, r, sig_z, id, n, hit, Q, gamma, inv_g, acc);
            }
            move_pair<G>(r.c, Q, inv_g);
            if (box_on<F>(r)) box_pair<G>(r, i0, i1, n, Q, s_tally);
        }
    }
    return s;
}

// K steps of the pair Q (electrons i0 and i1), the lanes of a warp in step: an emission is taken where it falls.
template <int G, int F, bool kTwoSites, bool kStream>
__device__ __forceinline__ void pair_loop(const TablesDev& t, const RunDevT<float>& r, const float* s_h,
                                          const float* sig_z, int64_t i0, int64_t i1, Pair& Q, int steps,
                                          const SumsCta& acc, unsigned long long* s_tally) {
    const uint32_t id[2] = {r.id0 + (uint32_t)i0, r.id0 + (uint32_t)i1};
    const uint32_t n0 = (uint32_t)r.step0;
    int s = 0;
    if constexpr (G != FK_CONST && !kStream) s = steps_before_pulse<G, F>(t, r, sig_z, id, i0, i1, Q, steps, acc, s_tally);
    float nf = (float)(n0 + (uint32_t)s);
    float2 n_above = P2(0.0f);                          // particle-steps with eta above the table (exact to 2^24)
    for (; s < steps; ++s, nf += 1.0f) {
        if (Q.act[0] || Q.act[1]) {
            const uint32_t n = n0 + (uint32_t)s;
            float2 gamma, inv_g, eta;
            const unsigned crossed = push_pair<G, F>(t, r, s_h, nf, Q, gamma, inv_g, eta, n_above);
            if (F != kFlagsBrems && crossed) emit_ncs_pair<G, kTwoSites>(t, r, id, n, crossed, Q, gamma, inv_g, eta, acc);
            if (brems_on<F>(r)) {
                const unsigned hit = brems_pair<G, F>(t, r, sig_z, id, n, Q, gamma, inv_g, acc);
                if (hit) emit_brems_pair<G, F>(t, r, sig_z, id, n, hit, Q, gamma, inv_g, acc);
            }
            move_pair<G>(r.c, Q, inv_g);
            if (box_on<F>(r)) box_pair<G>(r, i0, i1, n, Q, s_tally);
        }
    }
    const unsigned int na = __float2uint_rz(n_above.x) + __float2uint_rz(n_above.y);
    if (na) atomicAdd(s_tally + PE_T_N_ETA_ABOVE, (unsigned long long)na);
}

// The same with lanes that wait for their emissions.
//
// A warp that branches into an emission for one lane issues all of it, several times a step's length, for that lane.
// The lanes need not be at the same step: electrons are independent and their draws keyed on (electron, step).  So a
// lane with an emission waits where it is while the others step on, until the lane-steps lost by waiting reach
// kHoldSteps or no lane can step; then the waiting lanes emit together.  Measured with thresholds of 16, 24, 32
// and 64 lane-steps against none: the reflected job 16.2, 15.9, 15.9 and 16.2 against 17.7 ms, the bunch 8.32,
// 8.28, 8.27 and 8.39 against 8.72.  Where emissions are rare a lane waits long for company and in the end the warp
// waits for that lane: at 48 lane-steps the 1D job took 22.3 against 20.9 ms (hold_of chooses).
constexpr int kHoldSteps = 32;
template <int G, int F>
__device__ __forceinline__ void pair_loop_hold(const TablesDev& t, const RunDevT<float>& r, const float* s_h,
                                               const float* sig_z, int64_t i0, int64_t i1, Pair& Q, int steps,
                                               const SumsCta& acc, const Held& held_at, unsigned long long* s_tally) {
    const uint32_t id[2] = {r.id0 + (uint32_t)i0, r.id0 + (uint32_t)i1};
    int done = 0;
    if constexpr (G != FK_CONST) done = steps_before_pulse<G, F>(t, r, sig_z, id, i0, i1, Q, steps, acc, s_tally);
    uint32_t n = (uint32_t)r.step0 + (uint32_t)done;    // this lane's step
    float nf = (float)n;
    int left = (Q.act[0] || Q.act[1]) ? steps - done : 0;   // and its steps to go
    float2 n_above = P2(0.0f);
    unsigned held = 0;                                  // emissions waited for: bits 0, 1 NCS, bits 2, 3 brems
    int lost = 0;
    while (true) {
        const bool run = left > 0 && !held;
        bool test = false, move = false;
        float2 gamma, inv_g;
        if (run) {
            float2 eta;
            held = push_pair<G, F>(t, r, s_h, nf, Q, gamma, inv_g, eta, n_above);
            if (held) {
                *held_at.eta = eta;
                *held_at.gamma = gamma;
                *held_at.inv_g = inv_g;
            }
            test = !held;
        }
        const unsigned waiting = __ballot_sync(0xffffffffu, held != 0);
        if (waiting) {
            lost += __popc(waiting);
            if (lost >= kHoldSteps || !__any_sync(0xffffffffu, test)) {
                lost = 0;
                if (held) {
                    gamma = *held_at.gamma;
                    inv_g = *held_at.inv_g;
                    if (F != kFlagsBrems && (held & 3u)) {
                        emit_ncs_pair<G, false>(t, r, id, n, held, Q, gamma, inv_g, *held_at.eta, acc);
                        test = true;
                    } else {
                        emit_brems_pair<G, F>(t, r, sig_z, id, n, held >> 2, Q, gamma, inv_g, acc);
                        move = true;
                    }
                    held = 0;
                }
            }
        } else if (!__any_sync(0xffffffffu, test)) {
            break;                                      // no lane waits and none stepped: all are done
        }
        if (test) {
            move = true;
            if (brems_on<F>(r)) {
                held = brems_pair<G, F>(t, r, sig_z, id, n, Q, gamma, inv_g, acc) << 2;
                if (held) {
                    *held_at.gamma = gamma;
                    *held_at.inv_g = inv_g;
                    move = false;
                }
            }
        }
        if (move) {
            move_pair<G>(r.c, Q, inv_g);
            if (box_on<F>(r)) {
                box_pair<G>(r, i0, i1, n, Q, s_tally);
                if (!Q.act[0] && !Q.act[1]) left = 1;
            }
            ++n;
            nf += 1.0f;
            --left;
        }
    }
    const unsigned int na = __float2uint_rz(n_above.x) + __float2uint_rz(n_above.y);
    if (na) atomicAdd(s_tally + PE_T_N_ETA_ABOVE, (unsigned long long)na);
}

__device__ __forceinline__ void pair_clear(Pair& Q) {
    Q.x_lo = Q.y = Q.y_lo = Q.u0 = Q.u1 = Q.u2 = Q.tau_lo = P2(0.0f);
    Q.x = Q.tau = P2(__int_as_float(0x7fc00000));       // an empty slot is NaN, as a removed electron
    Q.wait[0] = Q.wait[1] = PE_WAIT_NEVER;
    Q.act[0] = Q.act[1] = false;
}

// Shared memory of the paired kernels: the CTA's sums and the held lanes' slots (kPairFixedBytes, a multiple of 16
// bytes), then h(eta) and sigma_Z(gamma): every row of a small set, otherwise that of the run's Z alone (a batch copies the
// row again when it comes to another run).  Rate tables of 2 / 20 / 36 / 100 KB (n_E = 256 / 2048 / 4000 / 4000 rows of
// 2 / 2 / 2 / 6 Z), 2e5 electrons x 300 steps: 0.54 / 0.65 / 0.67 / 1.54 ms with every row copied, 0.54 / 0.55 / 0.65 / 0.65 so.
constexpr int kPairFixedBytes = kSumsThreads * (16 * kEnergySums + 3 * 8) + 8 * PE_TALLY_WORDS + 4 * PE_HIST_WORDS +
                                4 * PE_T_E_NCS_STORED;
static_assert(kPairFixedBytes % 16 == 0, "tables after a 16-byte boundary");
struct PairShared {
    ulonglong2* sums;              // [kEnergySums][kSumsThreads]
    unsigned long long* tally;     // [PE_TALLY_WORDS]: the counts that are not per emission
    float2* held;                  // [3][kSumsThreads]
    uint32_t* hist;                // [PE_HIST_WORDS]
    uint32_t* cnt;                 // [PE_T_E_NCS_STORED]
    float *h, *sig;
    __device__ __forceinline__ explicit PairShared(unsigned char* smem, int n_eta) {
        sums = reinterpret_cast<ulonglong2*>(smem);
        tally = reinterpret_cast<unsigned long long*>(sums + kEnergySums * kSumsThreads);
        held = reinterpret_cast<float2*>(tally + PE_TALLY_WORDS);
        hist = reinterpret_cast<uint32_t*>(held + 3 * kSumsThreads);
        cnt = hist + PE_HIST_WORDS;
        h = reinterpret_cast<float*>(cnt + PE_T_E_NCS_STORED);
        sig = h + n_eta;
    }
    __device__ __forceinline__ void init(const TablesDev& t) const {
        uint4* w = reinterpret_cast<uint4*>(sums);
        for (int k = threadIdx.x; k < kPairFixedBytes / 16; k += blockDim.x) w[k] = make_uint4(0, 0, 0, 0);
#pragma unroll 4
        for (int k = threadIdx.x; k < t.n_eta; k += blockDim.x) h[k] = t.h32[k];
    }
    // row iz alone (stride 0) or all rows
    __device__ __forceinline__ void load_sigma(const TablesDev& t, int stride, int iz) const {
        const float* rows = t.sig32 + (stride ? 0 : (size_t)iz * t.n_E);
        const int n = stride ? t.n_Z * t.n_E : t.n_E;
#pragma unroll 4
        for (int k = threadIdx.x; k < n; k += blockDim.x) sig[k] = rows[k];
    }
    __device__ __forceinline__ SumsCta acc() const { return SumsCta{hist, cnt, sums + threadIdx.x}; }
    __device__ __forceinline__ Held slots() const {
        float2* s = held + threadIdx.x;
        return Held{s, s + kSumsThreads, s + 2 * kSumsThreads};
    }
    // add everything to the run's words and clear it
    __device__ __forceinline__ void flush(const RunDevT<float>& r) const {
        __syncthreads();
#pragma unroll 4
        for (int k = threadIdx.x; k < PE_HIST_WORDS; k += blockDim.x) {
            const uint32_t v = hist[k];
            if (v) { atomicAdd(r.hist + k, (unsigned long long)v); hist[k] = 0; }
        }
        if (threadIdx.x < PE_T_E_NCS_STORED) {
            const unsigned long long v = tally[threadIdx.x] + cnt[threadIdx.x];
            if (v) { atomicAdd(r.tally + threadIdx.x, v); tally[threadIdx.x] = 0; cnt[threadIdx.x] = 0; }
        }
        for (int k = 0; k < kEnergySums; ++k) {          // 128-bit sums: over the warp, then one add per warp
            ulonglong2 v = sums[k * kSumsThreads + threadIdx.x];
            if (!__any_sync(0xffffffffu, (v.x | v.y) != 0)) continue;
            sums[k * kSumsThreads + threadIdx.x] = make_ulonglong2(0, 0);
            v = warp_sum(v);
            if ((threadIdx.x & 31) == 0) fx_add_words(r.tally + PE_T_E_NCS_STORED + 2 * k, v);
        }
        __syncthreads();
    }
};

// K steps of the two electrons i0 = base + tid and i1 = base + tid + blockDim
template <int G, int F, bool kSingle, bool kHold>
__device__ __forceinline__ void tile_steps_pair(const TablesDev& t, const RunDevT<float>& r, const float* s_h,
                                                const float* sig_z, int64_t i0, int64_t i1, int steps,
                                                const SumsCta& acc, const Held& held,
                                                unsigned long long* s_tally) {
    Pair Q;
    pair_clear(Q);
    if (i0 < r.n) load_one(r, i0, Q, 0, s_tally);
    if (i1 < r.n) load_one(r, i1, Q, 1, s_tally);
    if constexpr (G != FK_GAUSS_LP && G != FK_GAUSS_CP) Q.y = Q.y_lo = P2(0.0f);   // 1D: y is not state
    retire<G>(Q);
    const bool live0 = i0 < r.n, live1 = i1 < r.n;
    if constexpr (kHold)
        pair_loop_hold<G, F>(t, r, s_h, sig_z, i0, i1, Q, steps, acc, held, s_tally);
    else
        pair_loop<G, F, kSingle, false>(t, r, s_h, sig_z, i0, i1, Q, steps, acc, s_tally);
    if (live0 && Q.act[0]) store_one(r, i0, unpack(Q, 0));
    if (live1 && Q.act[1]) store_one(r, i1, unpack(Q, 1));
}

// Resident CTAs of 128 threads per SM the register budget is sized for.  Plane wave, 1D job (1e6 x 4000) / batch of 64:
// 6 CTAs (80 registers) 18.06 / 21.2 ms, 7 (72) 18.07 / 20.8, 8 (64, with some 20 words spilled around the
// emissions) 17.81 / 20.4.
#ifndef PE_PAIR_MIN_CTAS
#define PE_PAIR_MIN_CTAS 8
#endif
// The 2D focus (2e6 electrons x 1000 steps): 4 CTAs 13.6 ms, 5 13.0, 6 12.8, 7 12.7; at 7 the batch instance (served
// requests) spills around its common path.
#ifndef PE_PAIR_MIN_CTAS_2D
#define PE_PAIR_MIN_CTAS_2D 6
#endif
// The reflected wave (2.5e5 electrons x 3000 steps): 5 CTAs 16.8 ms, 6 16.8, 7 14.9, 8 15.1.
#ifndef PE_PAIR_MIN_CTAS_REFL
#define PE_PAIR_MIN_CTAS_REFL 7
#endif
// The general instances (flags read at run time: the null-collision method, a process switched off, the box boundary)
// carry more live state than the others and spill 250 to 370 bytes at 7 CTAs.  At 6 small runs gain (3e5 electrons, plane
// wave with a box / by null collisions, 700 steps, the Au bunch by null collisions at dt = T / 10, 2500 steps: 1.99 / 1.60 /
// 2.86 ms, at 7 2.03 / 1.71 / 2.95), larger ones lose more (1e6 electrons 5.80 / 4.49 / 7.33, at 7 5.44 / 4.41 / 6.64).
#ifndef PE_PAIR_MIN_CTAS_GENERAL
#define PE_PAIR_MIN_CTAS_GENERAL 7
#endif
// Brems alone (the bunch by the direct method, 5e5 electrons x 2000 steps): 7 to 9 CTAs 5.73 to 5.78 ms, 10 5.84.
#ifndef PE_PAIR_MIN_CTAS_BREMS
#define PE_PAIR_MIN_CTAS_BREMS 8
#endif
template <int G, int F>
constexpr int pair_min_ctas() {
    constexpr int kind = (G == FK_GAUSS_LP || G == FK_GAUSS_CP) ? PE_PAIR_MIN_CTAS_2D
                         : (G == FK_REFL_LP || G == FK_REFL_CP) ? PE_PAIR_MIN_CTAS_REFL : PE_PAIR_MIN_CTAS;
    if (F == kFlagsBrems) return PE_PAIR_MIN_CTAS_BREMS;
    return F != kFlagsRun || kind < PE_PAIR_MIN_CTAS_GENERAL ? kind : PE_PAIR_MIN_CTAS_GENERAL;
}
// Persistent kernel of the paired form: 128 threads cover a tile of 256 electrons.  kHold: the lanes of a warp wait
// for one another's emissions (pair_loop_hold).
template <bool kSingle, int G, int F, bool kHold>
__global__ void __launch_bounds__(128, (pair_min_ctas<G, F>())) k_step_pair(TablesDev t, BatchDevT<float> b, int steps) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ RunDevT<float> s_run;
    const PairShared S(smem, t.n_eta);
    S.init(t);
    S.load_sigma(t, b.sig_stride, b.runs[0].iz);
    __syncthreads();
    const SumsCta acc = S.acc();
    const Held held = S.slots();

    const int64_t n_tiles = b.tile_start[b.n_runs];
    const uint32_t per_tile = 2u * (uint32_t)b.tile * (uint32_t)steps;   // most emissions of a tile (kMaxLaunchSteps)
    uint32_t since = 0;                                                 // and since the last flush
    int cur = -1;
    int run_idx = 0;
    for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        if (!kSingle) {
            while (run_idx + 1 < b.n_runs && b.tile_start[run_idx + 1] <= tile) ++run_idx;
            if (run_idx != cur) {
                if (cur >= 0) { S.flush(s_run); since = 0; }
                constexpr int kWords = sizeof(RunDevT<float>) / 4;
                for (int w = threadIdx.x; w < kWords; w += blockDim.x)
                    reinterpret_cast<uint32_t*>(&s_run)[w] = reinterpret_cast<const uint32_t*>(&b.runs[run_idx])[w];
                if (!b.sig_stride) S.load_sigma(t, 0, b.runs[run_idx].iz);
                __syncthreads();
                cur = run_idx;
            }
        }
        const RunDevT<float>& r = kSingle ? b.runs[0] : s_run;
        if (since > kSumsMax - per_tile) { S.flush(r); since = 0; }
        since += per_tile;
        const int64_t base = (tile - b.tile_start[run_idx]) * b.tile;
        const int64_t i0 = base + threadIdx.x, i1 = base + threadIdx.x + blockDim.x;
        tile_steps_pair<G, F, kSingle, kHold>(t, r, S.h, S.sig + (size_t)r.iz * b.sig_stride, i0, i1, steps, acc, held, S.tally);
    }
    if (kSingle) {
        if (n_tiles > 0) S.flush(b.runs[0]);
    } else if (cur >= 0) {
        S.flush(s_run);
    }
}


// ---------------------------------------------------------------------------
// Streaming form for launches of a few steps (the state round-trips HBM every launch).
// Each thread takes two adjacent electrons (2j, 2j + 1) of a 256-electron tile, so one
// 16-byte vector covers both position pairs (and both optical-depth pairs) and one 8-byte
// vector both values of each momentum component.  Each thread prefetches its two
// electrons of the CTA's next tile into its own slots of a shared-memory stage with
// per-thread asynchronous copies (cp.async, 16 and 8 bytes) while it steps the current
// tile, and waits only for its own copies (cp.async.wait_group): no barrier, no spin-wait.
// Results go back with streaming vector stores.  The arithmetic is that of the resident
// kernel (the paired step is elementwise in its two electrons), so the results are the
// same bit for bit.  Single run; the ragged end (an odd last electron) and the event words
// use plain loads.
// ---------------------------------------------------------------------------
constexpr int kStreamTile = 256;                       // electrons per tile (128 threads x 2)
constexpr int kStreamThreads = kStreamTile / 2;
// Measured on 6e6 / 1e6 electrons, 20 calls of one step in the rising pulse (us a call, the restore of the state included):
// CTAs x stages 4 x 2 75 / 20.7, 4 x 3 75 / 20.9, 3 x 3 78 / 21.7, 5 x 2 84 / 20.9; at the start, without the queue below
// and the overlapped launches, 5 x 2 120 / 30. The state's round trip is 49 us at the copy bandwidth.
#ifndef PE_STREAM_STAGES
#define PE_STREAM_STAGES 2    // stages per CTA: tiles in flight = stages - 1
#endif
#ifndef PE_STREAM_MIN_CTAS
#define PE_STREAM_MIN_CTAS 4  // resident CTAs of 128 threads per SM the registers are sized for
#endif
// What a launch of one step does and an instance's stages and resident CTAs.  The instances that read the flags at run time
// need more registers than 4 CTAs leave them: 6e6 electrons, us a step, with a box / by null collisions / without brems /
// neither process: 4 CTAs x 2 stages 83.8 / 86.2 / 79.1 / 68.3, 3 x 3 83.8 / 82.8 / 75.4 / 56.0, 4 x 3 88 / 90 / 82 / 73, 5 x 2
// 91 / 92 / 82 / 71, and with the queue below (spilled) 104 / 105 / 92 / 74; on 1e6 electrons 21.0 / 21.1 / 19.4 / 12.3 and
// 21.9 / 21.5 / 20.1 / 10.9.  In launches of 2 to 4 steps they keep 4 x 2 (1e6 electrons 11.3 / 10.7 / 9.5 / 5.1, 3 x 3 12.7 /
// 12.0 / 10.7 / 5.2).
template <int F, bool kOne>
struct StreamShape {
    static constexpr bool kQueue = kOne && F == kFlagsPaper;
    static constexpr int kStages = kOne && F != kFlagsPaper ? 3 : PE_STREAM_STAGES;
    static constexpr int kCtas = kOne && F != kFlagsPaper ? 3 : PE_STREAM_MIN_CTAS;
};
// one stage: x pairs (float4 per thread), tau pairs (float4), ux, uy, uz (float2 each), and in the instances that may have
// null collisions the waits (uint2)
template <int F>
constexpr int kStageBytes = kStreamThreads * (16 + 16 + 8 + 8 + 8 + (F == kFlagsRun ? 8 : 0));

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async8(uint32_t dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// all of this thread's copy groups but the most recent `n` have landed
template <int n>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(n) : "memory"); }

// this thread's slots of a stage
struct StageSlots {
    uint32_t x, tau, ux, uy, uz, wait; // shared addresses (for the copies)
    const float4* px;                  // generic pointers (for the reads)
    const float4* ptau;
    const float2 *pux, *puy, *puz;
    const uint2* pwait;
};
__device__ __forceinline__ StageSlots stage_slots(unsigned char* stage, int t) {
    StageSlots q;
    unsigned char* b = stage;
    q.px = reinterpret_cast<const float4*>(b) + t;
    q.ptau = reinterpret_cast<const float4*>(b + kStreamThreads * 16) + t;
    q.pux = reinterpret_cast<const float2*>(b + kStreamThreads * 32) + t;
    q.puy = reinterpret_cast<const float2*>(b + kStreamThreads * 40) + t;
    q.puz = reinterpret_cast<const float2*>(b + kStreamThreads * 48) + t;
    q.pwait = reinterpret_cast<const uint2*>(b + kStreamThreads * 56) + t;
    q.wait = smem_addr(q.pwait);
    q.x = smem_addr(q.px); q.tau = smem_addr(q.ptau);
    q.ux = smem_addr(q.pux); q.uy = smem_addr(q.puy); q.uz = smem_addr(q.puz);
    return q;
}
// copies of electrons 2j, 2j + 1 (both present) into the slots
template <int F>
__device__ __forceinline__ void stage_issue(const RunDevT<float>& r, int64_t j, const StageSlots& q) {
    cp_async16(q.x, reinterpret_cast<const float4*>(r.x) + j);
    cp_async16(q.tau, reinterpret_cast<const float4*>(r.tau) + j);
    cp_async8(q.ux, reinterpret_cast<const float2*>(r.ux) + j);
    cp_async8(q.uy, reinterpret_cast<const float2*>(r.uy) + j);
    cp_async8(q.uz, reinterpret_cast<const float2*>(r.uz) + j);
    if (F == kFlagsRun && r.wait) cp_async8(q.wait, reinterpret_cast<const uint2*>(r.wait) + j);
}
// a particle is removed (x NaN, finite momenta), live, or has a non-finite momentum
__device__ __forceinline__ bool finite3(float a, float b, float c) { return isfinite(a) && isfinite(b) && isfinite(c); }

// electrons 2j, 2j + 1 from the slots
template <int F>
__device__ __forceinline__ void stage_take(const RunDevT<float>& r, int64_t j, const StageSlots& q, Pair& Q,
                                           unsigned long long* tally) {
    const float4 x = *q.px, tau = *q.ptau;
    Q.x = make_float2(x.x, x.z);
    Q.x_lo = make_float2(x.y, x.w);
    Q.tau = make_float2(tau.x, tau.z);
    Q.tau_lo = make_float2(tau.y, tau.w);
    Q.u0 = *q.pux;
    Q.u1 = *q.puy;
    Q.u2 = *q.puz;
    Q.y = Q.y_lo = P2(0.0f);
    if (F == kFlagsRun && r.wait) {
        const uint2 w = *q.pwait;
        Q.wait[0] = w.x;
        Q.wait[1] = w.y;
    } else {
        Q.wait[0] = Q.wait[1] = PE_WAIT_NEVER;
    }
    Q.act[0] = !isnan(Q.x.x);
    Q.act[1] = !isnan(Q.x.y);
    if (!finite3(Q.u0.x, Q.u1.x, Q.u2.x) || !finite3(Q.u0.y, Q.u1.y, Q.u2.y)) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {             // rare: remove and count (as live_or_kill; the event word stays)
            Particle<float> P = unpack(Q, k);
            if (finite_momenta(P)) continue;
            kill_nonfinite(P, (uint32_t)r.step0, tally);
            store_one(r, 2 * j + k, P);
            Q.act[k] = false;
            repack(Q, k, P);
        }
    }
}

// electrons 2j, 2j + 1 from memory as pair_store left them (1D)
__device__ __forceinline__ void pair_load(const RunDevT<float>& r, int64_t j, Pair& Q) {
    const float4 x = reinterpret_cast<const float4*>(r.x)[j], tau = reinterpret_cast<const float4*>(r.tau)[j];
    Q.x = make_float2(x.x, x.z);
    Q.x_lo = make_float2(x.y, x.w);
    Q.tau = make_float2(tau.x, tau.z);
    Q.tau_lo = make_float2(tau.y, tau.w);
    Q.u0 = reinterpret_cast<const float2*>(r.ux)[j];
    Q.u1 = reinterpret_cast<const float2*>(r.uy)[j];
    Q.u2 = reinterpret_cast<const float2*>(r.uz)[j];
    Q.y = Q.y_lo = P2(0.0f);
    Q.wait[0] = r.wait ? r.wait[2 * j] : PE_WAIT_NEVER;
    Q.wait[1] = r.wait ? r.wait[2 * j + 1] : PE_WAIT_NEVER;
    Q.act[0] = !isnan(Q.x.x);
    Q.act[1] = !isnan(Q.x.y);
}

// electrons 2j, 2j + 1 back to memory (both present; removed ones were stored when removed)
__device__ __forceinline__ void pair_store(const RunDevT<float>& r, int64_t j, const Pair& Q, bool st0, bool st1) {
    if (st0 && st1) {
        __stcs(reinterpret_cast<float4*>(r.x) + j, make_float4(Q.x.x, Q.x_lo.x, Q.x.y, Q.x_lo.y));
        __stcs(reinterpret_cast<float4*>(r.tau) + j, make_float4(Q.tau.x, Q.tau_lo.x, Q.tau.y, Q.tau_lo.y));
        __stcs(reinterpret_cast<float2*>(r.ux) + j, Q.u0);
        __stcs(reinterpret_cast<float2*>(r.uy) + j, Q.u1);
        __stcs(reinterpret_cast<float2*>(r.uz) + j, Q.u2);
        if (r.wait) reinterpret_cast<uint2*>(r.wait)[j] = make_uint2(Q.wait[0], Q.wait[1]);
    } else {
        if (st0) store_one(r, 2 * j, unpack(Q, 0));
        if (st1) store_one(r, 2 * j + 1, unpack(Q, 1));
    }
}

// pairs of a warp whose emissions wait (fewer than 32 left by the last tile and at most 32 more): pair, crossings, eta
struct StreamQueue {
    int64_t j[64];
    float2 eta[64];
    uint32_t crossed[64];
};

// kOne: launches of one step.  With kQueue a pair with an emission is then stored as it is after the push and queued by its warp,
// which takes the queue 32 emissions at a time, the rest when its tiles are done, and goes through the rest of the step
// with them, so an emission is not issued for one or two lanes of every third tile (the same job 87 us a call at 5 x 2 without the queue).
template <int G, int F, bool kOne>
__global__ void __launch_bounds__(kStreamThreads, (StreamShape<F, kOne>::kCtas)) k_step_pair_stream(TablesDev t, BatchDevT<float> b,
                                                                                         int steps) {
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr bool kQueue = StreamShape<F, kOne>::kQueue;
    constexpr int kStages = StreamShape<F, kOne>::kStages;
    __shared__ StreamQueue s_queue[kQueue ? kStreamThreads / 32 : 1];
    const PairShared S(smem, t.n_eta);
    // the stages on a 16-byte boundary after the tables
    const uint32_t table_bytes = kPairFixedBytes + 4 * (t.n_eta + (b.sig_stride ? t.n_Z * t.n_E : t.n_E));
    unsigned char* stage_buf = smem + ((table_bytes + 15u) & ~15u);
    const RunDevT<float>& r = b.runs[0];
    S.init(t);
    S.load_sigma(t, b.sig_stride, r.iz);
    __syncthreads();
    // what follows reads the state: the launch of this kernel may overlap the end of the one before
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const SumsCta acc = S.acc();                        // at most 2^31 / grid electrons, 4 steps: far below kSumsMax

    const int64_t n_tiles = b.tile_start[1];
    const int64_t n_pairs = r.n >> 1;                   // j < n_pairs: electrons 2j and 2j + 1 both present
    const int64_t stride = (int64_t)gridDim.x * kStreamThreads;
    const float* sig_z = S.sig + (size_t)r.iz * b.sig_stride;
    const uint32_t n0 = (uint32_t)r.step0;
    const int lane = threadIdx.x & 31;
    StreamQueue& W = s_queue[kQueue ? threadIdx.x >> 5 : 0];
    int queued = 0;                                     // pairs in W (the same on every lane)
    float2 n_above = P2(0.0f);
    // the rest of the step after the optical depth, and the pair back to memory
    auto finish = [&](int64_t j, Pair& Q, float2 gamma, float2 inv_g) {
        const uint32_t id[2] = {r.id0 + (uint32_t)(2 * j), r.id0 + (uint32_t)(2 * j + 1)};
        if (brems_on<F>(r)) {
            const unsigned hit = brems_pair<G, F>(t, r, sig_z, id, n0, Q, gamma, inv_g, acc);
            if (hit) emit_brems_pair<G, F>(t, r, sig_z, id, n0, hit, Q, gamma, inv_g, acc);
        }
        move_pair<G>(r.c, Q, inv_g);
        if (box_on<F>(r)) box_pair<G>(r, 2 * j, 2 * j + 1, n0, Q, S.tally);
        pair_store(r, j, Q, Q.act[0], Q.act[1]);
    };
    // the last `count` queued pairs, one to a lane
    auto drain = [&](int count) {
        if (lane < count) {
            const int at = queued - count + lane;
            const int64_t j = W.j[at];
            Pair Q;
            pair_load(r, j, Q);
            float2 gamma, inv_g;
            gamma_pair(Q, gamma, inv_g);
            const uint32_t id[2] = {r.id0 + (uint32_t)(2 * j), r.id0 + (uint32_t)(2 * j + 1)};
            emit_ncs_pair<G, false>(t, r, id, n0, W.crossed[at], Q, gamma, inv_g, W.eta[at], acc);
            finish(j, Q, gamma, inv_g);
        }
        queued -= count;
        __syncwarp();
    };
    // tile k of this CTA (k = 0, 1, ...) is tile blockIdx.x + k gridDim.x, staged in stage k mod S;
    // the copies of tiles k + 1 .. k + S - 1 are in flight while tile k is stepped
    const int64_t j0 = (int64_t)blockIdx.x * kStreamThreads + threadIdx.x;
#pragma unroll
    for (int k = 0; k < kStages - 1; ++k) {
        const int64_t jk = j0 + k * stride;
        if (jk < n_pairs) stage_issue<F>(r, jk, stage_slots(stage_buf + k * kStageBytes<F>, threadIdx.x));
        cp_async_commit();
    }
    int stage = 0;
    for (int64_t j = j0; j - threadIdx.x < n_tiles * kStreamThreads; j += stride) {
        const int64_t jn = j + (kStages - 1) * stride;
        const int sn = stage == 0 ? kStages - 1 : stage - 1;       // (stage + S - 1) mod S
        if (jn < n_pairs) stage_issue<F>(r, jn, stage_slots(stage_buf + sn * kStageBytes<F>, threadIdx.x));
        cp_async_commit();
        cp_async_wait<kStages - 1>();             // this thread's copies of the current tile
        Pair Q;
        const bool full = j < n_pairs;
        if (full) {
            stage_take<F>(r, j, stage_slots(stage_buf + stage * kStageBytes<F>, threadIdx.x), Q, S.tally);
        } else {
            pair_clear(Q);
            if (2 * j < r.n) load_one(r, 2 * j, Q, 0, S.tally);   // the odd last electron
        }
        if constexpr (kQueue) {
            unsigned crossed = 0;
            float2 gamma, inv_g, eta;
            const bool act = full && (Q.act[0] || Q.act[1]);
            if (act) crossed = push_pair<G, F>(t, r, S.h, (float)n0, Q, gamma, inv_g, eta, n_above);
            const unsigned mask = __ballot_sync(0xffffffffu, crossed != 0);
            if (crossed) {
                const int at = queued + __popc(mask & ((1u << lane) - 1u));
                W.j[at] = j;
                W.eta[at] = eta;
                W.crossed[at] = crossed;
                pair_store(r, j, Q, Q.act[0], Q.act[1]);
            } else if (act) {
                finish(j, Q, gamma, inv_g);
            }
            queued += __popc(mask);
            __syncwarp();
            if (queued >= 32) drain(32);
            if (!full && Q.act[0]) {                    // the odd last electron, alone
                pair_loop<G, F, false, true>(t, r, S.h, sig_z, 2 * j, 2 * j + 1, Q, 1, acc, S.tally);
                pair_store(r, j, Q, Q.act[0], false);
            }
        } else {
            const bool live0 = 2 * j < r.n, live1 = full;
            pair_loop<G, F, false, true>(t, r, S.h, sig_z, 2 * j, 2 * j + 1, Q, steps, acc, S.tally);
            pair_store(r, j, Q, live0 && Q.act[0], live1 && Q.act[1]);
        }
        stage = stage + 1 == kStages ? 0 : stage + 1;
    }
    cp_async_wait<0>();
    if constexpr (kQueue) {
        if (queued) drain(queued);
        const unsigned int na = __float2uint_rz(n_above.x) + __float2uint_rz(n_above.y);
        if (na) atomicAdd(S.tally + PE_T_N_ETA_ABOVE, (unsigned long long)na);
    }
    if (n_tiles > 0) S.flush(r);
}

}  // namespace pe
