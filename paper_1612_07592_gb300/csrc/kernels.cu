// kernels.cu -- the init kernel, the diagnostics kernels and their launchers.  The
// step kernels are instantiated per precision in kernels_paired.cu (FP32) and kernels_f64.cu.
#include <algorithm>
#include <climits>
#include <cmath>

#include "kernels.cuh"

namespace pe {

// ---------------------------------------------------------------------------
// init kernel
// ---------------------------------------------------------------------------
template <typename R>
__global__ void __launch_bounds__(256) k_init(RunDevT<double> r, int init_dist, double theta, double beam_u) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= r.n) return;
    uint32_t id = r.id0 + (uint32_t)i;
    uint4 w = draw(r, id, 0, PUR_TAU0);
    double tau0 = -log(uni53(w64(w.x, w.y)));
    if (sizeof(R) == 4) {
        float hi = (float)tau0;
        ((float2*)r.tau)[i] = make_float2(hi, (float)(tau0 - (double)hi));
    } else {
        ((double*)r.tau)[i] = tau0;
    }
    if (r.wait) {
        uint4 v = draw(r, id, 0, PUR_WAIT);
        r.wait[i] = wait_draw(r.x_hat, v.x, v.y);
    }
    if (init_dist == PE_CALLER) return;
    uint4 p = draw(r, id, 0, PUR_POS);
    const StepC<double>& c = r.c;
    // a beam enters at the front face of the slab
    double x = (init_dist == PE_BEAM) ? c.x0 : c.x0 + (c.x1 - c.x0) * uni32(p.x);
    double y = (r.geometry == PE_GAUSS_2D) ? -c.yh + 2.0 * c.yh * uni32(p.y) : 0.0;
    double u0 = 0, u1 = 0, u2 = 0;
    if (init_dist == PE_MAXWELL_JUTTNER) {
        // Sobol (1976) rejection sampling of the Maxwell-Juttner momentum magnitude
        double um = 0.0;
        for (uint32_t round = 0; round < 64; ++round) {
            uint4 m = draw(r, id, 0, PUR_MJ + round);
            double X1 = uni32(m.x), X2 = uni32(m.y), X3 = uni32(m.z), X4 = uni32(m.w);
            double uu = -theta * log(X1 * X2 * X3);
            double ee = -theta * log(X1 * X2 * X3 * X4);
            if (ee * ee - uu * uu > 1.0) { um = uu; break; }
        }
        double X5 = uni32(p.z), X6 = uni32(p.w);
        double sn = 2.0 * sqrt(X5 * (1.0 - X5));
        double sphi, cphi;
        sincos(2.0 * kPi * X6, &sphi, &cphi);
        u0 = um * (2.0 * X5 - 1.0);
        u1 = um * sn * cphi;
        u2 = um * sn * sphi;
    } else if (init_dist == PE_BEAM) {
        u0 = beam_u;
    }
    if (sizeof(R) == 4) {
        float xh = (float)x, yh = (float)y;
        ((float2*)r.x)[i] = make_float2(xh, (float)(x - (double)xh));
        ((float2*)r.y)[i] = make_float2(yh, (float)(y - (double)yh));
    } else {
        ((double*)r.x)[i] = x;
        ((double*)r.y)[i] = y;
    }
    ((R*)r.ux)[i] = (R)u0;
    ((R*)r.uy)[i] = (R)u1;
    ((R*)r.uz)[i] = (R)u2;
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
void launch_init(const RunDev& r, int precision, int init_dist, double theta, double beam_u, cudaStream_t s) {
    if (r.n == 0) return;
    int grid = (int)((r.n + 255) / 256);
    if (precision == PE_F32)
        k_init<float><<<grid, 256, 0, s>>>(r, init_dist, theta, beam_u);
    else
        k_init<double><<<grid, 256, 0, s>>>(r, init_dist, theta, beam_u);
}

size_t rate_table_bytes(const TablesDev& t, int precision) {
    return (precision == PE_F32 ? 4 : 8) * (t.n_eta + (size_t)t.n_Z * t.n_E);
}

}  // namespace pe

namespace pe {

// ---------------------------------------------------------------------------
// diagnostics: electron energy spectrum (Fig. 5) and photon (x, energy) map (Fig. 4)
// ---------------------------------------------------------------------------
// bin of v in [lo, hi) on log bins: -1 below, n_bins at or above
__device__ __forceinline__ int log_bin(double v, double ln_lo, double inv_dln, int n_bins) {
    if (!(v > 0.0)) return -1;
    const double b = (log(v) - ln_lo) * inv_dln;
    if (b < 0.0) return -1;
    return b >= (double)n_bins ? n_bins : (int)b;
}

// Both diagnostics bin in FP64, on GB300's narrow pipe (a logarithm and a square root are some 130 of its instructions,
// each 64 clocks of a scheduler).  Nearly every value is far enough from a bin edge for a float position with a known
// error to name the same bin, so the FP64 form runs only for the values within that error of an edge (or outside
// the float form's range): same counts.  3e6 electrons into 200 bins and 2.5e5 photons into 200 x 64: 341 us for both
// calls with every value in FP64, now 35 (the reads are 10 us at the copy bandwidth, the two clears and launches most of
// the rest).
struct FastBin {
    float ln_lo, inv_dln, eps;     // position = (ln v - ln_lo) inv_dln, off by at most eps + 3e-7 |position|
};
// bin of e (in units of m c^2; scale = ln of m c^2 in MeV) or kUnsure.  Errors of ln v - ln_lo for e < 2^25 (17 TeV):
// e itself 6e-7 relative, lg2.approx 2^-22 of its result (4.2e-6) and the result's rounding to float (0.7e-6), the FMA's
// rounding (1e-6): below 6.5e-6, taken as 8e-6 in eps; the difference's and ln_lo's own rounding are in eps's other terms.
// Further up the logarithm's documented error grows with its result, beyond eps: those bins are the FP64 form's.
constexpr int kUnsure = INT_MIN;
__device__ __forceinline__ int fast_log_bin(const FastBin& f, float e, float scale) {
    if (!(e > 1e-6f && e < 0x1p25f)) return kUnsure;
    const float pos = (fmaf(__log2f(e), 0.693147180559945309f, scale) - f.ln_lo) * f.inv_dln;
    const float fl = floorf(pos), w = pos - fl, eps = f.eps + 3e-7f * fabsf(pos);
    return w > eps && w < 1.0f - eps && fabsf(pos) < 1e6f ? (int)fl : kUnsure;
}

template <typename R>
__device__ __forceinline__ void spectrum_one(float x_hi, R u0, R u1, R u2, const FastBin& f, double ln_lo,
                                             double inv_dln, int n_bins, unsigned int* s_bins) {
    if (isnan(x_hi)) return;
    const float a = (float)u0, b = (float)u1, c = (float)u2;
    const float uu = fmaf(c, c, fmaf(b, b, a * a));
    // gamma - 1 = u^2 / (1 + gamma); below 1e-6 the FP64 form's own cancellation decides the bin
    int k = fast_log_bin(f, uu / (1.0f + sqrtf(1.0f + uu)), -0.671387683f);
    if (k == kUnsure) {
        const double d0 = u0, d1 = u1, d2 = u2;
        const double ek = (sqrt(1.0 + d0 * d0 + d1 * d1 + d2 * d2) - 1.0) * kMec2MeV;   // kinetic energy, MeV
        k = log_bin(ek, ln_lo, inv_dln, n_bins);
    }
    if (k >= 0 && k < n_bins) atomicAdd(&s_bins[k], 1u);
}

// Counts in 32-bit words of the CTA (native shared atomics; at most 2^31 / grid electrons).  FP32 state: four electrons
// to a thread, 16-byte loads (the buffers are 16-byte aligned).
template <typename R>
__global__ void __launch_bounds__(256) k_electron_spectrum(RunDevT<double> r, double ln_lo, double inv_dln, int n_bins,
                                                           FastBin f, unsigned long long* out) {
    extern __shared__ unsigned int s_bins[];
    for (int k = threadIdx.x; k < n_bins; k += blockDim.x) s_bins[k] = 0;
    __syncthreads();
    const int64_t first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    if constexpr (sizeof(R) == 4) {
        const int64_t quads = r.n >> 2;
        for (int64_t q = first; q < quads; q += stride) {
            const float4 xa = ((const float4*)r.x)[2 * q], xb = ((const float4*)r.x)[2 * q + 1];
            const float4 u0 = ((const float4*)r.ux)[q], u1 = ((const float4*)r.uy)[q], u2 = ((const float4*)r.uz)[q];
            spectrum_one<float>(xa.x, u0.x, u1.x, u2.x, f, ln_lo, inv_dln, n_bins, s_bins);
            spectrum_one<float>(xa.z, u0.y, u1.y, u2.y, f, ln_lo, inv_dln, n_bins, s_bins);
            spectrum_one<float>(xb.x, u0.z, u1.z, u2.z, f, ln_lo, inv_dln, n_bins, s_bins);
            spectrum_one<float>(xb.z, u0.w, u1.w, u2.w, f, ln_lo, inv_dln, n_bins, s_bins);
        }
        const int64_t i = 4 * quads + first;
        if (i < r.n)
            spectrum_one<float>(((const float2*)r.x)[i].x, ((const float*)r.ux)[i], ((const float*)r.uy)[i],
                                ((const float*)r.uz)[i], f, ln_lo, inv_dln, n_bins, s_bins);
    } else {
        for (int64_t i = first; i < r.n; i += stride)
            spectrum_one<R>(isnan(((const double*)r.x)[i]) ? __int_as_float(0x7fc00000) : 0.0f, ((const R*)r.ux)[i],
                            ((const R*)r.uy)[i], ((const R*)r.uz)[i], f, ln_lo, inv_dln, n_bins, s_bins);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < n_bins; k += blockDim.x)
        if (s_bins[k]) atomicAdd(out + k, (unsigned long long)s_bins[k]);
}

__global__ void __launch_bounds__(256) k_photon_map(const uint8_t* photons, const unsigned long long* tally,
                                                    int64_t capacity, double x_lo, double inv_dx, int nx,
                                                    double ln_lo, double inv_dln, int ne, FastBin f, float fx_lo,
                                                    float finv_dx, float eps_x, unsigned long long* out) {
    const unsigned long long appended = tally[PE_T_N_PHOTONS];
    const int64_t count = appended < (unsigned long long)capacity ? (int64_t)appended : capacity;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
        const float4 a = reinterpret_cast<const float4*>(photons + i * 32)[0];   // x, y, energy (m c^2), kx
        // x position: the difference and the product round by 1.2e-7 relative, fx_lo by 6e-8 of x_lo (eps_x)
        const float px = (a.x - fx_lo) * finv_dx, fl = floorf(px), w = px - fl, eps = eps_x + 3e-7f * fabsf(px);
        int xb, eb = fast_log_bin(f, a.z, -0.671387683f);
        if (w > eps && w < 1.0f - eps && fabsf(px) < 1e6f) {
            xb = (int)fl;
        } else {
            const double xd = ((double)a.x - x_lo) * inv_dx;
            if (!(xd >= 0.0) || xd >= (double)nx) continue;
            xb = (int)xd;
        }
        if (xb < 0 || xb >= nx) continue;
        if (eb == kUnsure) eb = log_bin((double)a.z * kMec2MeV, ln_lo, inv_dln, ne);
        if (eb < 0 || eb >= ne) continue;
        atomicAdd(out + (size_t)xb * ne + eb, 1ull);
    }
}

static FastBin fast_bin(double ln_lo, double inv_dln) {
    // ln v's error and ln_lo's own rounding to float
    return FastBin{(float)ln_lo, (float)inv_dln, (float)(inv_dln * (8e-6 + 1.2e-7 * std::fabs(ln_lo)))};
}

void launch_electron_spectrum(const RunDev& r, int precision, double e_lo, double e_hi, int n_bins,
                              unsigned long long* out, cudaStream_t s) {
    const double ln_lo = std::log(e_lo), inv_dln = n_bins / (std::log(e_hi) - std::log(e_lo));
    const int64_t threads = precision == PE_F32 ? (r.n + 3) / 4 : r.n;
    const int grid = (int)std::min<int64_t>((threads + 255) / 256, 1024);
    if (grid <= 0) return;
    const size_t smem = sizeof(unsigned int) * (size_t)n_bins;
    const FastBin f = fast_bin(ln_lo, inv_dln);
    if (precision == PE_F32) k_electron_spectrum<float><<<grid, 256, smem, s>>>(r, ln_lo, inv_dln, n_bins, f, out);
    else k_electron_spectrum<double><<<grid, 256, smem, s>>>(r, ln_lo, inv_dln, n_bins, f, out);
}

void launch_photon_map(const RunDev& r, double x_lo, double x_hi, int nx, double e_lo, double e_hi, int ne,
                       unsigned long long* out, cudaStream_t s) {
    if (r.capacity <= 0) return;
    // the stored count is read on the device: a grid-stride launch sized for the capacity
    const int grid = (int)std::min<int64_t>((r.capacity + 255) / 256, 2048);
    const double ln_lo = std::log(e_lo), inv_dln = ne / (std::log(e_hi) - std::log(e_lo)), inv_dx = nx / (x_hi - x_lo);
    k_photon_map<<<grid, 256, 0, s>>>(r.photons, r.tally, r.capacity, x_lo, inv_dx, nx, ln_lo, inv_dln, ne,
                                      fast_bin(ln_lo, inv_dln), (float)x_lo, (float)inv_dx,
                                      (float)(inv_dx * 1.2e-7 * std::fabs(x_lo) + 1e-7), out);
}

}  // namespace pe
