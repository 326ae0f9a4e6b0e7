// Single electrons in analytic plane waves, many at once: the paper's
// validation path (Sec. 3), batched over scans of amplitude and initial
// momentum.  One thread integrates one electron in double precision (a
// reference integrator, not the PIC hot path):
//   - the leapfrog pusher of Sec. 3: Boris rotation for the Lorentz force plus
//     the RR kick of Eqs. (f_r, pertfull, estim1, estimgamma), fields at
//     (t_n, x^n), then x^{n+1} = x^n + dt v_x^{n+1/2};
//   - classical RK4 on the lab-frame LL equation, Eq. (3dLL), with or without
//     its field-derivative term.
// Plane waves travel along +x with phase phi = t - x and B = x_hat x E:
//   wave 0: LP, Ey = a0 cos(phi);
//   wave 1: CP, (Ey, Ez) = (a0/sqrt2)(cos(phi), sin(phi));
//   wave 2: LP pulse, Ey = a0 sin^2(pi phi/tau) cos(phi) for 0 <= phi <= tau.
// Bound: FP64 issue.  An FP64 warp instruction occupies its scheduler for 64 cycles,
// whatever the number of active lanes (RK4 on 4096 electrons took the same time as
// 128 warps of 32 and as 512 warps of 8), so a step's time is its FP64 instructions,
// and few of them are needed:
//   - in a plane wave B = x_hat x E the terms of the force collapse (ll_force),
//   - reciprocals of square roots and of sums come from the approximate instructions
//     and one third-order correction (5 and 3 operations) in the place of square
//     roots and quotients, sine and cosine from their series,
//   - wave, radiation reaction and derivative term are template arguments, electrons
//     are grouped by wave, so that a warp has one kind, and every warp is a block of
//     its own, so that a few thousand electrons spread over all SMs,
//   - when there are schedulers to spare, four lanes take one electron: all of them
//     hold its state, and each evaluates one of the sines and cosines of a stage (the
//     pulse needs four).
// 4096 electrons x 2000 RK4 steps: 47.1 -> 18.5 ms; 20,000 x 1000 leapfrog steps:
// 15.6 -> 4.5 ms.
#include <new>
#include <string>
#include <vector>

#include "picrr.h"
#include "picrr_internal.cuh"

namespace picrr {

namespace {

constexpr int ELEC_T = 32;  // a warp of electrons in one kind of wave
constexpr double kPiD = 3.14159265358979323846;

struct Wave {
    double a0, tau, k;  // k = pi / tau
};

// 1/sqrt(a) and 1/a to about one unit in the last place (a >= 1): from the hardware's
// approximation y with e = 1 - a y^2 (1 - a y), |e| <= 2^-19, by the series of
// (1 - e)^(-1/2) ((1 - e)^-1) up to e^2.
__device__ __forceinline__ double or_zero_at_inf(double a, double y) {
    return __double2hiint(a) == 0x7ff00000 && __double2loint(a) == 0 ? 0.0 : y;
}
__device__ __forceinline__ double rsqrt_f64(double a) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
    const double e = fma(-(a * y), y, 1.0);
    return or_zero_at_inf(a, fma(y * e, fma(0.375, e, 0.5), y));
}
__device__ __forceinline__ double rcp_f64(double a) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
    const double e = fma(-a, y, 1.0);
    return or_zero_at_inf(a, fma(y, fma(e, e, e), y));
}

constexpr double PHASE_MAX = 1e6;  // phases below this take the short reduction

// sin (shift 0) or cos (shift 1) of |x| < PHASE_MAX: x - q pi/2 with pi/2 in two
// doubles (the first product's difference is exact below 2^20 quadrants), then the
// Taylor series of the sine or cosine on |r| <= pi/4 (remainders r^19/19! and
// r^18/18!, below 2^-58); which one is decided by selecting the coefficients.
__device__ __forceinline__ double sin_shifted(double x, int shift) {
    const double magic = 6755399441055744.0;  // 1.5 * 2^52: adds round to whole numbers
    const double t = fma(x, 0.63661977236758134308, magic);
    const int q = __double2loint(t) + shift;
    const double kd = t - magic;
    const double r = fma(kd, -6.123233995736766036e-17, fma(kd, -1.57079632679489661923, x));
    const double z = r * r;
    const bool odd = q & 1;  // cosine series: 1 + z (-1/2! + z (1/4! - ...)); sine: r + r z (-1/3! + ...)
    double p = fma(z, odd ? 1.0 / 20922789888000.0 : 1.0 / 355687428096000.0,
                   odd ? -1.0 / 87178291200.0 : -1.0 / 1307674368000.0);
    p = fma(z, p, odd ? 1.0 / 479001600.0 : 1.0 / 6227020800.0);
    p = fma(z, p, odd ? -1.0 / 3628800 : -1.0 / 39916800.0);
    p = fma(z, p, odd ? 1.0 / 40320 : 1.0 / 362880);
    p = fma(z, p, odd ? -1.0 / 720 : -1.0 / 5040);
    p = fma(z, p, odd ? 1.0 / 24 : 1.0 / 120);
    p = fma(z, p, odd ? -0.5 : -1.0 / 6);
    const double a = odd ? 1.0 : r;
    const double v = fma(a * z, p, a);
    return q & 2 ? -v : v;
}

// What a stage needs of sin(phi), cos(phi), sin(theta), cos(theta): the last two with
// SE and CE only.  With 4 lanes an electron's lane j evaluates the j-th of them.
template <int LANES, bool SHORT, bool S, bool SE, bool CE>
__device__ __forceinline__ void sines(double phi, double theta, double& s, double& c, double& se, double& ce) {
    s = c = se = ce = 0.0;
    if constexpr (!SHORT) {
        sincos(phi, &s, &c);
        if constexpr (SE) sincos(theta, &se, &ce);
    } else if constexpr (LANES == 1 || !(S || SE)) {
        if constexpr (S) s = sin_shifted(phi, 0);
        c = sin_shifted(phi, 1);
        if constexpr (SE) se = sin_shifted(theta, 0);
        if constexpr (CE) ce = sin_shifted(theta, 1);
    } else {
        const int lane = threadIdx.x & 31, j = lane & 3;
        const unsigned quad = 0xfu << (lane & ~3);  // the lanes of this electron, which branch alike
        const double v = sin_shifted(SE && (j & 2) ? theta : phi, j & 1);
        if constexpr (S) s = __shfl_sync(quad, v, 0, 4);
        c = __shfl_sync(quad, v, 1, 4);
        if constexpr (SE) se = __shfl_sync(quad, v, 2, 4);
        if constexpr (CE) ce = __shfl_sync(quad, v, 3, 4);
    }
}

// E(phi) and, with DERIV, dE/dphi (x component zero); B = (0, -Ez, Ey).  Ez is zero
// but for kind 1.
template <int KIND, bool DERIV, int LANES, bool SHORT>
__device__ __forceinline__ void wave_at(const Wave& w, double phi, double& ey, double& ez, double& dey, double& dez) {
    double s, c, se, ce;
    ez = dey = dez = 0.0;
    if constexpr (KIND == 0) {
        sines<LANES, SHORT, DERIV, false, false>(phi, 0.0, s, c, se, ce);
        ey = w.a0 * c;
        if constexpr (DERIV) dey = -w.a0 * s;
    } else if constexpr (KIND == 1) {
        sines<LANES, SHORT, true, false, false>(phi, 0.0, s, c, se, ce);
        const double a = w.a0 * 0.70710678118654752440;
        ey = a * c;
        ez = a * s;
        dey = -ez;
        dez = ey;
    } else {
        // outside the pulse the field is zero at any phase, infinities and NaN too
        const bool in = phi >= 0.0 && phi <= w.tau;
        const double at = in ? phi : 0.0;
        sines<LANES, SHORT, DERIV, true, DERIV>(at, w.k * at, s, c, se, ce);
        const double h = in ? w.a0 * se : 0.0;
        ey = h * se * c;
        if constexpr (DERIV) dey = h * (2.0 * w.k * ce * c - se * s);
    }
}

// Lab-frame LL force of Eq. (3dLL) on an electron (charge -1) with momentum p
// in the wave at phase phi.  With B = x_hat x E and u = 1 - v_x:
//   E + v x B = (v.E, u Ey, u Ez), so (E + v x B)^2 - (v.E)^2 = u^2 E^2,
//   (E + v x B) x B + (v.E) E = (u E^2, 0, 0),
// and (d/dt + v.grad) of a field of t - x is u d/dphi.
template <int KIND, bool RR, bool DERIV, int LANES, bool SHORT>
__device__ __forceinline__ void ll_force(const Wave& w, double phi, const double p[3], double eps, double f[3],
                                         double* vx_out) {
    const double g2 = 1.0 + p[0] * p[0] + p[1] * p[1] + p[2] * p[2], ig = rsqrt_f64(g2);
    const double vx = p[0] * ig, vy = p[1] * ig, vz = p[2] * ig;
    double ey, ez, dey, dez;
    wave_at<KIND, DERIV, LANES, SHORT>(w, phi, ey, ez, dey, dez);
    const double u = 1.0 - vx;
    double fx, fy, fz = 0.0;
    if constexpr (KIND == 1) fx = vy * ey + vz * ez;
    else fx = vy * ey;
    if constexpr (DERIV && RR) {
        const double k = eps * (g2 * ig) * u;
        if constexpr (KIND == 1) fx += k * (vy * dey + vz * dez);
        else fx += k * (vy * dey);
        fy = u * (ey + k * dey);
        if constexpr (KIND == 1) fz = u * (ez + k * dez);
    } else {
        fy = u * ey;
        if constexpr (KIND == 1) fz = u * ez;
    }
    if constexpr (RR) {
        double e2 = ey * ey;
        if constexpr (KIND == 1) e2 += ez * ez;
        const double r = eps * (u * e2), sq = g2 * u * r;
        f[0] = (r - sq * vx) - fx;
        f[1] = -(sq * vy) - fy;
        f[2] = KIND == 1 ? -(sq * vz) - fz : -(sq * vz);
    } else {
        f[0] = -fx;
        f[1] = -fy;
        f[2] = -fz;
    }
    *vx_out = vx;
}

template <int KIND, bool RR, bool DERIV, int LANES, bool SHORT>
__device__ __forceinline__ void rk4_step(const Wave& w, double t, double dt, double eps, double& x, double p[3]) {
    const double h = 0.5 * dt, d6 = dt / 6.0;
    const double ph = (t + h) - x;  // phase at the middle of the step, before the electron's motion
    double f1[3], f2[3], f3[3], f4[3], v1, v2, v3, v4, q[3];
    ll_force<KIND, RR, DERIV, LANES, SHORT>(w, t - x, p, eps, f1, &v1);
#pragma unroll
    for (int i = 0; i < 3; ++i) q[i] = p[i] + h * f1[i];
    ll_force<KIND, RR, DERIV, LANES, SHORT>(w, ph - h * v1, q, eps, f2, &v2);
#pragma unroll
    for (int i = 0; i < 3; ++i) q[i] = p[i] + h * f2[i];
    ll_force<KIND, RR, DERIV, LANES, SHORT>(w, ph - h * v2, q, eps, f3, &v3);
#pragma unroll
    for (int i = 0; i < 3; ++i) q[i] = p[i] + dt * f3[i];
    ll_force<KIND, RR, DERIV, LANES, SHORT>(w, (ph + h) - dt * v3, q, eps, f4, &v4);
    x += d6 * ((v1 + v4) + 2.0 * (v2 + v3));
#pragma unroll
    for (int i = 0; i < 3; ++i) p[i] += d6 * ((f1[i] + f4[i]) + 2.0 * (f2[i] + f3[i]));
}

// One step of the pusher of Sec. 3 for an electron: p holds p^{n-1/2} on
// entry and p^{n+1/2} on return; E = (0, ey, ez), B = (0, -ez, ey) at t_n, x^n.
template <int KIND, bool RR>
__device__ __forceinline__ void leapfrog_kick(double p[3], double ey, double ez, double dt, double eps) {
    constexpr bool Z = KIND == 1;  // the wave has an Ez
    const double h = -0.5 * dt;  // q/m (dt/2) for an electron
    // Boris: half E kick, rotation about B, half E kick.  t = (0, -tz, ty) is formed before it is squared or
    // multiplied by a momentum, so that amplitudes above 1e154 do not overflow
    const double mx = p[0], my = p[1] + h * ey, mz = Z ? p[2] + h * ez : p[2];
    const double b = h * rsqrt_f64(1.0 + mx * mx + my * my + mz * mz);
    const double ty = b * ey, tz = Z ? b * ez : 0.0;
    double t2 = 1.0 + ty * ty;
    if constexpr (Z) t2 += tz * tz;
    const double s = 2.0 * rcp_f64(t2);
    // m' = m + m x t ; m+ = m + m' x (s t)
    const double uy = my - mx * ty, uz = Z ? mz - mx * tz : mz;
    double ux = mx + my * ty, ut = uy * ty;
    if constexpr (Z) {
        ux += mz * tz;
        ut += uz * tz;
    }
    const double sx = s * ux;
    const double pLx = mx + s * ut, pLy = (my - sx * ty) + h * ey, pLz = Z ? (mz - sx * tz) + h * ez : mz;
    if constexpr (!RR) {
        p[0] = pLx;
        p[1] = pLy;
        p[2] = pLz;
        return;
    }
    // Eq. (estim1): p(n) = (p_L^{n+1/2} + p^{n-1/2}) / 2; Eq. (estimgamma): gamma(n) from it
    const double qx = 0.5 * (pLx + p[0]), qy = 0.5 * (pLy + p[1]), qz = 0.5 * (pLz + p[2]);
    const double g2 = 1.0 + qx * qx + qy * qy + qz * qz, iq = rsqrt_f64(g2);
    const double vx = qx * iq, vy = qy * iq, vz = qz * iq;
    // Eq. (f_r): f_R = -eps { f_L x B - (v.E) E + gamma^2 [f_L^2 - (v.E)^2] v } with
    // f_L = -(E + v x B); the terms collapse as in ll_force
    double e2 = ey * ey;
    if constexpr (Z) e2 += ez * ez;
    const double u = 1.0 - vx, r = dt * eps * (u * e2), sq = g2 * u * r;
    // Eq. (pertfull): p^{n+1/2} = p_L^{n+1/2} + dt f_R
    p[0] = pLx + (r - sq * vx);
    p[1] = pLy - sq * vy;
    p[2] = pLz - sq * vz;
}

template <int KIND, bool RR, int LANES, bool SHORT>
__device__ __forceinline__ void leapfrog_step(const Wave& w, double t, double dt, double eps, double& x, double p[3]) {
    double ey, ez, dey, dez;
    wave_at<KIND, false, LANES, SHORT>(w, t - x, ey, ez, dey, dez);
    leapfrog_kick<KIND, RR>(p, ey, ez, dt, eps);
    x += dt * p[0] * rsqrt_f64(1.0 + p[0] * p[0] + p[1] * p[1] + p[2] * p[2]);
}

template <int KIND, bool RK4, bool RR, bool DERIV, int LANES>
__device__ void integrate(const pic_electron_case& C, double dt, int64_t nsteps, int every, double eps, double* out,
                          int64_t nsamples) {
    const Wave w{C.a0, C.tau, fmin(kPiD / C.tau, 1e300)};  // (finite, so that 0 times it is 0)
    double x = C.x0, p[3] = {C.p0[0], C.p0[1], C.p0[2]};
    int64_t k = 0;
    int left = every;  // steps to the next row
    for (int64_t s = 0; s < nsteps; ++s) {
        const double t = static_cast<double>(s) * dt;
        // |v| < 1: the phase stays within 2 dt of t - x during a step
        const bool small = fabs(t - x) + 2.0 * dt < PHASE_MAX;
        if constexpr (RK4) {
            if (small) rk4_step<KIND, RR, DERIV, LANES, true>(w, t, dt, eps, x, p);
            else rk4_step<KIND, RR, DERIV, LANES, false>(w, t, dt, eps, x, p);
        } else {
            if (small) leapfrog_step<KIND, RR, LANES, true>(w, t, dt, eps, x, p);
            else leapfrog_step<KIND, RR, LANES, false>(w, t, dt, eps, x, p);
        }
        if (--left == 0) {
            left = every;
            if (k == nsamples) continue;
            double* o = out + 5 * k++;
            if (LANES > 1 && (threadIdx.x & (LANES - 1))) continue;
            o[0] = static_cast<double>(s + 1) * dt;
            o[1] = x;
            o[2] = p[0];
            o[3] = p[1];
            o[4] = p[2];
        }
    }
}

// order: the electrons grouped by kind of wave, each group padded to whole warps (at
// one lane an electron) with -1
template <bool RK4, bool RR, bool DERIV, int LANES>
__global__ void __launch_bounds__(ELEC_T) k_electron(const pic_electron_case* cases, const int32_t* order, double dt,
                                                     int64_t nsteps, int every, double eps, double* out,
                                                     int64_t nsamples) {
    const int64_t c = order[(static_cast<int64_t>(blockIdx.x) * ELEC_T + threadIdx.x) / LANES];
    if (c < 0) return;
    const pic_electron_case C = cases[c];
    out += c * nsamples * 5;
    if (C.wave == 0) integrate<0, RK4, RR, DERIV, LANES>(C, dt, nsteps, every, eps, out, nsamples);
    else if (C.wave == 1) integrate<1, RK4, RR, DERIV, LANES>(C, dt, nsteps, every, eps, out, nsamples);
    else integrate<2, RK4, RR, DERIV, LANES>(C, dt, nsteps, every, eps, out, nsamples);
}

template <int LANES>
void electron_launch(const pic_electron_case* cases, const int32_t* order, int64_t slots, int integrator, int flags,
                     double dt, int64_t nsteps, int every, double eps, double* out, int64_t nsamples, cudaStream_t st) {
    const unsigned g = static_cast<unsigned>(slots / ELEC_T) * LANES;
    const bool rr = (flags & PIC_ELECTRON_RR) != 0, deriv = rr && (flags & PIC_ELECTRON_DERIV) != 0;
#define PICRR_ELECTRON(K, R, D) \
    k_electron<K, R, D, LANES><<<g, ELEC_T, 0, st>>>(cases, order, dt, nsteps, every, eps, out, nsamples)
    if (integrator == PIC_INTEGRATOR_RK4) {
        if (deriv) PICRR_ELECTRON(true, true, true);
        else if (rr) PICRR_ELECTRON(true, true, false);
        else PICRR_ELECTRON(true, false, false);
    } else {
        if (rr) PICRR_ELECTRON(false, true, false);
        else PICRR_ELECTRON(false, false, false);
    }
#undef PICRR_ELECTRON
}

}  // namespace

void launch_electron_scan(const pic_electron_case* cases, const int32_t* order, int64_t slots, int integrator, int flags,
                          double dt, int64_t nsteps, int every, double eps, double* out, int64_t nsamples,
                          cudaStream_t st) {
    // four lanes an electron while their warps find a scheduler each (152 SMs of four)
    if (slots / ELEC_T * 4 <= 4 * 152)
        electron_launch<4>(cases, order, slots, integrator, flags, dt, nsteps, every, eps, out, nsamples, st);
    else
        electron_launch<1>(cases, order, slots, integrator, flags, dt, nsteps, every, eps, out, nsamples, st);
}

}  // namespace picrr

extern "C" pic_status pic_electron_scan(const pic_electron_case* cases, int64_t n, int integrator, int flags,
                                        double dt, int64_t nsteps, int every, double lambda_um, int device,
                                        double* out, int64_t nsamples) {
    using picrr::set_null_handle_error;
    if (n < 0 || n > (int64_t{1} << 31) || (n > 0 && (!cases || !out)))
        return set_null_handle_error("need 0 <= n <= 2^31 and non-NULL cases and out"), PIC_ERR_INVALID_ARG;
    if (integrator != PIC_INTEGRATOR_LEAPFROG && integrator != PIC_INTEGRATOR_RK4)
        return set_null_handle_error("unknown integrator"), PIC_ERR_INVALID_ARG;
    if ((flags & ~(PIC_ELECTRON_RR | PIC_ELECTRON_DERIV)) != 0 ||
        ((flags & PIC_ELECTRON_DERIV) && integrator != PIC_INTEGRATOR_RK4))
        return set_null_handle_error("bad flags (the derivative term is an RK4 option)"), PIC_ERR_INVALID_ARG;
    if (!(dt > 0.0) || nsteps < 0 || every < 1 || nsamples < 0 || nsamples > nsteps / every ||
        !(lambda_um > 0.0))
        return set_null_handle_error("need dt > 0, every >= 1, 0 <= nsamples <= nsteps/every, lambda_um > 0"),
               PIC_ERR_INVALID_ARG;
    for (int64_t c = 0; c < n; ++c)
        if (cases[c].wave < 0 || cases[c].wave > 2 || (cases[c].wave == 2 && !(cases[c].tau > 0.0)))
            return set_null_handle_error("bad wave (0, 1, or 2 with tau > 0)"), PIC_ERR_INVALID_ARG;
    if (n == 0) return PIC_OK;
    // electrons grouped by the kind of their wave, each group padded to whole warps
    std::vector<int32_t> order;
    try {
        order.reserve(static_cast<size_t>(n) + 3 * picrr::ELEC_T);
    } catch (const std::bad_alloc&) {
        return set_null_handle_error("out of host memory"), PIC_ERR_OOM;
    }
    for (int kind = 0; kind < 3; ++kind) {
        for (int64_t c = 0; c < n; ++c)
            if (cases[c].wave == kind) order.push_back(static_cast<int32_t>(c));
        while (order.size() % picrr::ELEC_T) order.push_back(-1);
    }
    int prev = -1;
    cudaGetDevice(&prev);
    if (cudaSetDevice(device) != cudaSuccess) {
        cudaGetLastError();
        return set_null_handle_error("bad device"), PIC_ERR_INVALID_ARG;
    }
    const double eps = (4.0 / 3.0) * 3.14159265358979323846 * 2.8179403262e-9 / lambda_um;  // r_e in um (CODATA)
    cudaStream_t st = nullptr;
    pic_electron_case* dc = nullptr;
    int32_t* dorder = nullptr;
    double* dout = nullptr;
    const size_t out_bytes = static_cast<size_t>(n) * static_cast<size_t>(nsamples) * 5 * sizeof(double);
    cudaError_t e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaMallocAsync(&dc, sizeof(pic_electron_case) * n, st);
    if (e == cudaSuccess) e = cudaMallocAsync(&dorder, sizeof(int32_t) * order.size(), st);
    if (e == cudaSuccess) e = cudaMallocAsync(&dout, out_bytes ? out_bytes : 16, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dc, cases, sizeof(pic_electron_case) * n, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(dorder, order.data(), sizeof(int32_t) * order.size(), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) {
        picrr::launch_electron_scan(dc, dorder, static_cast<int64_t>(order.size()), integrator, flags, dt, nsteps, every, eps, dout, nsamples, st);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) picrr::touch_pages(out, out_bytes);  // while the kernel runs
    if (e == cudaSuccess && out_bytes) e = cudaMemcpyAsync(out, dout, out_bytes, cudaMemcpyDeviceToHost, st);
    if (dc) cudaFreeAsync(dc, st);
    if (dorder) cudaFreeAsync(dorder, st);
    if (dout) cudaFreeAsync(dout, st);
    const cudaError_t e2 = st ? cudaStreamSynchronize(st) : cudaSuccess;
    if (st) cudaStreamDestroy(st);
    if (prev >= 0) cudaSetDevice(prev);
    if (e == cudaSuccess) e = e2;
    if (e != cudaSuccess) {
        cudaGetLastError();
        set_null_handle_error(std::string("electron scan: ") + cudaGetErrorString(e));
        return PIC_ERR_CUDA;
    }
    return PIC_OK;
}
