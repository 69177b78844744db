// bd_update.cuh -- the arithmetic of one pixel update shared by the sweep
// kernel's forms (bd_sweep.cu, bd_rows.cu): proposal, prior terms, twiddles,
// photon-count step.
#pragma once

#include "bd_device.cuh"

namespace bd {

// One entry of the patch prior change: X' = X + delta w, with
//   |X'|^2 - |X|^2 = delta (2 Re(X conj w) + delta)        (|w| = 1)
// accumulates  wa log(|X'|^2/|X|^2),  mult (|X'| - |X|),  mult |X|.
// The ratio form q = (|X'|^2 - |X|^2)/|X|^2 is free of cancellation while
// the coefficient does not shrink much (q > -1/2).  When it shrinks toward
// zero, q rounds to -1 (log1p = -inf, and with wa < 0 an infinite gain that
// the exact Eq. 7-8 change never has), so there the log is taken of the
// ratio |X'|^2/|X|^2 itself, with X' the value an accepted update stores.
// X' exactly 0 is rejected (the Dirichlet density is singular there).
// The same entry with the roundings written out (float), split into the part
// that depends on the coefficient alone (head), shared by the proposals scored
// against one spectrum, and the rest (tail).
struct PriorHead { float mo, i2; };

__device__ __forceinline__ PriorHead prior_head(float xr, float xi)
{
    using P = Prec<float>;
    const float n2 = fmaf(xr, xr, mul_rn(xi, xi));
    return {P::sqrt(n2), P::rcp(n2)};
}

__device__ __forceinline__ void twiddle_mul(float2 eh, float2 ew, float& wr, float& wi)
{
    wr = fmaf(eh.x, ew.x, -mul_rn(eh.y, ew.y));
    wi = fmaf(eh.x, ew.y, mul_rn(eh.y, ew.x));
}

// The fast part of one proposal: adds its mult (|X'| - |X|) to accS and returns
// log(|X'|^2 / |X|^2) as log1p(q); rare is set where prior_rare has to replace it.
__device__ __forceinline__ float prior_tail(float xr, float xi, const PriorHead& h, float wr, float wi, float delta, float mult,
                                            float& accS, bool& rare)
{
    using P = Prec<float>;
    const float dd = mul_rn(delta, fmaf(2.0f, fmaf(xr, wr, mul_rn(xi, wi)), delta));
    const float rn = fmaf(delta, wr, xr), in = fmaf(delta, wi, xi);
    const float n2n = fmaf(rn, rn, mul_rn(in, in));
    const float mn = P::sqrt(n2n);
    const float q = mul_rn(dd, h.i2);
    accS = fmaf(mult, mul_rn(dd, P::rcp(add_rn(mn, h.mo))), accS);
    rare = rare || !(n2n > 0.0f) || !(q > -0.5f);
    return P::log1p(q);
}

__device__ __forceinline__ void prior_rare(float xr, float xi, const PriorHead& h, float wr, float wi, float delta, float& lg,
                                           bool& bad)
{
    const float dd = mul_rn(delta, fmaf(2.0f, fmaf(xr, wr, mul_rn(xi, wi)), delta));
    const float rn = fmaf(delta, wr, xr), in = fmaf(delta, wi, xi);
    const float n2n = fmaf(rn, rn, mul_rn(in, in));
    if (!(n2n > 0.0f)) bad = true;
    if (!(mul_rn(dd, h.i2) > -0.5f)) lg = Prec<float>::log(mul_rn(n2n, h.i2));
}

template <typename T>
__device__ __forceinline__ void prior_term(T xr, T xi, T wr, T wi, T delta, T wa, T mult, T& accP, T& accS,
                                           T& accA, bool& bad)
{
    using P = Prec<T>;
    const T n2 = xr * xr + xi * xi;
    const T dd = delta * ((T)2 * (xr * wr + xi * wi) + delta);
    const T rn = fma(delta, wr, xr), in = fma(delta, wi, xi);
    const T n2n = rn * rn + in * in;
    if (!(n2n > (T)0)) bad = true;
    const T mo = P::sqrt(n2), mn = P::sqrt(n2n);
    const T i2 = P::rcp(n2);
    const T q = dd * i2;
    accP += wa * (q > (T)-0.5 ? P::log1p(q) : P::log(n2n * i2));
    accS += mult * (dd * P::rcp(mn + mo));
    accA += mult * mo;
}

// The target (Eq. 9) has a finite density at every state a chain can reach,
// so a proposal whose log acceptance ratio is not finite (and that is not
// impossible: mu' <= 0, a zero coefficient) is an arithmetic failure.  It is
// rejected, the numeric error bit raised, and the first such update recorded
// for the host: err[2] chain, err[3] pixel, err[8] sweep, dL and dP as
// doubles at err + 4.
static __device__ __noinline__ void report_nonfinite(int* err, int chain, int m, int t, double dL, double dP)
{
    atomicOr(err, kErrRatio);
    if (atomicCAS(err + 1, 0, 1) == 0) {
        err[2] = chain;
        err[3] = m;
        err[8] = t;
        double* d = reinterpret_cast<double*>(err + 4);
        d[0] = dL;
        d[1] = dP;
    }
}

// x mod n for 0 <= x < 2^22 through a float reciprocal (exact after one correction)
__device__ __forceinline__ int small_mod(int x, int n, float inv_n)
{
    int r = x - n * __float2int_rz((float)x * inv_n);
    r += r < 0 ? n : 0;
    r -= r >= n ? n : 0;
    return r;
}

template <typename T>
__device__ __forceinline__ void twiddle(const T* tw, const Shape& sh, int kl, int u, int v, T& wr, T& wi)
{
    const int k = kl >> 16, l = kl & 0xffff;
    const T* eh = tw + 2 * (sh.twh_off + small_mod(k * u, sh.ph, sh.inv_ph));
    const T* ew = tw + 2 * (sh.tww_off + small_mod(l * v, sh.pw, sh.inv_pw));
    wr = eh[0] * ew[0] - eh[1] * ew[1];
    wi = eh[0] * ew[1] + eh[1] * ew[0];
}

// a2: the proposal of one update from its Philox counter (m, t, chain, 0):
// z standard normal (Box-Muller), log u, the log-space move hz = s_m z (s_m
// the pixel's scale: its adapted one, else the problem's step) and
// rho' = rho exp(hz); hz is also the Hastings term of the decision.
template <typename T>
__device__ __forceinline__ void proposal(const Image& im, const Chain& ch, int m, int t, T r_old, T& hz, T& lu,
                                         T& r_new, T& delta)
{
    using P = Prec<T>;
    const uint4 x = philox4x32_10(make_uint4((uint32_t)m, (uint32_t)t, (uint32_t)ch.chain, 0u), im.seed_lo,
                                  im.seed_hi);
    const T z = P::gauss(uniform23<T>(x.x), uniform23<T>(x.y));
    const T sm = ch.steps != nullptr ? reinterpret_cast<const T*>(ch.steps)[m] : (T)im.step;
    hz = sm * z;
    lu = P::log(uniform23<T>(x.z));
    r_new = r_old * P::exp(hz);
    delta = r_new - r_old;
}

// Photon-count step of the augmented sampler for one patch (camera grid), one
// thread's share: draws phi_n ~ p(phi | w_n, mu_n) (Philox counter (n, t,
// chain, 1)) for the camera pixels centred on the patch; returns the warp's
// change of the log joint density.
template <typename T>
__device__ __forceinline__ double phi_step_partial(const Image& im, const Chain& ch, int pi, int pj, int t, int lt, int NT,
                                                   const Dat4<T>* dat_g, int* err)
{
    const Shape& shp = im.shape[shape_index(im, pi, pj)];
    const T* mu_g = reinterpret_cast<const T*>(ch.mu);
    T* phi_g = reinterpret_cast<T*>(ch.phi);
    double dj = 0.0;
    int bad = 0;
    for (int e = lt; e < shp.ph * shp.pw; e += NT) {
        const int uu = e / shp.pw, vv = e - (e / shp.pw) * shp.pw;
        const int aa = pi * im.S + uu - im.R, bb = pj * im.S + vv - im.R;
        if (aa < 0 || bb < 0 || aa >= im.H || bb >= im.W) continue;
        const size_t idx = (size_t)aa * im.mu_pitch + bb;
        const T mu = __ldcg(mu_g + idx);
        const Dat4<T> dv = dat_g[(size_t)aa * im.W + bb];
        const uint4 x = philox4x32_10(make_uint4((uint32_t)(aa * im.W + bb), (uint32_t)t, (uint32_t)ch.chain, 1u),
                                      im.seed_lo, im.seed_hi);
        const int pn = sample_phi<T>(mu, dv.c, dv.is2, uniform23<T>(x.x), bad);
        const int po = (int)phi_g[idx];
        if (pn != po) {   // an unchanged count changes nothing
            const double lmu = ::log((double)mu);
            dj += phi_logterm_tab(pn, lmu, (double)dv.c, (double)dv.is2, im.lgam) -
                  phi_logterm_tab(po, lmu, (double)dv.c, (double)dv.is2, im.lgam);
            phi_g[idx] = (T)pn;
        }
    }
    if (bad) atomicOr(err, kErrNumeric);
    return warp_sum(dj);
}

}  // namespace bd
