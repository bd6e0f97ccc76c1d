// Antenna phasors and pixel weights of the direct sums (k_simt.cu, k_gd.cu), templated on the real
// type.
#pragma once

#include "fm_internal.cuh"

namespace fm {

template <typename R> struct V2;
template <> struct V2<float> { using t = float2; };
template <> struct V2<double> { using t = double2; };

// ---------------------------------------------------------------- phasors
// FP32: phase in turns from two-float products so its fractional part keeps ~2^-24
// absolute accuracy even at 60 turns; every product and sum of the error-free
// transformations is explicitly rounded (no contraction into FMAs).
__device__ __forceinline__ float phase_frac_2f(const float *__restrict__ kap, const float *__restrict__ s)
{
    float accf = 0.f, acce = 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        float kh = kap[2 * c], kl = kap[2 * c + 1], sh = s[2 * c], sl = s[2 * c + 1];
        float p = __fmul_rn(kh, sh);
        float e = __fmaf_rn(kh, sh, -p);                 // exact rounding error of p
        float f = __fsub_rn(p, rintf(p));                // exact: p minus its nearest integer
        accf = __fadd_rn(accf, f);
        acce = __fadd_rn(acce, __fadd_rn(e, __fmaf_rn(kh, sl, __fmul_rn(kl, sh))));
    }
    float t = __fadd_rn(accf, acce);
    return __fsub_rn(t, rintf(t));
}

template <typename R> struct Phasor;
template <> struct Phasor<float> {
    static __device__ __forceinline__ void eval(const DevGeom &g, int f, int i, int t, int p, float &re, float &im)
    {
        float fr = phase_frac_2f(g.kap32 + ((size_t)f * g.A + i) * 6, g.s32 + ((size_t)t * g.npix + p) * 6);
        float sn, cs;
        sincospif(2.0f * fr, &sn, &cs);
        re = cs;
        im = -sn;
    }
};
template <> struct Phasor<double> {
    static __device__ __forceinline__ void eval(const DevGeom &g, int f, int i, int t, int p, double &re, double &im)
    {
        const double *k = g.kap64 + ((size_t)f * g.A + i) * 3;
        const double *s = g.s64 + ((size_t)t * g.npix + p) * 3;
        double ph = k[0] * s[0] + k[1] * s[1] + k[2] * s[2];
        ph -= rint(ph);
        double sn, cs;
        sincospi(2.0 * ph, &sn, &cs);
        re = cs;
        im = -sn;
    }
};

// Beam-weighted solid angle dOmega_d A(za; nu) of pixel p at LST t.
// (Gaussian beam from the squared zenith angle; the Airy beam from its table)
template <typename R>
__device__ __forceinline__ R pixel_weight(const DevGeom &g, int f, int t, int p)
{
    if (g.beam64) return Tab<R>::domega(g)[p / g.R] * (R)g.beam64[((size_t)f * g.T + t) * g.npix + p];
    R z2 = Tab<R>::za2(g)[(size_t)t * g.npix + p];
    if (z2 < R(0)) return R(0);
    return Tab<R>::domega(g)[p / g.R] * exp(Tab<R>::bcoef(g)[f] * z2);
}
template <>
__device__ __forceinline__ float pixel_weight<float>(const DevGeom &g, int f, int t, int p)
{
    if (g.beam32) return g.domega32[p / g.R] * g.beam32[((size_t)f * g.T + t) * g.npix + p];
    float z2 = g.za2_32[(size_t)t * g.npix + p];
    if (z2 < 0.f) return 0.f;
    return g.domega32[p / g.R] * __expf(g.bcoef32[f] * z2);
}

}  // namespace fm
