// Drift scans in hour-angle Fourier modes: the contraction of k_ha.cu with every fringe group's response
// kept as its band of modes.
//
// Under one primary beam, V_u(t) = sum_d sum_j P_u(tau_t + j, d) y(j, d), j = (R - 1 - r) q: a correlation along
// hour angle in cells of 1 / q RA pixel, tau_t = (LST_t - LST_min) in cells.  P_u is a beam of a few degrees
// times a fringe, so its Fourier series over a window of L cells is a band of some 35 modes around the fringe
// rate, where the cells in use number nh = 251 (37 antennas) or 503 (127 antennas).  With
//   P_u(n, d) = sum_m c_u(m, d) e^{2 pi i m n / L},   Y(m, d) = sum_j y(j, d) e^{2 pi i m j / L},
//   V_u(t) = sum_{m in band(u)} e^{2 pi i m tau_t / L} sum_d c_u(m, d) Y(m, d),
// and the transpose gives the pixel gradient.  tau_t need not be a whole number where the cells sample the fringes
// above their Nyquist rate: LSTs off the pixel grid take the same path.  Y comes from the mode transform of
// k_modes.cu with the RA basis functions replaced by their Fourier sums, so the pixels are never formed.  Cells
// outside 0 .. nh - 1 meet no pixel: there P_u is continued by its own formula, to where the beam is below MM_EDGE
// of its maximum, so that the window has no step and the band ends; what a band leaves out is below MM_EPS of the
// response's l2 norm, far under the FP32 rounding (6e-8) of the table that keeps it.  All of these are relative to
// the largest response in the window, and a grid whose hour angles stay off the meridian has it in cells that meet
// no pixel: what is left in those in use is then wrong by 3e-8 times the ratio of the two (a beam of 4.2 degrees
// FWHM, the nearest cell in use 5 degrees off the meridian: 2e-6; 10 degrees off: 1e-2).  The form is taken up to a
// ratio of MM_PEAK = 4, where that is 1e-7, below the FP32 sums' own 2.8e-7.
//
// The sky is real, so modes m and -m share Y: an element e = (|m|, u, sign) keeps c_u(m) or conj(c_u(-m)).
// The table [e][declination] is sorted by |m|: the forward is one dot product over declinations per element, the
// adjoint one sum over the elements of |m| per declination, both bound by one pass over the table in HBM.
//
// The tensor-core forms make the response of every cell anew from antenna phasors (bound by the producers and the
// MMA issue of N = 64: k_ha.cu, k_tc.cu).  Measured with FP16 x3, their time first, the figures of chi^2 and
// gradient: 37 antennas, 64 channels, 60 LSTs: forward 189 -> 36 us (k_mm_fwd 28 of them, 142 MB of table at 5.1
// TB/s), adjoint 188 -> 40 us (k_mm_adj 26); LSTs off the grid (12 of them): 10.02 ms -> 82 us; 127 antennas, 128
// channels, 120 LSTs: 7.26 -> 0.61 ms (k_mm_fwd 477 us, 3.1 GB at 6.5 TB/s) and 4.98 -> 0.65 ms.  The errors against
// 64 bits fall to those of the mode transforms (V of 7 antennas 1.3e-6 -> 2.6e-7).
// FP32 handles: 37 antennas, 64 channels, 60 LSTs, chi^2 and gradient 3.13 ms (each distinct fringe on the CUDA
// cores, k_hs.cu) -> 0.27 ms; gradient against 64 bits 1.0e-7 in the mean of 14 geometries (1.2e-7 before), V 1.7e-7
// (2.8e-7).
#include <algorithm>
#include <cmath>
#include <vector>

#include "fm_internal.cuh"

namespace fm {
namespace {

constexpr double MM_EDGE = 4e-9;       // beam at the window's ends, relative to its maximum
constexpr double MM_EPS = 1e-9;        // l2 share of a response outside its band
constexpr double MM_PEAK = 4.0;        // beam in the cells around those in use, relative to its maximum in them
constexpr int MM_MAXL = 2048;
constexpr int MM_MAXQ = 8;             // cells per RA pixel, LSTs off the pixel grid
constexpr int MM_ROWS = 8;             // forward: elements a warp sums at a time
constexpr int MM_TC = 16;              // LSTs of a CTA of k_mm_vis

// window transform: L = product of radices 2 .. 5
struct MmFft {
    int L, ns, rad[12];
};

bool smooth_factors(int L, MmFft &p)
{
    p.L = L;
    p.ns = 0;
    for (int r : {4, 5, 3, 2})
        while (L % r == 0 && p.ns < 12) {
            p.rad[p.ns++] = r;
            L /= r;
        }
    return L == 1;
}

// Stockham passes over shared memory: out[o] = sum_i in[j + i L / r] tw[(i rem L / (Ns r)) mod L]; tw =
// e^{-2 pi i x / L}.  The result is in `a` or `b`, whichever is returned.
template <typename C2>
__device__ __forceinline__ C2 *mm_fft(const MmFft &p, C2 *a, C2 *b, const C2 *tw)
{
    int Ns = 1;
    for (int s = 0; s < p.ns; ++s) {
        const int r = p.rad[s], span = Ns * r, Lr = p.L / r, step = p.L / span;
        __syncthreads();
        for (int o = threadIdx.x; o < p.L; o += blockDim.x) {
            const int blk = o / span, rem = o - blk * span;
            const int j = blk * Ns + rem % Ns;
            C2 v = a[j];
            int e = 0;
            for (int i = 1; i < r; ++i) {
                e += rem * step;
                if (e >= p.L) e -= p.L;
                const C2 x = a[j + i * Lr], w = tw[e];
                v.x += x.x * w.x - x.y * w.y;
                v.y += x.x * w.y + x.y * w.x;
            }
            b[o] = v;
        }
        C2 *t = a;
        a = b;
        b = t;
        Ns = span;
    }
    __syncthreads();
    return a;
}

struct MmGeo {
    double lst0, ra_min, dra, dec_min, ddec, lat;
    int R, D, q, L, p0;
};

struct MmDir { double x, y, z, w; };

// direction (east, north, up) and squared zenith angle of cell n' - p0 at declination d; < 0 below the horizon
__global__ void k_mm_geo(MmGeo a, MmDir *__restrict__ geo)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= a.D * a.L) return;
    const int d = e / a.L, n = e % a.L - a.p0;
    const double H = a.lst0 - (a.ra_min + ((double)((a.R - 1) * a.q - n) + 0.5 * a.q) * (a.dra / a.q));
    const double dec = a.dec_min + (d + 0.5) * a.ddec;
    double sd, cd, sh, ch, sl, cl;
    sincos(dec, &sd, &cd);
    sincos(H, &sh, &ch);
    sincos(a.lat, &sl, &cl);
    const double sE = -cd * sh, sN = cl * sd - sl * cd * ch, sU = sl * sd + cl * cd * ch;
    double za2 = -1.0;
    if (sU > 0.0) {
        const double za = acos(sU > 1.0 ? 1.0 : sU);
        za2 = za * za;
    }
    geo[e] = MmDir{sE, sN, sU, za2};
}

// dOmega A of every (channel, declination, cell), formed in FP64
__global__ void k_mm_weight(int F, int D, int L, const MmDir *__restrict__ geo, const double *__restrict__ bcoef,
                            const double *__restrict__ domega, float *__restrict__ w)
{
    const long long n = (long long)F * D * L;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const int dl = (int)(e % ((long long)D * L)), f = (int)(e / ((long long)D * L));
        const double za2 = geo[dl].w;
        w[e] = za2 < 0.0 ? 0.f : (float)(domega[dl / L] * exp(bcoef[f] * za2));
    }
}

// Band of every (channel, group): the shortest run of modes around the strongest one that leaves out at most
// MM_EPS of the l2 norm, over every dstep-th declination and the last, and one mode more at each end.
__global__ void __launch_bounds__(256) k_mm_band(MmFft p, int D, int U, int A, int dstep, const MmDir *__restrict__ geo,
                                                 const double2 *__restrict__ tw, const double *__restrict__ bcoef,
                                                 const double *__restrict__ domega, const double *__restrict__ kap,
                                                 const int2 *__restrict__ uij, const int *__restrict__ ant,
                                                 int2 *__restrict__ band)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double2 *sa = reinterpret_cast<double2 *>(smem_raw), *sb = sa + p.L, *st = sb + p.L;
    double *en = reinterpret_cast<double *>(st + p.L);
    const int f = blockIdx.x / U, u = blockIdx.x % U, L = p.L;
    const int2 ij = uij[u];
    const double *ki = kap + ((size_t)f * A + ant[ij.x]) * 3, *kj = kap + ((size_t)f * A + ant[ij.y]) * 3;
    const double k0 = ki[0] - kj[0], k1 = ki[1] - kj[1], k2 = ki[2] - kj[2];
    for (int n = threadIdx.x; n < L; n += blockDim.x) {
        st[n] = tw[n];
        en[n] = 0.0;
    }
    for (int d = 0;; d = min(d + dstep, D - 1)) {
        __syncthreads();
        for (int n = threadIdx.x; n < L; n += blockDim.x) {
            const MmDir g = geo[(size_t)d * L + n];
            double2 v = make_double2(0.0, 0.0);
            if (g.w >= 0.0) {
                const double w = domega[d] * exp(bcoef[f] * g.w);
                double ph = k0 * g.x + k1 * g.y + k2 * g.z;
                ph -= rint(ph);
                double sn, cs;
                sincospi(2.0 * ph, &sn, &cs);
                v = make_double2(w * cs, -w * sn);
            }
            sa[n] = v;
        }
        const double2 *r = mm_fft(p, sa, sb, st);
        for (int n = threadIdx.x; n < L; n += blockDim.x) en[n] += r[n].x * r[n].x + r[n].y * r[n].y;
        if (d == D - 1) break;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        int at = 0;
        for (int n = 0; n < L; ++n) {
            tot += en[n];
            if (en[n] > en[at]) at = n;
        }
        const double most = 0.5 * MM_EPS * MM_EPS * tot;
        int lo = at - L / 2, hi = lo + L - 1;         // inclusive, around the strongest mode
        auto val = [&](int m) { return en[((m % L) + L) % L]; };
        double cum = 0.0;
        while (lo < at && cum + val(lo) <= most) cum += val(lo++);
        cum = 0.0;
        while (hi > at && cum + val(hi) <= most) cum += val(hi--);
        if (hi - lo + 1 <= L - 2) {
            --lo;
            ++hi;
        }
        band[blockIdx.x] = make_int2(lo, hi - lo + 1);
    }
}

// The table: CTA = (channel, group), two declinations a turn.  code[(seg wmax + i) 64 + (u & 63)] = 2 e +
// conjugated for mode lo + i of group u, -1 outside its band.
__global__ void __launch_bounds__(256) k_mm_fill(MmFft p, int F, int D, int U, int A, int p0, int wmax, float scale,
                                                 const MmDir *__restrict__ geo, const float *__restrict__ wt,
                                                 const double2 *__restrict__ tw, const double *__restrict__ kap,
                                                 const int2 *__restrict__ uij, const int *__restrict__ ant,
                                                 const int2 *__restrict__ band, const int *__restrict__ code,
                                                 float4 *__restrict__ tab)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int L = p.L, f = blockIdx.x / U, u = blockIdx.x % U, np = (D + 1) / 2;
    float2 *s0 = reinterpret_cast<float2 *>(smem_raw), *s1 = s0 + L, *s2 = s1 + L, *s3 = s2 + L, *st = s3 + L;
    const int2 ij = uij[u], bd = band[blockIdx.x];
    const double *ki = kap + ((size_t)f * A + ant[ij.x]) * 3, *kj = kap + ((size_t)f * A + ant[ij.y]) * 3;
    const double k0 = ki[0] - kj[0], k1 = ki[1] - kj[1], k2 = ki[2] - kj[2];
    for (int n = threadIdx.x; n < L; n += blockDim.x) st[n] = make_float2((float)tw[n].x, (float)tw[n].y);
    const int *cd = code + (size_t)((u >> 6) * F + f) * wmax * 64 + (u & 63);
    for (int pr = 0; pr < np; ++pr) {
        __syncthreads();
        for (int e = threadIdx.x; e < 2 * L; e += blockDim.x) {
            const int h = e >= L, n = e - h * L, d = 2 * pr + h;
            float2 v = make_float2(0.f, 0.f);
            if (d < D) {
                const MmDir g = geo[(size_t)d * L + n];
                const float w = wt[((size_t)f * D + d) * L + n];
                double ph = k0 * g.x + k1 * g.y + k2 * g.z;
                ph -= rint(ph);
                float sn, cs;
                sincospif(2.f * (float)ph, &sn, &cs);
                v = make_float2(w * cs, -w * sn);
            }
            (h ? s2 : s0)[n] = v;
        }
        const float2 *r0 = mm_fft(p, s0, s1, st), *r1 = mm_fft(p, s2, s3, st);
        for (int i = threadIdx.x; i < bd.y; i += blockDim.x) {
            const int c = cd[(size_t)i * 64], m = (((bd.x + i) % L) + L) % L;
            float2 w = st[(int)((long long)m * p0 % L)];          // c(m) = P(m) e^{2 pi i m p0 / L} / L
            w = make_float2(w.x * scale, -w.y * scale);
            const float2 a = r0[m], b = r1[m];
            float2 x = make_float2(a.x * w.x - a.y * w.y, a.x * w.y + a.y * w.x);
            float2 y = make_float2(b.x * w.x - b.y * w.y, b.x * w.y + b.y * w.x);
            if (c & 1) {
                x.y = -x.y;
                y.y = -y.y;
            }
            tab[(size_t)(c >> 1) * np + pr] = make_float4(x.x, y.x, x.y, y.y);
        }
    }
}

// RA basis of the modes: rows 2 m and 2 m + 1 = Re and Im of sum_r Phi[r][a] e^{2 pi i m j_r / L} (pix: of the
// pixel r itself), times scale
__global__ void k_mm_basis(int R, int M, int q, int L, int rows, double scale, const double2 *__restrict__ tw,
                           const double *__restrict__ phi, double *__restrict__ b64, float *__restrict__ b32,
                           float *__restrict__ pix)
{
    const long long n = (long long)rows / 2 * M;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const int m = (int)(e / M), a = (int)(e % M);
        double re = 0.0, im = 0.0;
        for (int r = 0; r < R; ++r) {
            const double2 w = tw[(int)((long long)m * (R - 1 - r) * q % L)];
            const double v = phi[(size_t)r * M + a];
            re += v * w.x;
            im -= v * w.y;
        }
        b64[(size_t)(2 * m) * M + a] = scale * re;
        b64[(size_t)(2 * m + 1) * M + a] = scale * im;
        b32[(size_t)(2 * m) * M + a] = (float)(scale * re);
        b32[(size_t)(2 * m + 1) * M + a] = (float)(scale * im);
    }
    const long long np = (long long)rows / 2 * R;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < np; e += (long long)gridDim.x * blockDim.x) {
        const int m = (int)(e / R), r = (int)(e % R);
        const double2 w = tw[(int)((long long)m * (R - 1 - r) * q % L)];
        pix[(size_t)(2 * m) * R + r] = (float)(scale * w.x);
        pix[(size_t)(2 * m + 1) * R + r] = (float)(-scale * w.y);
    }
}

// ------------------------------------------------------------ forward
// One warp per item (channel f, mode |m|, up to MM_ROWS of its elements): lanes over pairs of declinations,
// eight 16-byte loads of the table in flight each, packed FMAs on the pairs; the 2 MM_ROWS sums are then
// halved lane by lane (16 shuffles for 16 sums instead of 80).  NS skies share the table's loads.
template <int NS>
__global__ void __launch_bounds__(256, 2) k_mm_fwd(int nitem, const int4 *__restrict__ items, int D, int ld, long long ys,
                                                const float4 *__restrict__ tab, const float *__restrict__ Y,
                                                long long zs, float *__restrict__ z)
{
    const int it = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (it >= nitem) return;
    const int4 w = items[it];                       // f, m, first element, elements
    const int np = (D + 1) / 2;
    const float *Yf = Y + (size_t)w.x * D * ld + 2 * w.y;
    const float4 *tp = tab + (size_t)w.z * np;
    float2 re[NS][MM_ROWS], im[NS][MM_ROWS];
#pragma unroll
    for (int s = 0; s < NS; ++s)
#pragma unroll
        for (int r = 0; r < MM_ROWS; ++r) re[s][r] = im[s][r] = make_float2(0.f, 0.f);
#pragma unroll 2
    for (int i = lane; i < np; i += 32) {
        float4 c[MM_ROWS];
#pragma unroll
        for (int r = 0; r < MM_ROWS; ++r)
            c[r] = r < w.w ? __ldg(tp + (size_t)r * np + i) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const float *y = Yf + s * ys + (size_t)(2 * i) * ld;
            const float2 a = *reinterpret_cast<const float2 *>(y);
            const float2 b = 2 * i + 1 < D ? *reinterpret_cast<const float2 *>(y + ld) : make_float2(0.f, 0.f);
            const float2 yr = make_float2(a.x, b.x), yi = make_float2(a.y, b.y), ni = make_float2(-a.y, -b.y);
#pragma unroll
            for (int r = 0; r < MM_ROWS; ++r) {
                const float2 cr = make_float2(c[r].x, c[r].y), ci = make_float2(c[r].z, c[r].w);
                re[s][r] = __ffma2_rn(ci, ni, __ffma2_rn(cr, yr, re[s][r]));
                im[s][r] = __ffma2_rn(ci, yr, __ffma2_rn(cr, yi, im[s][r]));
            }
        }
    }
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        float v[2 * MM_ROWS];
#pragma unroll
        for (int r = 0; r < MM_ROWS; ++r) {
            v[2 * r] = re[s][r].x + re[s][r].y;
            v[2 * r + 1] = im[s][r].x + im[s][r].y;
        }
#pragma unroll
        for (int h = MM_ROWS; h >= 1; h >>= 1) {     // lane bit 2 h takes the upper half
            const bool up = lane & (2 * h);
#pragma unroll
            for (int q = 0; q < h; ++q) {
                const float keep = up ? v[q + h] : v[q], give = up ? v[q] : v[q + h];
                v[q] = keep + __shfl_xor_sync(0xffffffffu, give, 2 * h);
            }
        }
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
        if (!(lane & 1) && (lane >> 2) < w.w) z[s * zs + 2 * (size_t)w.z + (lane >> 1)] = v[0];
    }
}

// V_u(t) of MM_TC LSTs of 64 groups: CTA = (segment, LST chunk, sky).  The groups' modes and the LSTs' phasors
// ph[t][m - mlo] = e^{2 pi i m tau_t / L} are staged in shared memory; four modes share one phasor, the three
// after it follow by Horner's rule in s = e^{2 pi i tau_t / L} (the last column).  Rows 2 u and 2 u + 1 of an LST go
// out as the forward's one partial sum (HaVSrc).
__global__ void __launch_bounds__(256) k_mm_vis(int F, int T, int U, int mlo, int pw, int wmax,
                                                const int *__restrict__ code, const int2 *__restrict__ band,
                                                const float2 *__restrict__ ph, const float2 *__restrict__ z, long long zs,
                                                int slot_rows, int N, float *__restrict__ vpart)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *sz = reinterpret_cast<float2 *>(smem_raw);           // [w4][64]
    const int w4 = (wmax + 3) & ~3;
    float2 *sp = sz + w4 * 64;                                   // [MM_TC][pw]
    const int seg = blockIdx.x, f = seg % F, mt = seg / F, tid = threadIdx.x;
    const int tb = blockIdx.y * MM_TC, nt = min(MM_TC, T - tb);
    const float2 *zz = z + blockIdx.z * zs;
    for (int e0 = tid; e0 < w4 * 64; e0 += 4 * 256) {            // four gathers in flight
        int c[4];
        float2 v[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) c[r] = e0 + 256 * r < wmax * 64 ? code[(size_t)seg * wmax * 64 + e0 + 256 * r] : -1;
#pragma unroll
        for (int r = 0; r < 4; ++r) v[r] = c[r] >= 0 ? zz[c[r] >> 1] : make_float2(0.f, 0.f);
#pragma unroll
        for (int r = 0; r < 4; ++r)
            if (e0 + 256 * r < w4 * 64) sz[e0 + 256 * r] = make_float2(v[r].x, (c[r] & 1) ? -v[r].y : v[r].y);
    }
#pragma unroll 4
    for (int e = tid; e < MM_TC * pw; e += 256) sp[e] = e < nt * pw ? ph[(size_t)tb * pw + e] : make_float2(0.f, 0.f);
    __syncthreads();
    const int ul = tid & 63, u = mt * 64 + ul, tl = tid >> 6;
    const int2 bd = u < U ? band[(size_t)f * U + u] : make_int2(mlo, 0);
    const float2 *pt = sp + tl * pw + (bd.x - mlo);
    float2 s[4], acc[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        s[j] = sp[(tl + 4 * j) * pw + pw - 1];
        acc[j] = make_float2(0.f, 0.f);
    }
    for (int i = 0; i < bd.y; i += 4) {                          // modes past the band are zero
        const float2 z0 = sz[i * 64 + ul], z1 = sz[(i + 1) * 64 + ul], z2 = sz[(i + 2) * 64 + ul],
                     z3 = sz[(i + 3) * 64 + ul];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float2 ss = s[j], w = pt[4 * j * pw + i];
            float2 h = make_float2(z2.x + z3.x * ss.x - z3.y * ss.y, z2.y + z3.x * ss.y + z3.y * ss.x);
            h = make_float2(z1.x + h.x * ss.x - h.y * ss.y, z1.y + h.x * ss.y + h.y * ss.x);
            h = make_float2(z0.x + h.x * ss.x - h.y * ss.y, z0.y + h.x * ss.y + h.y * ss.x);
            acc[j].x += h.x * w.x - h.y * w.y;
            acc[j].y += h.x * w.y + h.y * w.x;
        }
    }
    float2 *out = reinterpret_cast<float2 *>(vpart + ((size_t)seg * N + (size_t)blockIdx.z * slot_rows + tb) * 128) + ul;
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if (tl + 4 * j < nt) out[(size_t)(tl + 4 * j) * 64] = acc[j];
}

// ------------------------------------------------------------ adjoint
// w_e of every element from the group sums Q_u(t): sum_t conj(Q_u(t)) e^{2 pi i m tau_t / L}, conjugated for
// the conjugated elements.  CTA = (channel, 8 groups), one warp a group, lanes over the modes of its band, so
// that the phasors are read in a row; Q is staged MM_QT LSTs at a time and the phasors of ten LSTs are in
// flight.  (Lanes over groups, four modes each, gathered 32 phasors a load: 27 us at 37 antennas, 64 channels,
// 60 LSTs; Q read word by word from L2: 20 us.)
constexpr int MM_QT = 60;
__global__ void __launch_bounds__(256) k_mm_q(int T, int U, int mlo, int pw, int wmax, const int *__restrict__ code,
                                              const int2 *__restrict__ band, const float2 *__restrict__ ph,
                                              const float2 *__restrict__ q32, float2 *__restrict__ w)
{
    __shared__ float2 sq[MM_QT][8];
    const int f = blockIdx.y, F = gridDim.y, u0 = blockIdx.x * 8, uw = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int u = u0 + uw;
    const int2 bd = u < U ? band[(size_t)f * U + u] : make_int2(mlo, 0);
    const int *cd = code + (size_t)((u >> 6) * F + f) * wmax * 64 + (u & 63);
    for (int ib = 0; ib < wmax; ib += 64) {
        const int i = ib + lane;
        const bool one = i < bd.y, two = i + 32 < bd.y;
        const float2 *pm = ph + (bd.x + i - mlo);
        float2 a = make_float2(0.f, 0.f), b = a;
        for (int tb = 0; tb < T; tb += MM_QT) {
            const int nt = min(MM_QT, T - tb);
            __syncthreads();
            for (int e = threadIdx.x; e < MM_QT * 8; e += 256) {
                const int t = e >> 3, v = u0 + (e & 7);
                sq[t][e & 7] = t < nt && v < U ? q32[((size_t)f * T + tb + t) * U + v] : make_float2(0.f, 0.f);
            }
            __syncthreads();
            if (!one) continue;
            for (int t = 0; t < nt; t += 10) {
                float2 x[10], y[10];
#pragma unroll
                for (int r = 0; r < 10; ++r) {
                    const float2 *p = pm + (size_t)(tb + min(t + r, nt - 1)) * pw;
                    x[r] = __ldg(p);
                    y[r] = two ? __ldg(p + 32) : make_float2(0.f, 0.f);
                }
#pragma unroll
                for (int r = 0; r < 10; ++r) {
                    const float2 v = sq[t + r][uw];           // zero past the last LST
                    a.x += v.x * x[r].x + v.y * x[r].y;       // conj(Q) e^{...}
                    a.y += v.x * x[r].y - v.y * x[r].x;
                    b.x += v.x * y[r].x + v.y * y[r].y;
                    b.y += v.x * y[r].y - v.y * y[r].x;
                }
            }
        }
        if (one) {
            const int c = cd[(size_t)i * 64];
            w[c >> 1] = make_float2(a.x, (c & 1) ? -a.y : a.y);
        }
        if (two) {
            const int c = cd[(size_t)(i + 32) * 64];
            w[c >> 1] = make_float2(b.x, (c & 1) ? -b.y : b.y);
        }
    }
}
static_assert(MM_QT % 10 == 0, "k_mm_q reads LSTs in tens");

// G[f][d][2 m] = Re, [2 m + 1] = -Im of X(m, d) = sum over the elements of |m| of c_e(d) w_e: two warps per
// (channel, m, 32 pairs of declinations), one for each half of the elements (their numbers differ tenfold between
// modes, and with one warp each the longest ran alone at the end: 27.7 -> 26.0 us for 37 antennas), eight 16-byte
// loads of the table in flight a lane.  The channels run against the forward's order, so that what the forward read
// last is still in L2.
__global__ void __launch_bounds__(256) k_mm_adj(int F, int D, int nm, int ld, const int *__restrict__ moff,
                                                const float4 *__restrict__ tab, const float2 *__restrict__ w,
                                                float *__restrict__ G)
{
    __shared__ float4 half[4][32];
    const int np = (D + 1) / 2, nchunk = (np + 31) / 32, nmc = ld / 2;
    const int wl = threadIdx.x >> 5, second = wl >> 2, lane = threadIdx.x & 31;
    const int wi = blockIdx.x * 4 + (wl & 3);
    const int m = wi % nmc, fc = wi / nmc, ch = fc % nchunk, f = F - 1 - fc / nchunk;
    const int i = ch * 32 + lane;
    const bool on = f >= 0 && i < np;
    float2 re = make_float2(0.f, 0.f), im = re;
    auto add = [&](const float4 &c, const float2 &x) {
        const float2 cr = make_float2(c.x, c.y), ci = make_float2(c.z, c.w);
        const float2 wx = make_float2(x.x, x.x), wy = make_float2(x.y, x.y), ny = make_float2(-x.y, -x.y);
        re = __ffma2_rn(ci, ny, __ffma2_rn(cr, wx, re));
        im = __ffma2_rn(ci, wx, __ffma2_rn(cr, wy, im));
    };
    if (on && m < nm) {
        const int e0 = moff[f * (nm + 1) + m], e2 = moff[f * (nm + 1) + m + 1], mid = e0 + (e2 - e0 + 1) / 2;
        const int e1 = second ? e2 : mid;
        int e = second ? mid : e0;
        const float4 *tp = tab + (size_t)e * np + i;
        const float2 *wp = w + e;
        for (; e + 8 <= e1; e += 8, tp += (size_t)8 * np, wp += 8) {
            float4 c[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) c[r] = __ldg(tp + (size_t)r * np);
#pragma unroll
            for (int r = 0; r < 8; ++r) add(c[r], __ldg(wp + r));
        }
        if (e < e1) {
            float4 c[7];
#pragma unroll
            for (int r = 0; r < 7; ++r) c[r] = e + r < e1 ? __ldg(tp + (size_t)r * np) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int r = 0; r < 7; ++r) add(c[r], e + r < e1 ? __ldg(wp + r) : make_float2(0.f, 0.f));
        }
    }
    if (second) half[wl & 3][lane] = make_float4(re.x, re.y, im.x, im.y);
    __syncthreads();
    if (second || !on) return;
    const float4 o = half[wl & 3][lane];
    float *g = G + ((size_t)f * D + 2 * i) * ld + 2 * m;
    *reinterpret_cast<float2 *>(g) = make_float2(re.x + o.x, -(im.x + o.z));
    if (2 * i + 1 < D) *reinterpret_cast<float2 *>(g + ld) = make_float2(re.y + o.y, -(im.y + o.w));
}

// Response maps of the mass matrix in hour-angle modes.  Its blocks sum conj(R) R over the LSTs, where a
// group's responses at the LSTs are R = E Y (E the phasors of its band, Y its modes, at every declination), and
// E^H E = f f^H with nf columns, fewer than there are LSTs (17 for 60 within 15 degrees): the maps conj(f_j) Y serve as
// nf LSTs.  X[j][plane][u][d][c] = sqrt(W_u) / sigma times the real (plane 0) and imaginary part of map j0 + j, in the
// columns of launch_mm_to_modes.  Mass matrix of 37 antennas, 64 channels, 60 LSTs: 83.1 -> 34.9 ms (maps of every
// LST: transforms 39.8, Gram 27.1 ms; these: 10.3 and 8.6, and 2.3 for the maps, bound by their 8 GB).
constexpr int MM_JMAX = 16, MM_MAPP = 4;
__global__ void __launch_bounds__(256) k_mm_maps(int f, int F, int D, int U, int L, int wmax, int ld, int nj,
                                                 const float2 *__restrict__ fac, const int *__restrict__ code,
                                                 const int2 *__restrict__ band, const float4 *__restrict__ tab,
                                                 const float *__restrict__ W, float inv_sigma2, float *__restrict__ X)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *sf = reinterpret_cast<float2 *>(smem_raw);           // [nj][wmax]
    const int u = blockIdx.y, np = (D + 1) / 2, nmc = ld / 2, p0 = blockIdx.x * MM_MAPP;
    for (int e = threadIdx.x; e < nj * wmax; e += 256) sf[e] = fac[e];
    __syncthreads();
    const int2 bd = band[(size_t)f * U + u];
    const int *cd = code + (size_t)((u >> 6) * F + f) * wmax * 64 + (u & 63);
    const float wu = sqrt(W[(size_t)f * U + u] * inv_sigma2);
    for (int e = threadIdx.x; e < MM_MAPP * nmc; e += 256) {
        const int m = e % nmc, pr = p0 + e / nmc;
        if (pr >= np) break;
        // places of +m and -m in the band
        int ip = ((m - bd.x) % L + L) % L, in = ((-m - bd.x) % L + L) % L;
        if (2 * m > L || ip >= bd.y) ip = -1;
        if (2 * m >= L || m == 0 || in >= bd.y) in = -1;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
        if (ip >= 0) a = tab[(size_t)(cd[(size_t)ip * 64] >> 1) * np + pr];
        if (in >= 0) b = tab[(size_t)(cd[(size_t)in * 64] >> 1) * np + pr];
        a = make_float4(a.x * wu, a.y * wu, a.z * wu, a.w * wu);
        b = make_float4(b.x * wu, b.y * wu, b.z * wu, b.w * wu);
        for (int j = 0; j < nj; ++j) {
            const float2 fp = ip >= 0 ? sf[j * wmax + ip] : make_float2(0.f, 0.f);
            float2 fn = in >= 0 ? sf[j * wmax + in] : make_float2(0.f, 0.f);
            fn.y = -fn.y;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int d = 2 * pr + h;
                if (d >= D) break;
                const float2 x = h ? make_float2(a.y, a.w) : make_float2(a.x, a.z);
                const float2 y = h ? make_float2(b.y, b.w) : make_float2(b.x, b.z);
                const float2 s = make_float2(fp.x * x.x - fp.y * x.y, fp.x * x.y + fp.y * x.x);
                const float2 t = make_float2(fn.x * y.x - fn.y * y.y, fn.x * y.y + fn.y * y.x);
                float *o = X + ((((size_t)2 * j) * U + u) * D + d) * ld + 2 * m;
                *reinterpret_cast<float2 *>(o) = make_float2(s.x + t.x, -s.y - t.y);
                *reinterpret_cast<float2 *>(o + (size_t)U * D * ld) = make_float2(s.y - t.y, s.x - t.x);
            }
        }
    }
}

__global__ void k_mm_ug(long long FT, int U, int B, const int *__restrict__ moff, const int *__restrict__ mem,
                        const float2 *__restrict__ vis, float2 *__restrict__ ug)
{
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < FT * U; e += (long long)gridDim.x * blockDim.x) {
        const int u = (int)(e % U), code = mem[moff[u]];
        float2 v = vis[e / U * B + (code >> 1)];
        if (code & 1) v.y = -v.y;
        ug[e] = v;
    }
}

// several buffers from one allocation (a cudaMalloc takes tens of microseconds, and small handles are made often)
struct MmArena {
    size_t bytes = 0;
    std::vector<std::pair<void **, size_t>> at;
    template <typename T> void add(T **p, size_t count)
    {
        at.push_back({reinterpret_cast<void **>(p), bytes});
        bytes += (count * sizeof(T) + 255) / 256 * 256;
    }
    fm_status get(std::vector<void *> &owner)
    {
        char *q = nullptr;
        cudaError_t e = cudaMalloc(&q, bytes > 0 ? bytes : 16);
        if (e != cudaSuccess) return cuda_fail(e, "cudaMalloc (hour-angle modes)", __FILE__, __LINE__);
        owner.push_back(q);
        for (auto &x : at) *x.first = q + x.second;
        return FM_OK;
    }
};

// device buffers that live until the handle is complete
struct MmTemp {
    std::vector<void *> p;
    ~MmTemp() { for (void *q : p) cudaFree(q); }
};

// Smallest window of L cells around the nh in use (from LST lst0, q cells a pixel) whose ends the beam does not
// reach; 0 when there is none below 2 nh cells or a turn of hour angle, or when the beam is larger in the cells
// around those in use by more than MM_PEAK.
int mm_window(const Ctx &c, const std::vector<double> &bcoef, const std::vector<double> &domega, double lst0, int q,
              int nh, MmFft &p)
{
    const double dh = (c.cfg.ra_max - c.cfg.ra_min) / c.R / q, ddec = (c.cfg.dec_max - c.cfg.dec_min) / c.D;
    double bc = bcoef[0], bn = bcoef[0];           // of the widest and the narrowest beam
    for (double b : bcoef) {
        bc = std::fmax(bc, b);
        bn = std::fmin(bn, b);
    }
    if (!(bc < 0.0)) return 0;
    const double sl = std::sin(c.cfg.latitude_rad), cl = std::cos(c.cfg.latitude_rad);
    auto zenith_angle = [&](int d, int n) {        // of cell n; pi / 2 below the horizon (the step there)
        const double H = lst0 - (c.cfg.ra_min + ((double)((c.R - 1) * q - n) + 0.5 * q) * dh);
        const double dec = c.cfg.dec_min + (d + 0.5) * ddec;
        const double sU = sl * std::sin(dec) + cl * std::cos(dec) * std::cos(H);
        return sU > 0.0 ? std::acos(sU > 1.0 ? 1.0 : sU) : 0.5 * kPi;
    };
    auto weight = [&](int d, int n) {
        const double za = zenith_angle(d, n);
        return domega[d] * std::exp(bc * za * za);
    };
    // log of the narrowest beam's maximum over the declinations at cell n; none below the horizon
    auto narrow = [&](int n) {
        double t = -INFINITY;
        for (int d = 0; d < c.D; ++d) {
            const double za = zenith_angle(d, n);
            if (za < 0.5 * kPi && domega[d] > 0.0) t = std::fmax(t, std::log(domega[d]) + bn * za * za);
        }
        return t;
    };
    // the beam falls with |H|: its maximum in use is at the cell nearest the meridian
    const double turn = 2.0 * kPi / dh;
    double n0 = (c.R - 1) * q + 0.5 * q + (c.cfg.ra_min - lst0) / dh;
    n0 -= turn * std::rint((n0 - 0.5 * nh) / turn);
    const int at = (int)std::fmin(std::fmax(std::rint(n0), 0.0), nh - 1.0);
    const double used = narrow(at);
    double top = 0.0;
    for (int d = 0; d < c.D; ++d) top = std::fmax(top, weight(d, at));
    for (int L = nh + (nh & 1); L <= 2 * nh + 64 && L <= MM_MAXL && L * dh <= 2.0 * kPi; L += 2) {
        if (!smooth_factors(L, p)) continue;
        const int p0 = (L - nh) / 2;
        double edge = 0.0;
        for (int d = 0; d < c.D; ++d) edge = std::fmax(edge, std::fmax(weight(d, -p0), weight(d, L - 1 - p0)));
        if (edge <= MM_EDGE * top) {
            const int near = (int)std::fmin(std::fmax(std::rint(n0), -p0), L - 1 - p0);    // as `at`, in the window
            return narrow(near) - used <= std::log(MM_PEAK) ? L : 0;
        }
    }
    return 0;
}

// most turns of fringe per radian of hour angle of any baseline on the grid
double mm_rate(const Ctx &c)
{
    const double sl = std::sin(c.cfg.latitude_rad), cl = std::cos(c.cfg.latitude_rad);
    const double ddec = (c.cfg.dec_max - c.cfg.dec_min) / c.D;
    double cd = 0.0, nu = 0.0, b2 = 0.0;
    for (int d = 0; d < c.D; ++d) cd = std::fmax(cd, std::cos(c.cfg.dec_min + (d + 0.5) * ddec));
    for (double f : c.freq) nu = std::fmax(nu, f);
    for (int i = 0; i < c.A; ++i)
        for (int j = i + 1; j < c.A; ++j) {
            const double e = c.ant[3 * i] - c.ant[3 * j], n = c.ant[3 * i + 1] - c.ant[3 * j + 1],
                         u = c.ant[3 * i + 2] - c.ant[3 * j + 2], m = n * sl - u * cl;
            b2 = std::fmax(b2, e * e + m * m);
        }
    return std::sqrt(b2) * nu / kCLight * cd;
}

}  // namespace

// Table and index lists.  The form is used for Gaussian beams whose window fits (mm_window) and whose bands
// average at most half of the padded cells of the window, with the table in a quarter of the free device
// memory; otherwise c.mm.on stays false and the tensor-core forms run.
fm_status mm_setup(Ctx &c)
{
    MmState &s = c.mm;
    const FringeGroups &fg = c.fg;
    s.on = false;
    if (c.g.beam32 || c.R < 8 || c.F > 65535) return FM_OK;
    std::vector<double> bcoef(c.F), domega(c.D);
    FM_CK(cudaMemcpy(bcoef.data(), c.g.bcoef64, sizeof(double) * c.F, cudaMemcpyDeviceToHost));
    FM_CK(cudaMemcpy(domega.data(), c.g.domega64, sizeof(double) * c.D, cudaMemcpyDeviceToHost));
    const double dra = (c.cfg.ra_max - c.cfg.ra_min) / c.R;
    double lst0 = c.lst[0], lst1 = c.lst[0];
    for (double l : c.lst) {
        lst0 = std::fmin(lst0, l);
        lst1 = std::fmax(lst1, l);
    }
    // cells: those of the drift scan, whose whole-numbered tau_t allow any fringe rate; else as many a pixel
    // as put the fastest fringe and half a band below the Nyquist rate
    MmFft p;
    int q = fg.q, nh = fg.nh, L = 0;
    std::vector<double> tau(c.T);
    if (fg.drift) {
        for (int t = 0; t < c.T; ++t) tau[t] = (double)t * fg.k;
        L = mm_window(c, bcoef, domega, lst0, q, nh, p);
    } else {
        const double rate = mm_rate(c), span = (lst1 - lst0) / dra;
        if (!(span < 8.0 * c.R + 64.0)) return FM_OK;
        for (q = 1; q <= MM_MAXQ && L == 0; ++q) {
            nh = (c.R - 1) * q + (int)std::ceil(span * q) + 1;
            L = mm_window(c, bcoef, domega, lst0, q, nh, p);
            if (L == 0) return FM_OK;
            if (rate * L * (dra / q) + 24.0 > 0.45 * L) L = 0;
            else break;
        }
        for (int t = 0; t < c.T && L; ++t) tau[t] = (c.lst[t] - lst0) / dra * q;
    }
    if (L == 0) return FM_OK;
    s.L = L;
    s.q = q;
    const int p0 = (L - nh) / 2, U = fg.U, np = (c.D + 1) / 2;

    MmTemp tmp;
    size_t fr = 0, tot = 0;
    FM_CK(cudaMemGetInfo(&fr, &tot));
    if ((size_t)c.D * L * 32 + (size_t)c.F * c.D * L * 4 > fr / 4) return FM_OK;
    std::vector<double2> htw(L);
    for (int x = 0; x < L; ++x) htw[x] = make_double2(std::cos(2.0 * kPi * x / L), -std::sin(2.0 * kPi * x / L));
    double2 *tw = nullptr;
    MmDir *geo = nullptr;
    float *wt = nullptr;
    int2 *band = nullptr;
    MmArena ta;
    ta.add(&tw, L);
    ta.add(&geo, (size_t)c.D * L);
    ta.add(&band, (size_t)c.F * U);
    ta.add(&wt, (size_t)c.F * c.D * L);
    FM_TRY(ta.get(tmp.p));
    FM_CK(cudaMemcpy(tw, htw.data(), sizeof(double2) * L, cudaMemcpyHostToDevice));
    MmGeo ga;
    ga.lst0 = lst0; ga.ra_min = c.cfg.ra_min; ga.dra = dra;
    ga.dec_min = c.cfg.dec_min; ga.ddec = (c.cfg.dec_max - c.cfg.dec_min) / c.D; ga.lat = c.cfg.latitude_rad;
    ga.R = c.R; ga.D = c.D; ga.q = q; ga.L = L; ga.p0 = p0;
    k_mm_geo<<<cdiv(c.D * L, 256), 256>>>(ga, geo);
    FM_CK_LAUNCH();
    FM_CK(smem_opt_in(k_mm_band));
    k_mm_band<<<c.F * U, 256, (size_t)L * (3 * sizeof(double2) + sizeof(double))>>>(
        p, c.D, U, c.A, c.D > 16 ? c.D / 16 : 1, geo, tw, c.g.bcoef64, c.g.domega64, c.g.kap64, fg.uij, fg.ant, band);
    FM_CK_LAUNCH();
    std::vector<int2> hb((size_t)c.F * U);
    FM_CK(cudaMemcpy(hb.data(), band, sizeof(int2) * hb.size(), cudaMemcpyDeviceToHost));

    // elements sorted by |m|, then group, then place in the band
    auto signed_m = [&](int m) {
        m = ((m % L) + L) % L;
        return m > L / 2 ? m - L : m;
    };
    s.wmax = 1;
    s.nm = 2;
    s.ne = 0;
    int mlo = 0, mhi = 0;
    for (int2 &b : hb) {
        while (b.x + b.y / 2 > L / 2) b.x -= L;
        while (b.x + b.y / 2 <= -L / 2) b.x += L;
        if (!fg.drift && (b.x <= -L / 2 || b.x + b.y > L / 2)) return FM_OK;
        mlo = std::min(mlo, b.x);
        mhi = std::max(mhi, b.x + b.y + 3);
        s.wmax = std::max(s.wmax, b.y);
        s.ne += b.y;
        for (int i = 0; i < b.y; ++i) s.nm = std::max(s.nm, std::abs(signed_m(b.x + i)) + 1);
    }
    if (2 * s.ne > (long long)c.F * U * ((nh + 127) / 128 * 128)) return FM_OK;
    s.ld = (2 * s.nm + 3) / 4 * 4;
    s.mlo = mlo;
    s.pw = mhi - mlo + 2;
    s.vis_smem = ((size_t)((s.wmax + 3) / 4 * 4) * 64 + (size_t)MM_TC * s.pw) * sizeof(float2);
    FM_CK(cudaMemGetInfo(&fr, &tot));
    if (s.vis_smem > 200 * 1024 || s.ne >= (1LL << 29) || (size_t)s.ne * np * 16 > fr / 4) return FM_OK;
    const int nmt = (U + 63) / 64;
    std::vector<int> moff((size_t)c.F * (s.nm + 1)), code((size_t)nmt * c.F * s.wmax * 64, -1);
    std::vector<int4> items;
    int e = 0;
    std::vector<std::vector<int3>> at(s.nm);          // (group, place in its band, conjugated)
    for (int f = 0; f < c.F; ++f) {
        for (auto &v : at) v.clear();
        for (int u = 0; u < U; ++u) {
            const int2 b = hb[(size_t)f * U + u];
            for (int i = 0; i < b.y; ++i) {
                const int m = signed_m(b.x + i);
                at[std::abs(m)].push_back(make_int3(u, i, m < 0));
            }
        }
        for (int m = 0; m < s.nm; ++m) {
            moff[(size_t)f * (s.nm + 1) + m] = e;
            for (int r = 0; r < (int)at[m].size(); r += MM_ROWS)
                items.push_back(make_int4(f, m, e + r, std::min(MM_ROWS, (int)at[m].size() - r)));
            for (const int3 &x : at[m])
                code[(((size_t)(x.x >> 6) * c.F + f) * s.wmax + x.y) * 64 + (x.x & 63)] = 2 * e++ + x.z;
        }
        moff[(size_t)f * (s.nm + 1) + s.nm] = e;
    }
    s.nitem = (int)items.size();
    std::vector<float2> hph((size_t)c.T * s.pw);
    for (int t = 0; t < c.T; ++t)
        for (int i = 0; i < s.pw; ++i) {
            double turns = tau[t] * (i == s.pw - 1 ? 1 : mlo + i) / L;
            turns -= std::rint(turns);
            hph[(size_t)t * s.pw + i] = make_float2((float)std::cos(2.0 * kPi * turns), (float)std::sin(2.0 * kPi * turns));
        }
    // E^H E of a band by pivoted Cholesky, to 1e-10 of its trace (FP32 sums of the blocks: 1e-7)
    std::vector<std::vector<double>> fr_, fi_;
    {
        const int w = s.wmax;
        std::vector<double> kr(w, 0.0), ki(w, 0.0), left(w, (double)c.T);      // sum_t e^{2 pi i k tau_t / L}
        for (int k = 0; k < w; ++k)
            for (int t = 0; t < c.T; ++t) {
                const double ph = 2.0 * kPi * std::remainder(k * tau[t] / L, 1.0);
                kr[k] += std::cos(ph);
                ki[k] += std::sin(ph);
            }
        while ((int)fr_.size() < std::min(w, c.T)) {
            int pv = 0;
            double sum = 0.0;
            for (int i = 0; i < w; ++i) {
                sum += left[i];
                if (left[i] > left[pv]) pv = i;
            }
            if (sum <= 1e-10 * w * c.T) break;
            std::vector<double> r(w), q(w);
            const double inv = 1.0 / std::sqrt(left[pv]);
            for (int i = 0; i < w; ++i) {
                const int k = pv - i;                                            // K[i][pv] = k(pv - i)
                double a = kr[std::abs(k)], b = k < 0 ? -ki[-k] : ki[k];
                for (size_t j = 0; j < fr_.size(); ++j) {
                    a -= fr_[j][i] * fr_[j][pv] + fi_[j][i] * fi_[j][pv];
                    b -= fi_[j][i] * fr_[j][pv] - fr_[j][i] * fi_[j][pv];
                }
                r[i] = a * inv;
                q[i] = b * inv;
            }
            for (int i = 0; i < w; ++i) left[i] = std::fmax(0.0, left[i] - r[i] * r[i] - q[i] * q[i]);
            left[pv] = 0.0;
            fr_.push_back(r);
            fi_.push_back(q);
        }
    }
    s.nf = (int)fr_.size();
    std::vector<float2> hfac((size_t)s.nf * s.wmax);
    for (int j = 0; j < s.nf; ++j)
        for (int i = 0; i < s.wmax; ++i) hfac[(size_t)j * s.wmax + i] = make_float2((float)fr_[j][i], (float)-fi_[j][i]);
    MmArena pa;
    pa.add(&s.fac, hfac.size());
    pa.add(&s.tab, (size_t)s.ne * np);
    pa.add(&s.moff, moff.size());
    pa.add(&s.code, code.size());
    pa.add(&s.items, items.size());
    pa.add(&s.band, hb.size());
    pa.add(&s.ph, hph.size());
    pa.add(&s.z, 2 * (size_t)s.ne);
    pa.add(&s.w, s.ne);
    pa.add(&s.Y, 2 * (size_t)c.F * c.D * s.ld);
    pa.add(&s.G, (size_t)c.F * c.D * s.ld);
    pa.add(&s.b64, (size_t)s.ld * c.M);
    pa.add(&s.b32, (size_t)s.ld * c.M);
    pa.add(&s.pix, (size_t)s.ld * c.R);
    FM_TRY(pa.get(c.allocs));
    FM_CK(cudaMemcpy(s.fac, hfac.data(), sizeof(float2) * hfac.size(), cudaMemcpyHostToDevice));
    FM_CK(cudaMemcpy(s.moff, moff.data(), sizeof(int) * moff.size(), cudaMemcpyHostToDevice));
    FM_CK(cudaMemcpy(s.code, code.data(), sizeof(int) * code.size(), cudaMemcpyHostToDevice));
    FM_CK(cudaMemcpy(s.items, items.data(), sizeof(int4) * items.size(), cudaMemcpyHostToDevice));
    FM_CK(cudaMemcpy(s.band, hb.data(), sizeof(int2) * hb.size(), cudaMemcpyHostToDevice));
    FM_CK(cudaMemcpy(s.ph, hph.data(), sizeof(float2) * hph.size(), cudaMemcpyHostToDevice));

    // the basis holds sums of R values of at most 1: stored over 2^e >= R, which the table takes up
    const int e2 = (int)std::ceil(std::log2((double)c.R));
    k_mm_basis<<<1024, 128>>>(c.R, c.M, q, L, s.ld, std::ldexp(1.0, -e2), tw, c.g.phi64, s.b64, s.b32, s.pix);
    FM_CK_LAUNCH();
    k_mm_weight<<<2048, 256>>>(c.F, c.D, L, geo, c.g.bcoef64, c.g.domega64, wt);
    FM_CK_LAUNCH();
    FM_CK(smem_opt_in(k_mm_fill));
    k_mm_fill<<<c.F * U, 256, (size_t)L * 5 * sizeof(float2)>>>(p, c.F, c.D, U, c.A, p0, s.wmax,
                                                                (float)(std::ldexp(1.0, e2) / L), geo, wt, tw, c.g.kap64,
                                                                fg.uij, fg.ant, s.band, s.code, s.tab);
    FM_CK_LAUNCH();
    FM_CK(smem_opt_in(k_mm_vis));
    FM_CK(smem_opt_in(k_mm_maps));
    FM_CK(cudaDeviceSynchronize());
    s.on = true;
    return FM_OK;
}

// the groups' monopole visibilities from those of their first members
fm_status mm_group_monopole(Ctx &c, float *ug)
{
    k_mm_ug<<<1024, 256>>>((long long)c.F * c.T, c.fg.U, c.B, c.fg.moff, c.fg.mem, reinterpret_cast<const float2 *>(c.dc_u),
                           reinterpret_cast<float2 *>(ug));
    FM_CK_LAUNCH();
    FM_CK(cudaDeviceSynchronize());
    return FM_OK;
}

// forward of `nsky` skies whose modes are in c.mm.Y: rows of HaVSrc, `N` a contributor, sky s from row
// s * slot_rows
fm_status launch_mm_forward(Ctx &c, int nsky, int slot_rows, int N, float *vpart, cudaStream_t st)
{
    const MmState &s = c.mm;
    const int nmt = (c.fg.U + 63) / 64;
    return profiled(c, 0, st, [&]() -> fm_status {
        auto *kern = nsky == 2 ? k_mm_fwd<2> : k_mm_fwd<1>;
        kern<<<cdiv(s.nitem, 8), 256, 0, st>>>(s.nitem, s.items, c.D, s.ld, (long long)c.F * c.D * s.ld, s.tab, s.Y, 2 * s.ne,
                                               reinterpret_cast<float *>(s.z));
        FM_CK_LAUNCH();
        k_mm_vis<<<dim3(nmt * c.F, cdiv(c.T, MM_TC), nsky), 256, s.vis_smem, st>>>(
            c.F, c.T, c.fg.U, s.mlo, s.pw, s.wmax, s.code, s.band, s.ph, s.z, s.ne, slot_rows, N, vpart);
        FM_CK_LAUNCH();
        return FM_OK;
    });
}

// response maps j0 .. j0 + nj - 1 of channel f (k_mm_maps) for the group weights W[F][U]
fm_status launch_mm_maps(Ctx &c, int f, int j0, int nj, const float *W, float *X, cudaStream_t st)
{
    const MmState &s = c.mm;
    const int U = c.fg.U;
    if (nj > MM_JMAX) {
        set_error("at most %d response maps a launch", MM_JMAX);
        return FM_ERR_STATE;
    }
    k_mm_maps<<<dim3(cdiv((c.D + 1) / 2, MM_MAPP), U), 256, sizeof(float2) * (size_t)nj * s.wmax, st>>>(
        f, c.F, c.D, U, s.L, s.wmax, s.ld, nj, s.fac + (size_t)j0 * s.wmax, s.code, s.band, s.tab, W, (float)c.g.inv_sigma2, X);
    FM_CK_LAUNCH();
    return FM_OK;
}

fm_status launch_mm_adjoint(Ctx &c, const float *q32, cudaStream_t st)
{
    const MmState &s = c.mm;
    const int U = c.fg.U, nchunk = ((c.D + 1) / 2 + 31) / 32;
    return profiled(c, 1, st, [&]() -> fm_status {
        k_mm_q<<<dim3(cdiv(U, 8), c.F), 256, 0, st>>>(
            c.T, U, s.mlo, s.pw, s.wmax, s.code, s.band, s.ph, reinterpret_cast<const float2 *>(q32), s.w);
        FM_CK_LAUNCH();
        k_mm_adj<<<cdiv((long long)c.F * nchunk * (s.ld / 2), 4), 256, 0, st>>>(c.F, c.D, s.nm, s.ld, s.moff, s.tab, s.w, s.G);
        FM_CK_LAUNCH();
        return FM_OK;
    });
}

}  // namespace fm
