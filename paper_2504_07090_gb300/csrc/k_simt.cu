// CUDA-core kernels of the forward model and its adjoint, templated on the real type
// (double for the complex128 path, float for the plain FP32 path):
//   - separable mode <-> pixel transforms (Eq. fg_separable) as strided batched GEMMs;
//   - antenna phasors E_ip = exp(-2 pi i nu r_i . s_p / c) generated in-kernel, never
//     stored (b_pq = r_p - r_q makes K_pq = E_p conj(E_q), Eq. rime_discrete);
//   - the fringe contraction V_pq = sum_p w_p E_p conj(E_q), w = dOmega A x;
//   - gains, residual, chi^2 partials in FP64 and the adjoint weights (Eq. likelihood);
//   - the pixel adjoint xbar_p = dOmega A sum_{p<q} Re[conj(omega_pq) K_pq];
//   - deterministic reductions (fixed order, no floating-point atomics).
#include <algorithm>
#include <type_traits>

#include "fm_internal.cuh"
#include "phasor.cuh"

namespace fm {

__host__ __device__ __forceinline__ int pair_index(int i, int j, int A)
{
    return i * A - (i * (i + 1)) / 2 + (j - i - 1);
}

// ---------------------------------------------------------------- GEMM
struct GemmArgs {
    int M, N, K;
    long long sAb, sAi, sAk, sBb, sBk, sBj, sCb, sCi, sCj;
    int zero_b00;      // read B[0][0] of every batch as zero (drops the monopole mode a_00)
};

// FP32: 64 x 64 tiles, 128 threads of 8 x 4 sums (packed FMAs on column pairs: three 16-byte shared loads for 16 of
// them), the next 16 K values on their way in registers while the last are summed.  Each sum runs over K in order,
// 16 terms at a time (their rounding errors grow with K / 16 + 16, not K).  The four products of the mode transforms
// of 127 antennas, 128 channels, 256 x 256 modes: 1.10 (256 threads of 4 x 4 sums, no prefetch) -> 0.65 ms, 40
// TFLOP/s (0.58 ms with one running sum, whose errors were up to twice as large: FP32 gradient of 37 antennas
// against 64 bits 1.3e-7, now 5e-8).
constexpr int GM_LD = 68;
__global__ void __launch_bounds__(128) k_gemm(GemmArgs a, const float *__restrict__ A, const float *__restrict__ B,
                                              float *__restrict__ C)
{
    __shared__ __align__(16) float sA[2][16][GM_LD], sB[2][16][GM_LD];      // [slot][k][i], [k][j]
    const int b = blockIdx.z, i0 = blockIdx.y * 64, j0 = blockIdx.x * 64, tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    const float *Ab = A + b * a.sAb, *Bb = B + b * a.sBb;
    // element q of this thread in a 64 x 16 operand tile; the fastest thread index runs along the unit stride
    auto at = [&](bool k_fast, int q, int &i, int &k) {
        if (k_fast) {
            k = tid & 15;
            i = (tid >> 4) + 8 * q;
        } else {
            i = tid & 63;
            k = (tid >> 6) + 2 * q;
        }
    };
    const bool ak = a.sAk == 1, bk = a.sBk == 1;
    float ra[8], rb[8];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            int i, k;
            at(ak, q, i, k);
            ra[q] = i0 + i < a.M && k0 + k < a.K ? __ldg(Ab + (i0 + i) * a.sAi + (k0 + k) * a.sAk) : 0.f;
            at(bk, q, i, k);
            rb[q] = j0 + i < a.N && k0 + k < a.K && !(a.zero_b00 && j0 + i == 0 && k0 + k == 0)
                        ? __ldg(Bb + (k0 + k) * a.sBk + (j0 + i) * a.sBj)
                        : 0.f;
        }
    };
    auto stage = [&](int s) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            int i, k;
            at(ak, q, i, k);
            sA[s][k][i] = ra[q];
            at(bk, q, i, k);
            sB[s][k][i] = rb[q];
        }
    };
    float2 acc[8][2];
#pragma unroll
    for (int u = 0; u < 8; ++u) acc[u][0] = acc[u][1] = make_float2(0.f, 0.f);
    fetch(0);
    stage(0);
    __syncthreads();
    for (int k0 = 0, s = 0; k0 < a.K; k0 += 16, s ^= 1) {
        const bool more = k0 + 16 < a.K;
        if (more) fetch(k0 + 16);
        float2 t[8][2];
#pragma unroll
        for (int u = 0; u < 8; ++u) t[u][0] = t[u][1] = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const float4 p = *reinterpret_cast<const float4 *>(&sA[s][k][8 * ty]),
                         q = *reinterpret_cast<const float4 *>(&sA[s][k][8 * ty + 4]),
                         v = *reinterpret_cast<const float4 *>(&sB[s][k][4 * tx]);
            const float av[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
            const float2 b0 = make_float2(v.x, v.y), b1 = make_float2(v.z, v.w);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const float2 w = make_float2(av[u], av[u]);
                t[u][0] = __ffma2_rn(w, b0, t[u][0]);
                t[u][1] = __ffma2_rn(w, b1, t[u][1]);
            }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
#pragma unroll
            for (int q = 0; q < 2; ++q) acc[u][q] = make_float2(acc[u][q].x + t[u][q].x, acc[u][q].y + t[u][q].y);
        if (more) stage(s ^ 1);                 // last read before the previous barrier
        __syncthreads();
    }
    float *Cb = C + b * a.sCb;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int i = i0 + 8 * ty + u;
        const float v[4] = {acc[u][0].x, acc[u][0].y, acc[u][1].x, acc[u][1].y};
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (i < a.M && j0 + 4 * tx + q < a.N) Cb[i * a.sCi + (j0 + 4 * tx + q) * a.sCj] = v[q];
    }
}

// 16 x 16 tiles, one output a thread: the FP64 form.  FP64 runs at 2 lanes per SM and clock, so the shared
// memory reads of an untiled product are no bound, and small tiles waste nothing on padding and reach
// every SM (16 channels of 96 x 16 x 32: 111 us in 64 x 64 tiles on 32 SMs).
template <typename R>
__global__ void __launch_bounds__(256) k_gemm16(GemmArgs a, const R *__restrict__ A, const R *__restrict__ B,
                                                R *__restrict__ C)
{
    __shared__ R sA[16][17], sB[16][17];               // [i][k], [k][j]
    const int b = blockIdx.z, i0 = blockIdx.y * 16, j0 = blockIdx.x * 16, tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const R *Ab = A + b * a.sAb, *Bb = B + b * a.sBb;
    // the fastest thread index runs along the operand's unit stride
    const int ai = a.sAk == 1 ? ty : tx, ak = a.sAk == 1 ? tx : ty;
    const int bk = a.sBj == 1 ? ty : tx, bj = a.sBj == 1 ? tx : ty;
    R acc = R(0);
    for (int k0 = 0; k0 < a.K; k0 += 16) {
        sA[ai][ak] = i0 + ai < a.M && k0 + ak < a.K ? Ab[(i0 + ai) * a.sAi + (k0 + ak) * a.sAk] : R(0);
        sB[bk][bj] = k0 + bk < a.K && j0 + bj < a.N && !(a.zero_b00 && k0 + bk == 0 && j0 + bj == 0)
                         ? Bb[(k0 + bk) * a.sBk + (j0 + bj) * a.sBj]
                         : R(0);
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 16; ++k) acc += sA[ty][k] * sB[k][tx];
        __syncthreads();
    }
    if (i0 + ty < a.M && j0 + tx < a.N) C[b * a.sCb + (i0 + ty) * a.sCi + (j0 + tx) * a.sCj] = acc;
}

template <typename R>
static fm_status gemm(const GemmArgs &a, int batch, const R *A, const R *B, R *C, cudaStream_t st)
{
    if constexpr (std::is_same<R, double>::value)
        k_gemm16<R><<<dim3(cdiv(a.N, 16), cdiv(a.M, 16), batch), 256, 0, st>>>(a, A, B, C);
    else
        k_gemm<<<dim3(cdiv(a.N, 64), cdiv(a.M, 64), batch), 128, 0, st>>>(a, A, B, C);
    FM_CK_LAUNCH();
    return FM_OK;
}

template <typename R> static const R *tab_phi(const Ctx &c);
template <> const double *tab_phi<double>(const Ctx &c) { return c.g.phi64; }
template <> const float *tab_phi<float>(const Ctx &c) { return c.g.phi32; }
template <typename R> static const R *tab_leg(const Ctx &c);
template <> const double *tab_leg<double>(const Ctx &c) { return c.g.leg64; }
template <> const float *tab_leg<float>(const Ctx &c) { return c.g.leg32; }

// x[f][d][r] = sum_n P[d][n] sum_m Phi[r][m] a[f][m][n]   (Eq. fg_separable)
template <typename R>
fm_status launch_modes_forward(Ctx &c, const R *a, R *x, cudaStream_t st, int skip_dc, unsigned *xmax,
                               const StripArgs *strips)
{
    if constexpr (std::is_same<R, float>::value)
        if (c.mtc.on) return launch_modes_tc_forward(c, a, x, st, skip_dc, xmax, strips);
    if (xmax || strips) {
        set_error("channel maxima are formed only by the tensor-core mode transform");
        return FM_ERR_STATE;
    }
    R *t1 = (R *)c.tmp;
    GemmArgs s1{c.R, c.N, c.M, 0, c.M, 1, c.nk, c.N, 1, (long long)c.R * c.N, c.N, 1, skip_dc};
    FM_TRY(gemm<R>(s1, c.F, tab_phi<R>(c), a, t1, st));
    GemmArgs s2{c.D, c.R, c.N, 0, c.N, 1, (long long)c.R * c.N, 1, c.N, c.npix, c.R, 1, 0};
    return gemm<R>(s2, c.F, tab_leg<R>(c), t1, x, st);
}

// abar[f][m][n] = sum_r Phi[r][m] sum_d xbar[f][d][r] P[d][n]   (transpose of the above)
template <typename R>
fm_status launch_modes_adjoint(Ctx &c, const R *xbar, R *abar, cudaStream_t st)
{
    if constexpr (std::is_same<R, float>::value)
        if (c.mtc.on) return launch_modes_tc_adjoint(c, xbar, abar, st);
    R *t2 = (R *)c.tmp;
    GemmArgs s1{c.R, c.N, c.D, c.npix, 1, c.R, 0, c.N, 1, (long long)c.R * c.N, c.N, 1, 0};
    FM_TRY(gemm<R>(s1, c.F, xbar, tab_leg<R>(c), t2, st));
    GemmArgs s2{c.M, c.N, c.R, 0, 1, c.M, (long long)c.R * c.N, c.N, 1, c.nk, c.N, 1, 0};
    return gemm<R>(s2, c.F, tab_phi<R>(c), t2, abar, st);
}

// the same between sky modes (or pixels) and hour-angle modes (k_mm.cu): Y[f][d][c] with the RA basis B[c][m]
fm_status launch_mm_from_modes(Ctx &c, const float *a, int slot, cudaStream_t st, int skip_dc)
{
    const MmState &s = c.mm;
    float *y = s.Y + (size_t)slot * c.F * c.D * s.ld;
    if (s.ra.img) return launch_modes_tc_forward(c, a, y, st, skip_dc, nullptr, nullptr, &s.ra);
    const long long tn = (long long)s.ld * c.N;
    GemmArgs s1{s.ld, c.N, c.M, 0, c.M, 1, c.nk, c.N, 1, tn, c.N, 1, skip_dc};
    FM_TRY(gemm<float>(s1, c.F, s.b32, a, s.tmp, st));
    GemmArgs s2{c.D, s.ld, c.N, 0, c.N, 1, tn, 1, c.N, (long long)c.D * s.ld, s.ld, 1, 0};
    return gemm<float>(s2, c.F, tab_leg<float>(c), s.tmp, y, st);
}

fm_status launch_mm_from_pixels(Ctx &c, const float *x, int slot, cudaStream_t st)
{
    const MmState &s = c.mm;
    GemmArgs g{c.D, s.ld, c.R, c.npix, c.R, 1, 0, 1, c.R, (long long)c.D * s.ld, s.ld, 1, 0};
    return gemm<float>(g, c.F, x, s.pix, s.Y + (size_t)slot * c.F * c.D * s.ld, st);
}

fm_status launch_mm_to_modes(Ctx &c, float *abar, cudaStream_t st)
{
    const MmState &s = c.mm;
    if (s.ra.img) return launch_modes_tc_adjoint(c, s.G, abar, st, &s.ra);
    const long long tn = (long long)s.ld * c.N;
    GemmArgs s1{s.ld, c.N, c.D, (long long)c.D * s.ld, 1, s.ld, 0, c.N, 1, tn, c.N, 1, 0};
    FM_TRY(gemm<float>(s1, c.F, s.G, tab_leg<float>(c), s.tmp, st));
    GemmArgs s2{c.M, c.N, s.ld, 0, 1, c.M, tn, c.N, 1, c.nk, c.N, 1, 0};
    return gemm<float>(s2, c.F, s.b32, s.tmp, abar, st);
}

// ---------------------------------------------------------------- gains
template <typename R>
__global__ void k_gains(DevGeom g, const R *__restrict__ gamma, R *__restrict__ out)
{
    int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= g.F * g.A) return;
    int f = e / g.A, i = e % g.A;
    const R *X = Tab<R>::gleg(g) + (size_t)f * g.NG;
    R re = 0, im = 0;
    for (int k = 0; k < g.NG; ++k) {
        re += X[k] * gamma[(i * g.NG + k) * 2];
        im += X[k] * gamma[(i * g.NG + k) * 2 + 1];
    }
    out[2 * e] = re;
    out[2 * e + 1] = im;
}

template <typename R>
fm_status launch_gains(Ctx &c, const R *gamma, R *g, cudaStream_t st)
{
    k_gains<R><<<cdiv(c.F * c.A, 128), 128, 0, st>>>(c.g, gamma, g);
    FM_CK_LAUNCH();
    return FM_OK;
}

// m_pq = g_p conj(g_q) V_pq
template <typename R>
__global__ void k_apply_gains(DevGeom g, const R *__restrict__ vis, const R *__restrict__ gains, R *__restrict__ out)
{
    long long n = (long long)g.F * g.T * g.B;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        int b = (int)(e % g.B);
        int f = (int)(e / ((long long)g.T * g.B));
        int i = g.bl_i[b], j = g.bl_j[b];
        R gir = gains[2 * (f * g.A + i)], gii = gains[2 * (f * g.A + i) + 1];
        R gjr = gains[2 * (f * g.A + j)], gji = gains[2 * (f * g.A + j) + 1];
        R ggr = gir * gjr + gii * gji, ggi = gii * gjr - gir * gji;   // g_i conj(g_j)
        R vr = vis[2 * e], vi = vis[2 * e + 1];
        out[2 * e] = ggr * vr - ggi * vi;
        out[2 * e + 1] = ggr * vi + ggi * vr;
    }
}

template <typename R>
fm_status launch_apply_gains(Ctx &c, const R *vis, const R *g, R *out, cudaStream_t st)
{
    k_apply_gains<R><<<1024, 256, 0, st>>>(c.g, vis, g, out);
    FM_CK_LAUNCH();
    return FM_OK;
}

// ---------------------------------------------------------------- forward contraction
// One CTA per (channel, LST).  Pixels stream through shared memory in chunks of PC:
// E and w E are generated there, then each thread accumulates 4x4 antenna tiles
// (p-block <= q-block) of sum_p (w E_p) conj(E_q).  Threads are split into pixel
// groups whose partial sums are added in a fixed order at the end.
template <typename R, int TPT>
__global__ void __launch_bounds__(256) k_vis_simt(DevGeom g, const R *__restrict__ x, R *__restrict__ vis, int nbk,
                                                  int ntile, int tpg, int ngrp, int pc)
{
    using C2 = typename V2<R>::t;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C2 *sEw = reinterpret_cast<C2 *>(smem_raw);
    C2 *sE = sEw + (size_t)pc * g.apad;
    const int ft = blockIdx.x, f = ft / g.T, t = ft % g.T;
    const int tid = threadIdx.x, grp = tid / tpg, lane = tid % tpg;
    int tbi[TPT], tbj[TPT];
    bool tact[TPT];
#pragma unroll
    for (int k = 0; k < TPT; ++k) {
        int tile = lane + k * tpg;
        tact[k] = (grp < ngrp) && (tile < ntile);
        int bi = 0, off = 0;
        if (tact[k]) {
            while (off + (nbk - bi) <= tile) { off += nbk - bi; ++bi; }
        }
        tbi[k] = bi;
        tbj[k] = bi + (tile - off);
    }
    R acc[TPT][4][4][2];
#pragma unroll
    for (int k = 0; k < TPT; ++k)
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[k][u][v][0] = acc[k][u][v][1] = R(0);

    const R *xf = x + (size_t)f * g.npix;
    R *sW = reinterpret_cast<R *>(sE + (size_t)pc * g.apad);       // [pc]
    for (int p0 = 0; p0 < g.npix; p0 += pc) {
        __syncthreads();
        for (int pl = tid; pl < pc; pl += blockDim.x) {
            int p = p0 + pl;
            sW[pl] = (p < g.npix) ? pixel_weight<R>(g, f, t, p) * xf[p] : R(0);
        }
        __syncthreads();
        for (int e = tid; e < pc * g.apad; e += blockDim.x) {
            int pl = e / g.apad, i = e % g.apad, p = p0 + pl;
            C2 ev, ew;
            ev.x = ev.y = ew.x = ew.y = R(0);
            if (i < g.A && p < g.npix) {
                R w = sW[pl];
                R er, ei;
                Phasor<R>::eval(g, f, i, t, p, er, ei);
                ev.x = er; ev.y = ei;
                ew.x = w * er; ew.y = w * ei;
            }
            sE[e] = ev;
            sEw[e] = ew;
        }
        __syncthreads();
        if (grp < ngrp) {
            // chunk partial sums first, then one add into the running total: the
            // rounding error grows with pc/ngrp + npix/pc terms instead of npix/ngrp
#pragma unroll
            for (int k = 0; k < TPT; ++k) {
                if (!tact[k]) continue;
                R part[4][4][2];
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int v = 0; v < 4; ++v) part[u][v][0] = part[u][v][1] = R(0);
                for (int pl = grp; pl < pc; pl += ngrp) {
                    const C2 *rw = sEw + (size_t)pl * g.apad;
                    const C2 *rv = sE + (size_t)pl * g.apad;
                    C2 av[4], bv[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) { av[q] = rw[4 * tbi[k] + q]; bv[q] = rv[4 * tbj[k] + q]; }
#pragma unroll
                    for (int u = 0; u < 4; ++u)
#pragma unroll
                        for (int v = 0; v < 4; ++v) {
                            part[u][v][0] += av[u].x * bv[v].x + av[u].y * bv[v].y;
                            part[u][v][1] += av[u].y * bv[v].x - av[u].x * bv[v].y;
                        }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        acc[k][u][v][0] += part[u][v][0];
                        acc[k][u][v][1] += part[u][v][1];
                    }
            }
        }
    }
    __syncthreads();
    R *red = reinterpret_cast<R *>(smem_raw);       // [ngrp][ntile][16][2]
#pragma unroll
    for (int k = 0; k < TPT; ++k) {
        if (!tact[k]) continue;
        int tile = lane + k * tpg;
        R *dst = red + ((size_t)grp * ntile + tile) * 32;
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                dst[(u * 4 + v) * 2] = acc[k][u][v][0];
                dst[(u * 4 + v) * 2 + 1] = acc[k][u][v][1];
            }
    }
    __syncthreads();
    for (int e = tid; e < ntile * 16; e += blockDim.x) {
        int tile = e / 16, q = e % 16, u = q / 4, v = q % 4;
        int bi = 0, off = 0;
        while (off + (nbk - bi) <= tile) { off += nbk - bi; ++bi; }
        int bj = bi + (tile - off);
        int i = 4 * bi + u, j = 4 * bj + v;
        if (i < j && j < g.A) {
            R re = 0, im = 0;
            for (int gq = 0; gq < ngrp; ++gq) {
                re += red[((size_t)gq * ntile + tile) * 32 + 2 * q];
                im += red[((size_t)gq * ntile + tile) * 32 + 2 * q + 1];
            }
            size_t o = ((size_t)ft * g.B + pair_index(i, j, g.A)) * 2;
            vis[o] = re;
            vis[o + 1] = im;
        }
    }
}

// antenna tiles (ntile of them, TPT a thread) and shared memory of the direct forward, and whether the
// array fits; the drift-scan form takes the same arrays, so that what an FP64 or FP32 handle supports
// does not depend on its LSTs
struct VisSimtPlan {
    int nbk, ntile, tpt, tpg, ngrp, pc;
    size_t smem;
};

template <typename R>
static fm_status vis_simt_plan(const Ctx &c, VisSimtPlan &p)
{
    p.nbk = (c.A + 3) / 4;
    p.ntile = p.nbk * (p.nbk + 1) / 2;
    p.tpt = p.ntile <= 256 ? 1 : p.ntile <= 512 ? 2 : p.ntile <= 1024 ? 4 : 8;
    p.tpg = (((int)cdiv(p.ntile, p.tpt) + 31) / 32) * 32;
    if (p.tpg > 256) { set_error("direct forward: %d antennas exceed the tile layout", c.A); return FM_ERR_UNSUPPORTED; }
    p.ngrp = 256 / p.tpg;
    // pixels staged per round: 64, halved while the phasor tiles exceed shared memory
    const size_t sm_r = (size_t)p.ngrp * p.ntile * 32 * sizeof(R);
    for (p.pc = 64;; p.pc /= 2) {
        const size_t sm_e = 2 * (size_t)p.pc * c.g.apad * 2 * sizeof(R) + p.pc * sizeof(R);
        p.smem = sm_e > sm_r ? sm_e : sm_r;
        if (p.smem <= 227 * 1024 || p.pc <= 8) break;
    }
    if (p.smem > 227 * 1024) { set_error("direct forward: tiles exceed shared memory"); return FM_ERR_UNSUPPORTED; }
    return FM_OK;
}

template <typename R>
static size_t adj_simt_smem(const Ctx &c) { return ((size_t)c.A * 128 + c.B) * 2 * sizeof(R); }

template <typename R>
fm_status simt_supports(const Ctx &c, bool adjoint)
{
    VisSimtPlan p;
    if (!adjoint) return vis_simt_plan<R>(c, p);
    if (adj_simt_smem<R>(c) <= 227 * 1024) return FM_OK;
    set_error("direct adjoint: %d antennas exceed shared memory", c.A);
    return FM_ERR_UNSUPPORTED;
}
template fm_status simt_supports<float>(const Ctx &, bool);
template fm_status simt_supports<double>(const Ctx &, bool);

template <typename R, int TPT>
static fm_status vis_simt_launch(Ctx &c, const VisSimtPlan &p, const R *x, R *vis, cudaStream_t st)
{
    FM_CK(smem_opt_in(k_vis_simt<R, TPT>));
    k_vis_simt<R, TPT><<<c.F * c.T, 256, p.smem, st>>>(c.g, x, vis, p.nbk, p.ntile, p.tpg, p.ngrp, p.pc);
    FM_CK_LAUNCH();
    return FM_OK;
}

template <typename R>
fm_status launch_vis(Ctx &c, const R *x, R *vis, cudaStream_t st)
{
    VisSimtPlan p;
    FM_TRY(vis_simt_plan<R>(c, p));
    switch (p.tpt) {
    case 1: return vis_simt_launch<R, 1>(c, p, x, vis, st);
    case 2: return vis_simt_launch<R, 2>(c, p, x, vis, st);
    case 4: return vis_simt_launch<R, 4>(c, p, x, vis, st);
    default: return vis_simt_launch<R, 8>(c, p, x, vis, st);
    }
}

// ---------------------------------------------------------------- chi^2 epilogue
// ---- pieces of the per-(channel, LST) epilogues k_chi2_ft and k_hvp_ft

__device__ __forceinline__ float hv_scale(const HaVSrc &hv, int f)
{
    const float mx = __uint_as_float(hv.xmax[f]);
    float s2 = 1.f;
    if (mx > 0.f && isfinite(mx)) {
        int ex;
        frexpf(mx, &ex);
        s2 = ldexpf(1.f, 14 - ex);
    }
    return 1.f / (hv.sp * s2);
}

// the contributors' partial rows 2 u, 2 u + 1 of the forward at LST t of channel f, added in rank order
__device__ __forceinline__ float2 hv_row(const HaVSrc &hv, int f, int t, int u)
{
    const int seg = (u >> 6) * hv.F + f, nc = hv.ncontrib[seg];
    const float2 *src = reinterpret_cast<const float2 *>(hv.vpart + ((size_t)seg * hv.J * hv.npad + t) * 128) + (u & 63);
    const size_t js = (size_t)hv.npad * 64;
    float2 a = make_float2(0.f, 0.f);
    for (int j0 = 0; j0 < nc; j0 += 4) {
        float2 v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = j0 + q < nc ? src[(size_t)(j0 + q) * js] : make_float2(0.f, 0.f);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (j0 + q < nc) {
                a.x += v[q].x;
                a.y += v[q].y;
            }
    }
    return a;
}

// sV[u]: V of every group at LST t of channel f, with the roundings of k_ha_vfinish, so that a member's value
// (sV[u], conjugated when reversed) equals the finished forward's bitwise
template <int NT>
__device__ __forceinline__ void group_vis(const HaVSrc &hv, int f, int t, int ft, int U, float2 *sV)
{
    const float sc = hv_scale(hv, f), cf = hv.dc ? hv.dc[(size_t)f * hv.dcs] : 0.f;
    for (int u = threadIdx.x; u < U; u += NT) {
        const float2 v = hv_row(hv, f, t, u);
        float2 V = make_float2(__fmul_rn(v.x, sc), __fmul_rn(v.y, sc));
        if (hv.dc) {
            const float2 m = reinterpret_cast<const float2 *>(hv.ug)[(size_t)ft * U + u];
            V = make_float2(__fmaf_rn(cf, m.x, V.x), __fmaf_rn(cf, m.y, V.y));
        }
        sV[u] = V;
    }
}

__device__ __forceinline__ float2 member_vis(const float2 *sV, int code)
{
    const float2 v = sV[code >> 1];
    return make_float2(v.x, (code & 1) ? -v.y : v.y);
}

// q32[ft][u] = the groups' sums of sW (conjugated for reversed members); returns the largest |Re|, |Im| that
// this thread stored.  Four lanes a group, each every fourth member, added in a fixed order: one lane a
// group left three quarters of the threads idle over up to 126 members.
template <int NT, typename C2>
__device__ __forceinline__ float group_sums(const C2 *sW, int ft, int U, const int *__restrict__ moff,
                                            const int *__restrict__ mem, float *__restrict__ q32)
{
    const int tid = threadIdx.x;
    float qm = 0.f;
    for (int u0 = 0; u0 < U; u0 += NT / 4) {
        const int u = u0 + (tid >> 2);
        float qr = 0.f, qi = 0.f;
        if (u < U) {
            const int m1 = moff[u + 1];
#pragma unroll 2
            for (int m = moff[u] + (tid & 3); m < m1; m += 4) {
                const int code = mem[m], b = code >> 1;
                qr += (float)sW[b].x;
                qi += (code & 1) ? -(float)sW[b].y : (float)sW[b].y;
            }
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            qr += __shfl_xor_sync(0xffffffffu, qr, o);
            qi += __shfl_xor_sync(0xffffffffu, qi, o);
        }
        if (u < U && (tid & 3) == 0) {
            *reinterpret_cast<float2 *>(q32 + ((size_t)ft * U + u) * 2) = make_float2(qr, qi);
            qm = fmaxf(qm, fmaxf(fabsf(qr), fabsf(qi)));
        }
    }
    return qm;
}

// sZ[tid]: chunk c = tid mod nc, nc = NT / A, of Z_a, a = tid div nc: partners j = c, c + nc, ... (j != a);
// pair_index(a, j) = rowa + j for j > a
template <int NT, typename C2>
__device__ __forceinline__ void antenna_chunks(const C2 *sTi, const C2 *sTj, int A, C2 *sZ)
{
    using R = decltype(C2::x);
    const int tid = threadIdx.x, nc = NT / A;
    if (tid >= nc * A) return;
    const int a = tid / nc, c = tid - a * nc;
    const int rowa = a * A - (a * (a + 1)) / 2 - a - 1;
    R zr = 0, zi = 0;
    for (int j = c; j < A; j += nc) {
        if (j == a) continue;
        const C2 t = j > a ? sTi[rowa + j] : sTj[pair_index(j, a, A)];
        zr += t.x;
        zi += t.y;
    }
    sZ[tid].x = zr;
    sZ[tid].y = zi;
}

// after a barrier: zpart[ft][a] = the chunks of Z_a in order, over sigma^2
template <int NT, typename R, typename C2>
__device__ __forceinline__ void antenna_totals(const C2 *sZ, int A, int ft, R is2, R *__restrict__ zpart)
{
    const int tid = threadIdx.x, nc = NT / A;
    if (tid >= A) return;
    R zr = 0, zi = 0;
    for (int c = 0; c < nc; ++c) {
        zr += sZ[tid * nc + c].x;
        zi += sZ[tid * nc + c].y;
    }
    zpart[((size_t)ft * A + tid) * 2] = zr * is2;
    zpart[((size_t)ft * A + tid) * 2 + 1] = zi * is2;
}

// One CTA per (channel, LST): model, residual, chi^2 partial (a warp's terms summed in the
// working type, the warps' sums in FP64), the adjoint weights
// omega_pq = conj(g_p) g_q r_pq / sigma^2 and the per-antenna gain partials
// Z_a = [sum_{q>a} r_aq g_q conj(V_aq) + sum_{p<a} conj(r_pa) g_p V_pa] / sigma^2.  The two
// terms of every baseline are formed once, with its residual; Z_a then sums its A - 1 terms
// in NT / A interleaved chunks (one thread each) and adds the chunks in order.  The
// gains g_i(nu_f) = sum_k X_k(nu_f) gamma_ik are formed from the coefficients gamma in the
// prologue.  With q32 != NULL (hour-angle form) omega is not written: its sums over the
// baseline groups go to q32[f][t][u] and their largest |Re|, |Im| to qmax_ft[f][t].  With
// hv.vpart != NULL (hour-angle form, one LST pass) V is formed here from the forward's partial
// sums and the groups' monopole visibilities (HaVSrc) instead of being read from vis.  Needs
// A <= CF_THREADS.
//
// Eight CTAs of 256 threads an SM while a (channel, LST)'s terms (24 bytes a baseline) are small; handles of the
// hour-angle form run k_chi2_group below where they are not.
constexpr int CF_THREADS = 256;
template <typename R>
__global__ void __launch_bounds__(CF_THREADS, sizeof(R) == 4 ? 8 : 1) k_chi2_ft(DevGeom g, const R *__restrict__ vis, const R *__restrict__ data,
                                                        const R *__restrict__ gamma, R *__restrict__ omega,
                                                        R *__restrict__ zpart, double *__restrict__ chi2p, int U,
                                                        const int *__restrict__ moff, const int *__restrict__ mem,
                                                        float *__restrict__ q32, float *__restrict__ qmax_ft,
                                                        const R *__restrict__ rin, HaVSrc hv)
{
    using C2 = typename V2<R>::t;
    constexpr int NT = CF_THREADS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C2 *sG = reinterpret_cast<C2 *>(smem_raw);            // [A]
    C2 *sTi = sG + g.A;                                    // [B] term of baseline (i, j) in Z_i
    C2 *sTj = sTi + g.B;                                   // [B] term of baseline (i, j) in Z_j
    C2 *sW = sTj + g.B;                                    // [B] omega (hour-angle form)
    float2 *sV = reinterpret_cast<float2 *>(sW + g.B);     // [U] V of the groups (hv)
    __shared__ C2 sZ[NT];                          // chunk sums of Z_a
    __shared__ double dred[NT / 32];
    __shared__ float fred[NT / 32];
    const int ft = blockIdx.x, f = ft / g.T, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    {
        const R *X = Tab<R>::gleg(g) + (size_t)f * g.NG;
        for (int i = tid; i < g.A; i += NT) {     // as k_gains
            R re = 0, im = 0;
            for (int k = 0; k < g.NG; ++k) {
                re += X[k] * gamma[(i * g.NG + k) * 2];
                im += X[k] * gamma[(i * g.NG + k) * 2 + 1];
            }
            sG[i].x = re;
            sG[i].y = im;
        }
    }
    if (hv.vpart) group_vis<NT>(hv, f, ft - f * g.T, ft, U, sV);
    __syncthreads();
    const R is2 = (R)g.inv_sigma2;
    const C2 *vrow = vis ? reinterpret_cast<const C2 *>(vis) + (size_t)ft * g.B : nullptr;
    const C2 *drow = reinterpret_cast<const C2 *>(data) + (size_t)ft * g.B;
    // rin != NULL (delay filter): the residual weights come in precomputed, sigma^2 F^T W F r
    const C2 *rrow = rin ? reinterpret_cast<const C2 *>(rin) + (size_t)ft * g.B : nullptr;
    C2 *orow = reinterpret_cast<C2 *>(omega) + (size_t)ft * g.B;
    R c2 = 0;   // a warp's terms in the working type; FP64 across warps
    for (int b = tid; b < g.B; b += NT) {
        int i, j;
        C2 V;
        if (hv.vpart) {
            const int2 pr = __ldg(hv.pairs + b);
            i = pr.x & 0xffff;
            j = pr.x >> 16;
            const float2 v = member_vis(sV, pr.y);
            V.x = (R)v.x;
            V.y = (R)v.y;
        } else {
            i = g.bl_i[b];
            j = g.bl_j[b];
            V = vrow[b];
        }
        const C2 d = drow[b], gi = sG[i], gj = sG[j];
        const R ggr = gi.x * gj.x + gi.y * gj.y, ggi = gi.y * gj.x - gi.x * gj.y;     // g_i conj(g_j)
        C2 r, om, ti, tj;
        if (rrow) {
            r = rrow[b];
        } else {
            r.x = ggr * V.x - ggi * V.y - d.x;
            r.y = ggr * V.y + ggi * V.x - d.y;
        }
        c2 += r.x * r.x + r.y * r.y;
        om.x = (ggr * r.x + ggi * r.y) * is2;
        om.y = (ggr * r.y - ggi * r.x) * is2;
        if (q32) sW[b] = om;
        else orow[b] = om;
        {   // r g_j conj(V), the term in Z_i
            const R pr = r.x * gj.x - r.y * gj.y, pi = r.x * gj.y + r.y * gj.x;
            ti.x = pr * V.x + pi * V.y;
            ti.y = pi * V.x - pr * V.y;
        }
        {   // conj(r) g_i V, the term in Z_j
            const R pr = r.x * gi.x + r.y * gi.y, pi = r.x * gi.y - r.y * gi.x;
            tj.x = pr * V.x - pi * V.y;
            tj.y = pr * V.y + pi * V.x;
        }
        sTi[b] = ti;
        sTj[b] = tj;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c2 += __shfl_xor_sync(0xffffffffu, c2, o);
    if (lane == 0) dred[w] = (double)c2;
    __syncthreads();
    if (tid == 0) {
        double a = 0.0;
        for (int k = 0; k < NT / 32; ++k) a += dred[k];
        chi2p[ft] = a * g.inv_sigma2;
    }
    if (q32) {
        float qm = group_sums<NT>(sW, ft, U, moff, mem, q32);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) qm = fmaxf(qm, __shfl_xor_sync(0xffffffffu, qm, o));
        if (lane == 0) fred[w] = qm;
    }
    antenna_chunks<NT>(sTi, sTj, g.A, sZ);
    __syncthreads();
    if (q32 && tid == 0) {
        float m = 0.f;
        for (int k = 0; k < NT / 32; ++k) m = fmaxf(m, fred[k]);
        qmax_ft[ft] = m;
    }
    antenna_totals<NT>(sZ, g.A, ft, is2, zpart);
}

// The same for large arrays of the hour-angle form, whose visibilities are those of the fringe groups: V_u
// (finished here from the forward's partial sums, hv, or taken from the finished vis) and the residuals are all
// that a CTA keeps, 8 bytes a baseline instead of the 24 of both gain terms and omega.  The sums over the groups' members
// (q32, their largest |Re|, |Im| to qmax_ft) and over the antennas' partners form their terms again from those,
// the reversed partner of a pair as its conjugate.
//
// Bound: latency of the loads and barriers of one (channel, LST), so what counts is the CTAs an SM holds: three
// of 512 with 127 antennas (64 KB of residuals; 192 KB with 24 bytes a baseline, one CTA).  127 antennas, 128
// channels, 120 LSTs: 1.68 -> 1.10 ms (two CTAs of 1024: 1.23 ms).  With 37 antennas k_chi2_ft is the faster one
// (33 against 36 us).
constexpr int CG_THREADS = 512;
__global__ void __launch_bounds__(CG_THREADS, 3)
k_chi2_group(DevGeom g, const float *__restrict__ vis, const float *__restrict__ data, const float *__restrict__ gamma,
             float *__restrict__ zpart, double *__restrict__ chi2p, int U, const int2 *__restrict__ pairs,
             const int2 *__restrict__ gmem, const int *__restrict__ moff, float *__restrict__ q32,
             float *__restrict__ qmax_ft, const float *__restrict__ rin, HaVSrc hv)
{
    constexpr int NT = CG_THREADS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *sG = reinterpret_cast<float2 *>(smem_raw);     // [A]
    float2 *sV = sG + g.A;                                 // [U]
    float2 *sR = sV + U;                                   // [B] residuals
    __shared__ float2 sZ[NT];                              // chunk sums of Z_a
    __shared__ double dred[NT / 32];
    __shared__ float fred[NT / 32];
    const int ft = blockIdx.x, f = ft / g.T, t = ft - f * g.T, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    {
        const float *X = g.gleg32 + (size_t)f * g.NG;
        for (int i = tid; i < g.A; i += NT) {              // as k_gains
            float re = 0, im = 0;
            for (int k = 0; k < g.NG; ++k) {
                re += X[k] * gamma[(i * g.NG + k) * 2];
                im += X[k] * gamma[(i * g.NG + k) * 2 + 1];
            }
            sG[i] = make_float2(re, im);
        }
    }
    if (hv.vpart) {
        group_vis<NT>(hv, f, t, ft, U, sV);
    } else {
        const float2 *vrow = reinterpret_cast<const float2 *>(vis) + (size_t)ft * g.B;
        for (int u = tid; u < U; u += NT) {                // the first member's
            const int code = gmem[moff[u]].x;
            const float2 v = vrow[code >> 1];
            sV[u] = make_float2(v.x, (code & 1) ? -v.y : v.y);
        }
    }
    __syncthreads();
    const float is2 = (float)g.inv_sigma2;
    const float2 *drow = reinterpret_cast<const float2 *>(data) + (size_t)ft * g.B;
    // rin != NULL (delay filter): the residual weights come in precomputed, sigma^2 F^T W F r
    const float2 *rrow = rin ? reinterpret_cast<const float2 *>(rin) + (size_t)ft * g.B : nullptr;
    float c2 = 0;
#pragma unroll 2
    for (int b = tid; b < g.B; b += NT) {
        float2 r;
        if (rrow) {
            r = rrow[b];
        } else {
            const int2 p = __ldg(pairs + b);               // i | j << 16, 2 u + reversed
            const float2 d = __ldg(drow + b), gi = sG[p.x & 0xffff], gj = sG[p.x >> 16];
            float2 V = sV[p.y >> 1];
            if (p.y & 1) V.y = -V.y;
            const float ggr = gi.x * gj.x + gi.y * gj.y, ggi = gi.y * gj.x - gi.x * gj.y;     // g_i conj(g_j)
            r.x = ggr * V.x - ggi * V.y - d.x;
            r.y = ggr * V.y + ggi * V.x - d.y;
        }
        c2 += r.x * r.x + r.y * r.y;
        sR[b] = r;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c2 += __shfl_xor_sync(0xffffffffu, c2, o);
    if (lane == 0) dred[w] = (double)c2;
    __syncthreads();
    if (tid == 0) {
        double a = 0.0;
        for (int k = 0; k < NT / 32; ++k) a += dred[k];
        chi2p[ft] = a * g.inv_sigma2;
    }
    // sums of omega = conj(g_i) g_j r / sigma^2 over the groups' members: four lanes a group, each every fourth
    // member, added in a fixed order
    float qm = 0.f;
    for (int u0 = 0; u0 < U; u0 += NT / 4) {
        const int u = u0 + (tid >> 2);
        float qr = 0.f, qi = 0.f;
        if (u < U) {
            const int m1 = moff[u + 1];
#pragma unroll 4
            for (int m = moff[u] + (tid & 3); m < m1; m += 4) {
                const int2 p = __ldg(gmem + m);            // 2 b + reversed, i | j << 16
                const float2 r = sR[p.x >> 1], gi = sG[p.y & 0xffff], gj = sG[p.y >> 16];
                const float ggr = gi.x * gj.x + gi.y * gj.y, ggi = gi.y * gj.x - gi.x * gj.y;
                const float oi = ggr * r.y - ggi * r.x;
                qr += ggr * r.x + ggi * r.y;
                qi += (p.x & 1) ? -oi : oi;
            }
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            qr += __shfl_xor_sync(0xffffffffu, qr, o);
            qi += __shfl_xor_sync(0xffffffffu, qi, o);
        }
        if (u < U && (tid & 3) == 0) {
            qr *= is2;
            qi *= is2;
            *reinterpret_cast<float2 *>(q32 + ((size_t)ft * U + u) * 2) = make_float2(qr, qi);
            qm = fmaxf(qm, fmaxf(fabsf(qr), fabsf(qi)));
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) qm = fmaxf(qm, __shfl_xor_sync(0xffffffffu, qm, o));
    if (lane == 0) fred[w] = qm;
    // chunk c = tid mod nc of Z_a, a = tid div nc: partners j = c, c + nc, ... (j != a) of r g_j conj(V), r and V
    // conjugated for j < a
    const int nc = NT / g.A;
    if (tid < nc * g.A) {
        const int a = tid / nc, rowa = a * g.A - (a * (a + 1)) / 2 - a - 1;
        float zr = 0, zi = 0;
#pragma unroll 4
        for (int j = tid - a * nc; j < g.A; j += nc) {
            if (j == a) continue;
            const int b = j > a ? rowa + j : pair_index(j, a, g.A), code = __ldg(&pairs[b].y);
            const float sgn = j > a ? 1.f : -1.f;
            float2 r = sR[b], V = sV[code >> 1];
            const float2 gj = sG[j];
            r.y *= sgn;
            V.y *= (code & 1) ? -sgn : sgn;
            const float pr = r.x * gj.x - r.y * gj.y, pi = r.x * gj.y + r.y * gj.x;
            zr += pr * V.x + pi * V.y;
            zi += pi * V.x - pr * V.y;
        }
        sZ[tid] = make_float2(zr, zi);
    }
    __syncthreads();
    if (tid == 0) {
        float m = 0.f;
        for (int k = 0; k < NT / 32; ++k) m = fmaxf(m, fred[k]);
        qmax_ft[ft] = m;
    }
    antenna_totals<NT>(sZ, g.A, ft, is2, zpart);
}

// grad_gamma[a][k][c] = sum_{f,t} X_k(nu_f) zpart[f][t][a][c]: one CTA per (a, c); thread
// j takes the (channel, LST) pairs j, j + GR_THREADS, ... in batches of GR_U independent
// loads.  Per thread and across a warp (fixed shuffle order) the sums are in the working
// type; the warps' sums are added in order in FP64 (the FP64 pipe is narrow on this part,
// so it is kept off the per-element path).
constexpr int GR_NGMAX = 8, GR_THREADS = 1024, GR_U = 4;
template <typename R>
__global__ void __launch_bounds__(GR_THREADS) k_gain_reduce_ft(DevGeom g, const R *__restrict__ zpart,
                                                               R *__restrict__ out)
{
    __shared__ double red[GR_THREADS / 32][GR_NGMAX];
    const int a = blockIdx.x >> 1, c = blockIdx.x & 1, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const R *gl = Tab<R>::gleg(g);
    const int nthr = blockDim.x;
    R acc[GR_NGMAX];
#pragma unroll
    for (int k = 0; k < GR_NGMAX; ++k) acc[k] = 0;
    const int nft = g.F * g.T;
    for (int base = 0; base < nft; base += nthr * GR_U) {
        R z[GR_U];
        int f[GR_U];
#pragma unroll
        for (int u = 0; u < GR_U; ++u) {
            const int ft = base + u * nthr + (int)threadIdx.x;
            z[u] = ft < nft ? zpart[((size_t)ft * g.A + a) * 2 + c] : (R)0;
            f[u] = ft < nft ? ft / g.T : 0;
        }
#pragma unroll
        for (int u = 0; u < GR_U; ++u)
#pragma unroll
            for (int k = 0; k < GR_NGMAX; ++k)
                if (k < g.NG) acc[k] += gl[(size_t)f[u] * g.NG + k] * z[u];
    }
#pragma unroll
    for (int k = 0; k < GR_NGMAX; ++k) {
        if (k >= g.NG) break;
        R v = acc[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) red[w][k] = (double)v;
    }
    __syncthreads();
    if (threadIdx.x < g.NG) {
        double t = 0.0;
        for (int k = 0; k < nthr / 32; ++k) t += red[k][threadIdx.x];
        out[(a * g.NG + threadIdx.x) * 2 + c] = (R)t;
    }
}

template <typename R>
fm_status launch_chi2_chan(Ctx &c, const R *vis, const R *gamma, R *omega, R *zpart, double *chi2p, bool groups,
                           cudaStream_t st, const R *rin, const HaVSrc *hv)
{
    if (hv && (!std::is_same<R, float>::value || !groups || rin)) {
        set_error("V from the forward's partial sums: hour-angle form, FP32, no delay filter");
        return FM_ERR_STATE;
    }
    // the limit of k_chi2_ft without V of the groups holds for either kernel: k_chi2_group takes less (V of at most B
    // groups and the residuals), and k_chi2_ft runs with V of the groups only up to 56 KB without it
    const size_t base = (c.A + 3 * (size_t)c.B) * 2 * sizeof(R);
    if (base > 227 * 1024 || c.A > CF_THREADS) {
        set_error("chi^2 epilogue: %d antennas (at most %d, %zu bytes of shared memory)", c.A, CF_THREADS, base);
        return FM_ERR_UNSUPPORTED;
    }
    if constexpr (std::is_same<R, float>::value)
        if (groups && base > 56 * 1024) {              // fewer than four CTAs of k_chi2_ft an SM
            const size_t sm = ((size_t)c.A + c.ha.U + c.B) * sizeof(float2);
            FM_CK(smem_opt_in(k_chi2_group));
            k_chi2_group<<<c.F * c.T, CG_THREADS, sm, st>>>(c.g, vis, (const float *)c.data, gamma, zpart, chi2p, c.ha.U,
                                                            c.fg.pairs, c.fg.gmem, c.ha.moff, c.ha.q32, c.ha.qmax_ft, rin,
                                                            hv ? *hv : HaVSrc{});
            FM_CK_LAUNCH();
            return FM_OK;
        }
    const size_t smem = base + (hv ? sizeof(float) * 128 * (size_t)hv->nmt : 0);
    FM_CK(smem_opt_in(k_chi2_ft<R>));
    k_chi2_ft<R><<<c.F * c.T, CF_THREADS, smem, st>>>(c.g, vis, (const R *)c.data, gamma, omega, zpart, chi2p, c.ha.U, c.ha.moff,
                                                      c.ha.mem, groups ? c.ha.q32 : nullptr, c.ha.qmax_ft, rin,
                                                      hv ? *hv : HaVSrc{});
    FM_CK_LAUNCH();
    return FM_OK;
}

template <typename R>
fm_status launch_gain_reduce_chan(Ctx &c, const R *zpart, R *grad_gain, cudaStream_t st)
{
    if (c.NG > GR_NGMAX) return launch_gain_reduce<R>(c, zpart, grad_gain, st);
    // no more warps than there are terms: their FP64 shuffles alone took 20 us
    const int nthr = std::min(GR_THREADS, (c.F * c.T + 31) / 32 * 32);
    k_gain_reduce_ft<R><<<2 * c.A, nthr, 0, st>>>(c.g, zpart, grad_gain);
    FM_CK_LAUNCH();
    return FM_OK;
}

// Tangent of the epilogue for Hessian-vector products.  With dm = dg_p conj(g_q) V +
// g_p conj(dg_q) V + g_p conj(g_q) dV (JVP), the adjoint weights become
// omega' = [dm conj(g_p) g_q + full * r (conj(dg_p) g_q + conj(g_p) dg_q)] / sigma^2 and
// the gain partials follow the same pattern (full = 0 keeps only the dm terms: GN).
template <typename R>
__global__ void __launch_bounds__(256) k_hvp_mid(DevGeom g, const R *__restrict__ vis, const R *__restrict__ dvis,
                                                 const R *__restrict__ data, const R *__restrict__ gains,
                                                 const R *__restrict__ dgains, int full, R *__restrict__ omega,
                                                 R *__restrict__ zpart)
{
    using C2 = typename V2<R>::t;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C2 *sG = reinterpret_cast<C2 *>(smem_raw);
    C2 *sD = sG + g.A;
    C2 *sV = sD + g.A;
    C2 *sdV = sV + g.B;
    C2 *sRr = sdV + g.B;
    C2 *sdM = sRr + g.B;
    const int ft = blockIdx.x, f = ft / g.T;
    for (int i = threadIdx.x; i < g.A; i += blockDim.x) {
        sG[i].x = gains[2 * (f * g.A + i)];
        sG[i].y = gains[2 * (f * g.A + i) + 1];
        sD[i].x = dgains[2 * (f * g.A + i)];
        sD[i].y = dgains[2 * (f * g.A + i) + 1];
    }
    __syncthreads();
    const R is2 = (R)g.inv_sigma2;
    auto mul = [](C2 a, C2 b) { C2 r; r.x = a.x * b.x - a.y * b.y; r.y = a.x * b.y + a.y * b.x; return r; };
    auto cj = [](C2 a) { a.y = -a.y; return a; };
    auto add = [](C2 a, C2 b) { a.x += b.x; a.y += b.y; return a; };
    for (int b = threadIdx.x; b < g.B; b += blockDim.x) {
        int i = g.bl_i[b], j = g.bl_j[b];
        size_t o = ((size_t)ft * g.B + b) * 2;
        C2 V, dV, gi = sG[i], gj = sG[j], di = sD[i], dj = sD[j];
        V.x = vis[o]; V.y = vis[o + 1];
        dV.x = dvis[o]; dV.y = dvis[o + 1];
        C2 gg = mul(gi, cj(gj));
        C2 r = mul(gg, V);
        r.x -= data[o]; r.y -= data[o + 1];
        C2 dm = add(add(mul(mul(di, cj(gj)), V), mul(mul(gi, cj(dj)), V)), mul(gg, dV));
        C2 w = mul(dm, cj(gg));
        if (full) w = add(w, mul(r, add(mul(cj(di), gj), mul(cj(gi), dj))));
        omega[o] = w.x * is2;
        omega[o + 1] = w.y * is2;
        sV[b] = V; sdV[b] = dV; sRr[b] = r; sdM[b] = dm;
    }
    __syncthreads();
    for (int a = threadIdx.x; a < g.A; a += blockDim.x) {
        C2 z;
        z.x = z.y = R(0);
        for (int j = 0; j < g.A; ++j) {
            if (j == a) continue;
            if (j > a) {       // pair (a, j): c = conj(dm) conj(g_j) V + full conj(r)(conj(dg_j) V + conj(g_j) dV)
                int b = pair_index(a, j, g.A);
                C2 c = mul(mul(cj(sdM[b]), cj(sG[j])), sV[b]);
                if (full) c = add(c, mul(cj(sRr[b]), add(mul(cj(sD[j]), sV[b]), mul(cj(sG[j]), sdV[b]))));
                z = add(z, cj(c));
            } else {           // pair (j, a): c = conj(dm) g_j V + full conj(r)(dg_j V + g_j dV)
                int b = pair_index(j, a, g.A);
                C2 c = mul(mul(cj(sdM[b]), sG[j]), sV[b]);
                if (full) c = add(c, mul(cj(sRr[b]), add(mul(sD[j], sV[b]), mul(sG[j], sdV[b]))));
                z = add(z, c);
            }
        }
        zpart[((size_t)ft * g.A + a) * 2] = z.x * is2;
        zpart[((size_t)ft * g.A + a) * 2 + 1] = z.y * is2;
    }
}

// The same in one pass for the hour-angle form after its two-sky forward: V and dV are formed from the
// partial sums (hv, hd), the gains and their tangents from the coefficients, the omega' sums over the
// baseline groups go to q32 / qmax_ft, and the gain partials are k_chi2_ft's (a warp's or chunk's terms in
// order).  37 antennas, 64 channels, 60 LSTs: the separate finishing of V and dV, the gains, k_hvp_mid and
// the group sums took 91 us.  Bound: the latency of a CTA's chain of phases, as k_chi2_ft.
template <bool FULL>
__global__ void __launch_bounds__(CF_THREADS, 6) k_hvp_ft(DevGeom g, const float *__restrict__ data,
                                                          const float *__restrict__ gamma,
                                                          const float *__restrict__ dgamma, float *__restrict__ zpart,
                                                          int U, const int *__restrict__ moff,
                                                          const int *__restrict__ mem, float *__restrict__ q32,
                                                          float *__restrict__ qmax_ft, HaVSrc hv, HaVSrc hd)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *sG = reinterpret_cast<float2 *>(smem_raw), *sD = sG + g.A;       // [A] gains and tangents
    float2 *sTi = sD + g.A, *sTj = sTi + g.B, *sW = sTj + g.B;               // [B]
    float2 *sV = sW + g.B, *sdV = sV + 64 * hv.nmt;                          // [U] V and dV of the groups
    __shared__ float2 sZ[CF_THREADS];
    __shared__ float fred[CF_THREADS / 32];
    const int ft = blockIdx.x, f = ft / g.T, tid = threadIdx.x, lane = tid & 31;
    const float *X = g.gleg32 + (size_t)f * g.NG;
    for (int i = tid; i < 2 * g.A; i += CF_THREADS) {                        // as k_gains
        const float *c = (i < g.A ? gamma : dgamma) + 2 * (size_t)(i < g.A ? i : i - g.A) * g.NG;
        float re = 0, im = 0;
        for (int k = 0; k < g.NG; ++k) {
            re += X[k] * c[2 * k];
            im += X[k] * c[2 * k + 1];
        }
        sG[i] = make_float2(re, im);
    }
    group_vis<CF_THREADS>(hv, f, ft - f * g.T, ft, U, sV);
    group_vis<CF_THREADS>(hd, f, ft - f * g.T, ft, U, sdV);
    __syncthreads();
    const float is2 = (float)g.inv_sigma2;
    auto mul = [](float2 a, float2 b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); };
    auto mulc = [](float2 a, float2 b) { return make_float2(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y); };   // a conj(b)
    auto add = [](float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); };
    const float2 *drow = reinterpret_cast<const float2 *>(data) + (size_t)ft * g.B;
    for (int b = tid; b < g.B; b += CF_THREADS) {
        const int2 pr = __ldg(hv.pairs + b);
        const int i = pr.x & 0xffff, j = pr.x >> 16;
        const float2 gi = sG[i], gj = sG[j], di = sD[i], dj = sD[j];
        const float2 V = member_vis(sV, pr.y), dV = member_vis(sdV, pr.y);
        const float2 gg = mulc(gi, gj);
        const float2 dm = add(mul(add(mulc(di, gj), mulc(gi, dj)), V), mul(gg, dV));
        float2 om = mulc(dm, gg);
        float2 ti = mulc(mul(dm, gj), V);                  // dm g_j conj(V), the term in Z_i
        float2 tj = mulc(mul(gi, V), dm);                  // conj(dm) g_i V, the term in Z_j
        if (FULL) {
            const float2 d = drow[b];
            float2 r = mul(gg, V);
            r.x -= d.x;
            r.y -= d.y;
            om = add(om, mul(r, add(mulc(gj, di), mulc(dj, gi))));
            ti = add(ti, mul(r, add(mulc(dj, V), mulc(gj, dV))));
            tj = add(tj, mulc(add(mul(di, V), mul(gi, dV)), r));
        }
        sTi[b] = ti;
        sTj[b] = tj;
        sW[b] = make_float2(om.x * is2, om.y * is2);
    }
    __syncthreads();
    float qm = group_sums<CF_THREADS>(sW, ft, U, moff, mem, q32);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) qm = fmaxf(qm, __shfl_xor_sync(0xffffffffu, qm, o));
    if (lane == 0) fred[tid >> 5] = qm;
    antenna_chunks<CF_THREADS>(sTi, sTj, g.A, sZ);
    __syncthreads();
    if (tid == 0) {
        float m = 0.f;
        for (int k = 0; k < CF_THREADS / 32; ++k) m = fmaxf(m, fred[k]);
        qmax_ft[ft] = m;
    }
    antenna_totals<CF_THREADS>(sZ, g.A, ft, is2, zpart);
}

bool launch_hvp_ft_fits(const Ctx &c)
{
    return c.A <= CF_THREADS && (2 * c.A + 3 * (size_t)c.B) * 8 + 1024 * (size_t)c.ha.nmt <= 200 * 1024;
}

fm_status launch_hvp_ft(Ctx &c, const float *gamma, const float *dgamma, int full, float *zpart, const HaVSrc &hv,
                        const HaVSrc &hd, cudaStream_t st)
{
    const size_t smem = (2 * c.A + 3 * (size_t)c.B) * 8 + 1024 * (size_t)c.ha.nmt;
    auto *kern = full ? k_hvp_ft<true> : k_hvp_ft<false>;
    FM_CK(smem_opt_in(kern));
    kern<<<c.F * c.T, CF_THREADS, smem, st>>>(c.g, (const float *)c.data, gamma, dgamma, zpart, c.ha.U, c.ha.moff, c.ha.mem,
                                              c.ha.q32, c.ha.qmax_ft, hv, hd);
    FM_CK_LAUNCH();
    return FM_OK;
}

template <typename R>
fm_status launch_hvp_mid(Ctx &c, const R *vis, const R *dvis, const R *g, const R *dg, int full, R *omega, R *zpart,
                         cudaStream_t st)
{
    size_t smem = (2 * (size_t)c.A + 4 * (size_t)c.B) * 2 * sizeof(R);
    if (smem > 227 * 1024) return FM_ERR_UNSUPPORTED;
    FM_CK(smem_opt_in(k_hvp_mid<R>));
    k_hvp_mid<R><<<c.F * c.T, 256, smem, st>>>(c.g, vis, dvis, (const R *)c.data, g, dg, full, omega, zpart);
    FM_CK_LAUNCH();
    return FM_OK;
}

// ---------------------------------------------------------------- adjoint contraction
// One CTA per (channel, tile of PT pixels), looping over LSTs so xbar accumulates in
// registers without atomics.  For each LST the tile's phasors go to shared memory and
// each thread forms, for its pixel, sum_p Re[E_p conj(Y_p)] with
// Y_p = sum_{q>p} omega_pq E_q  (= sum_{p<q} Re[conj(omega_pq) E_p conj(E_q)]).
template <typename R>
__global__ void __launch_bounds__(128) k_adj_simt(DevGeom g, const R *__restrict__ omega, R *__restrict__ xbar)
{
    using C2 = typename V2<R>::t;
    constexpr int PT = 128;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C2 *sE = reinterpret_cast<C2 *>(smem_raw);        // [A][PT]
    C2 *sC = sE + (size_t)g.A * PT;                   // [B]
    const int f = blockIdx.y, p0 = blockIdx.x * PT, tid = threadIdx.x;
    const int p = p0 + tid;
    R accx = R(0);
    for (int t = 0; t < g.T; ++t) {
        __syncthreads();
        for (int e = tid; e < g.A * PT; e += blockDim.x) {
            int i = e / PT, pl = e % PT, pp = p0 + pl;
            C2 ev;
            ev.x = ev.y = R(0);
            if (pp < g.npix) Phasor<R>::eval(g, f, i, t, pp, ev.x, ev.y);
            sE[e] = ev;
        }
        const R *om = omega + ((size_t)(f * g.T + t) * g.B) * 2;
        for (int b = tid; b < g.B; b += blockDim.x) {
            sC[b].x = om[2 * b];
            sC[b].y = om[2 * b + 1];
        }
        __syncthreads();
        if (p < g.npix) {
            R w = pixel_weight<R>(g, f, t, p);
            if (w != R(0)) {
                R acc = R(0);
                for (int i = 0; i + 1 < g.A; ++i) {
                    R yr = 0, yi = 0;
                    int b0 = pair_index(i, i + 1, g.A) - (i + 1);
                    for (int j = i + 1; j < g.A; ++j) {
                        C2 cc = sC[b0 + j], ej = sE[(size_t)j * PT + tid];
                        yr += cc.x * ej.x - cc.y * ej.y;
                        yi += cc.x * ej.y + cc.y * ej.x;
                    }
                    C2 ei = sE[(size_t)i * PT + tid];
                    acc += ei.x * yr + ei.y * yi;
                }
                accx += w * acc;
            }
        }
    }
    if (p < g.npix) xbar[(size_t)f * g.npix + p] = accx;
}

template <typename R>
fm_status launch_adjoint(Ctx &c, const R *omega, R *xbar, cudaStream_t st)
{
    FM_TRY(simt_supports<R>(c, true));
    const size_t smem = adj_simt_smem<R>(c);
    FM_CK(smem_opt_in(k_adj_simt<R>));
    dim3 grid(cdiv(c.npix, 128), c.F);
    k_adj_simt<R><<<grid, 128, smem, st>>>(c.g, omega, xbar);
    FM_CK_LAUNCH();
    return FM_OK;
}

// ---------------------------------------------------------------- reductions
// grad_gamma[a][k][c] = sum_f X_k(nu_f) sum_t Z[f][t][a][c]   (FP64, fixed order).  CTA (a, c): 16 lanes a channel sum
// its LSTs, lane k multiplies by X_k, warp k adds the channels.  Bound: the FP64 pipe (2 lanes per SM and clock),
// where summing over the LSTs first leaves a conversion and an addition a term, and the products a channel; and the
// latency of the loads, four in flight a thread.  Product of 37 antennas, 64 channels, 60 LSTs: 214.3 (256 threads an
// antenna and coefficient, a product a term) -> 207.2 us.
constexpr int GN_MAX = 16, GN_FC = 64;     // most gain coefficients (fm_create's limit); channels at a time
template <typename R>
__global__ void __launch_bounds__(GN_MAX * GN_FC) k_gain_reduce(DevGeom g, const R *__restrict__ zpart, R *__restrict__ out)
{
    __shared__ double red[GN_MAX][GN_FC + 1];
    const int a = blockIdx.x, c = blockIdx.y, tid = threadIdx.x, q = tid % GN_MAX, fl = tid / GN_MAX;
    double acc = 0.0;                      // warp k < NG: the channels fl = lane, lane + 32 of coefficient k
    for (int f0 = 0; f0 < g.F; f0 += GN_FC) {
        const int f = f0 + fl;
        double s = 0.0;
        if (f < g.F) {
            const R *z = zpart + ((size_t)f * g.T * g.A + a) * 2 + c;
            for (int t0 = q; t0 < g.T; t0 += 4 * GN_MAX) {
                R v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = t0 + u * GN_MAX < g.T ? z[(size_t)(t0 + u * GN_MAX) * g.A * 2] : R(0);
                s += ((double)v[0] + (double)v[1]) + ((double)v[2] + (double)v[3]);
            }
        }
#pragma unroll
        for (int o = GN_MAX / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (f0) __syncthreads();           // the last channels are read
        if (q < g.NG) red[q][fl] = f < g.F ? (double)Tab<R>::gleg(g)[(size_t)f * g.NG + q] * s : 0.0;
        __syncthreads();
        if (tid / 32 < g.NG) acc += red[tid / 32][tid % 32] + red[tid / 32][tid % 32 + 32];
    }
    if (tid / 32 < g.NG) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (tid % 32 == 0) out[(a * g.NG + tid / 32) * 2 + c] = (R)acc;
    }
}

template <typename R>
fm_status launch_gain_reduce(Ctx &c, const R *zpart, R *grad_gain, cudaStream_t st)
{
    k_gain_reduce<R><<<dim3(c.A, 2), GN_MAX * GN_FC, 0, st>>>(c.g, zpart, grad_gain);
    FM_CK_LAUNCH();
    return FM_OK;
}

// fixed-order sum over a CTA of 256 threads: lane shuffles in T, then the 8 warps' sums in
// order in FP64; the result is valid in thread 0
template <typename T>
__device__ __forceinline__ double cta256_sum(T v, double *wred)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) wred[threadIdx.x >> 5] = (double)v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int k = 0; k < 8; ++k) t += wred[k];
    __syncthreads();
    return t;
}

template <typename R>
struct __align__(16) Pack16 { R v[16 / sizeof(R)]; };

// grad += lam (theta - mu) and the prior energy sum lam (theta - mu)^2 / 2 (a warp's terms
// summed in the working type, the warps' sums in FP64), then chi^2 = sum of the per-(f,t)
// partials (FP64, loads batched so that their latencies overlap) and U = chi^2 / 2 + prior.
// Each CTA writes its partial; the CTA that takes the last ticket adds the partials in
// index order (so the result does not depend on which CTA that is) and resets the ticket
// for the next launch.  With p != NULL the pass also applies the leapfrog momentum kick
// p -= frac eps grad with the finished gradient (eps = prm[0], read on the device).  vec: the
// arrays are 16-byte aligned.
constexpr int PT_THREADS = 256;
template <typename R>
__global__ void __launch_bounds__(PT_THREADS) k_prior_total(long long n, int vec, const R *__restrict__ theta,
                                                            const R *__restrict__ mu, const R *__restrict__ lam,
                                                            R *__restrict__ grad, double *part, int nft,
                                                            const double *__restrict__ chi2p, double *chi2_out,
                                                            double *u_out, int *status, unsigned *ticket,
                                                            R *__restrict__ p, const double *__restrict__ prm,
                                                            double frac)
{
    constexpr int W = 16 / sizeof(R);
    __shared__ double wred[8];
    __shared__ int last;
    const long long gtid = blockIdx.x * (long long)blockDim.x + threadIdx.x, gstride = (long long)gridDim.x * blockDim.x;
    R acc = 0;
    if (lam || p) {
        const R ak = p ? (R)(-frac * prm[0]) : (R)0;      // the kick's factor, as in a separate kick
        long long head = 0;
        if (vec) {
            const long long np = n / W;
            head = np * W;
            const Pack16<R> *th = reinterpret_cast<const Pack16<R> *>(theta);
            const Pack16<R> *mp = reinterpret_cast<const Pack16<R> *>(mu);
            const Pack16<R> *lp = reinterpret_cast<const Pack16<R> *>(lam);
            Pack16<R> *gp = reinterpret_cast<Pack16<R> *>(grad);
            Pack16<R> *pp = reinterpret_cast<Pack16<R> *>(p);
            // two packs a thread at a time (k and k + gstride), all their loads issued first;
            // the terms still go into acc in the order of k
            for (long long k0 = gtid; k0 < np; k0 += 2 * gstride) {
                const long long kk[2] = {k0, k0 + gstride};
                const bool has1 = kk[1] < np;
                Pack16<R> gr[2], t[2], m[2], l[2], pv[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    if (u == 1 && !has1) break;
                    gr[u] = gp[kk[u]];
                    if (lam) {
                        t[u] = th[kk[u]];
                        m[u] = mp[kk[u]];
                        l[u] = lp[kk[u]];
                    }
                    if (p) pv[u] = pp[kk[u]];
                }
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    if (u == 1 && !has1) break;
                    if (lam) {
#pragma unroll
                        for (int e = 0; e < W; ++e) {
                            const R dv = t[u].v[e] - m[u].v[e], ld = l[u].v[e] * dv;
                            gr[u].v[e] += ld;
                            acc += ld * dv;
                        }
                        gp[kk[u]] = gr[u];
                    }
                    if (p) {
#pragma unroll
                        for (int e = 0; e < W; ++e) pv[u].v[e] += ak * gr[u].v[e];
                        pp[kk[u]] = pv[u];
                    }
                }
            }
        }
        for (long long k = head + gtid; k < n; k += gstride) {
            R gk = grad[k];
            if (lam) {
                const R l = lam[k], dv = theta[k] - mu[k], ld = l * dv;
                gk += ld;
                grad[k] = gk;
                acc += ld * dv;
            }
            if (p) p[k] += ak * gk;
        }
    }
    const double blk = cta256_sum<R>((R)0.5 * acc, wred);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = blk;
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double a = 0.0, b = 0.0;
    for (int i0 = 0; i0 < nft; i0 += 8 * PT_THREADS) {
        double v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int i = i0 + u * PT_THREADS + (int)threadIdx.x;
            v[u] = i < nft ? __ldcg(chi2p + i) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) a += v[u];
    }
    for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) b += __ldcg(part + i);
    const double ta = cta256_sum<double>(a, wred), tb = cta256_sum<double>(b, wred);
    if (threadIdx.x == 0) {
        if (chi2_out) *chi2_out = ta;
        if (u_out) *u_out = 0.5 * ta + tb;
        if (!isfinite(ta) || !isfinite(tb)) atomicExch(status, (int)FM_ERR_NONFINITE);
        *ticket = 0u;
    }
}

template <typename R>
fm_status launch_prior_and_total(Ctx &c, const R *theta, R *grad, const double *chi2p, int nchi2, double *chi2_out,
                                 double *u_out, cudaStream_t st, R *kick_p, const double *kick_prm, double kick_frac)
{
    const R *mu = (const R *)c.mu, *lam = c.have_prior ? (const R *)c.lam : nullptr;
    auto al = [](const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; };
    const int vec = al(theta) && al(mu) && al(c.lam) && al(grad) && al(kick_p);
    const long long units = vec ? c.n_par / (16 / (long long)sizeof(R)) : c.n_par;
    const int nblk = (int)std::max(1LL, std::min<long long>(4 * 152, (long long)cdiv(units, PT_THREADS)));
    k_prior_total<R><<<nblk, PT_THREADS, 0, st>>>(c.n_par, vec, theta, mu, lam, grad, c.red, nchi2, chi2p, chi2_out,
                                                 u_out, c.status, c.ticket, kick_p, kick_prm, kick_frac);
    FM_CK_LAUNCH();
    return FM_OK;
}

template <typename R>
__global__ void k_prior_hvp(long long n, const R *__restrict__ v, const R *__restrict__ lam, R *__restrict__ hv)
{
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x)
        hv[k] += lam[k] * v[k];
}

template <typename R>
fm_status launch_prior_hvp(Ctx &c, const R *v, R *hv, cudaStream_t st)
{
    if (!c.have_prior) return FM_OK;
    k_prior_hvp<R><<<296, 256, 0, st>>>(c.n_par, v, (const R *)c.lam, hv);
    FM_CK_LAUNCH();
    return FM_OK;
}

// ---------------------------------------------------------------- monopole split
// vis[f][t][b] += c_f U[f][t][b] with c_f = src[f * stride]: puts back the visibility of
// the uniform part of the sky that the contraction kernels did not see.
template <typename R>
__global__ void k_add_dc(DevGeom g, const R *__restrict__ src, long long stride, const float *__restrict__ U,
                         R *__restrict__ vis)
{
    long long n = (long long)g.F * g.T * g.B;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        int f = (int)(e / ((long long)g.T * g.B));
        R cf = src[(long long)f * stride];
        vis[2 * e] += cf * (R)U[2 * e];
        vis[2 * e + 1] += cf * (R)U[2 * e + 1];
    }
}

template <typename R>
fm_status launch_add_dc(Ctx &c, const R *src, long long stride, R *vis, cudaStream_t st)
{
    k_add_dc<R><<<1024, 256, 0, st>>>(c.g, src, stride, c.dc_u, vis);
    FM_CK_LAUNCH();
    return FM_OK;
}

// per-channel mean of x (fixed-order tree) and x' = x - mean
template <typename R>
__global__ void __launch_bounds__(256) k_center(int npix, const R *__restrict__ x, R *__restrict__ xc,
                                                R *__restrict__ mean)
{
    __shared__ double red[256];
    const int f = blockIdx.x;
    double s = 0.0;
    for (int p = threadIdx.x; p < npix; p += blockDim.x) s += (double)x[(size_t)f * npix + p];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    const R m = (R)(red[0] / npix);
    if (threadIdx.x == 0) mean[f] = m;
    for (int p = threadIdx.x; p < npix; p += blockDim.x) xc[(size_t)f * npix + p] = x[(size_t)f * npix + p] - m;
}

template <typename R>
fm_status launch_center(Ctx &c, const R *x, R *xc, R *mean, cudaStream_t st)
{
    k_center<R><<<c.F, 256, 0, st>>>(c.npix, x, xc, mean);
    FM_CK_LAUNCH();
    return FM_OK;
}

__global__ void k_d2f(long long n, const double *__restrict__ a, float *__restrict__ b)
{
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
        b[e] = (float)a[e];
}

fm_status launch_d2f(long long n, const double *a, float *b, cudaStream_t st)
{
    k_d2f<<<1024, 256, 0, st>>>(n, a, b);
    FM_CK_LAUNCH();
    return FM_OK;
}

#define FM_INST(R)                                                                                       \
    template fm_status launch_chi2_chan<R>(Ctx &, const R *, const R *, R *, R *, double *, bool, cudaStream_t, const R *, \
                                           const HaVSrc *);                                              \
    template fm_status launch_gain_reduce_chan<R>(Ctx &, const R *, R *, cudaStream_t);                 \
    template fm_status launch_modes_forward<R>(Ctx &, const R *, R *, cudaStream_t, int, unsigned *,        \
                                               const StripArgs *);                                           \
    template fm_status launch_modes_adjoint<R>(Ctx &, const R *, R *, cudaStream_t);                     \
    template fm_status launch_gains<R>(Ctx &, const R *, R *, cudaStream_t);                             \
    template fm_status launch_vis<R>(Ctx &, const R *, R *, cudaStream_t);                               \
    template fm_status launch_adjoint<R>(Ctx &, const R *, R *, cudaStream_t);                           \
    template fm_status launch_apply_gains<R>(Ctx &, const R *, const R *, R *, cudaStream_t);            \
    template fm_status launch_hvp_mid<R>(Ctx &, const R *, const R *, const R *, const R *, int, R *, R *, \
                                         cudaStream_t);                                                  \
    template fm_status launch_gain_reduce<R>(Ctx &, const R *, R *, cudaStream_t);                       \
    template fm_status launch_prior_and_total<R>(Ctx &, const R *, R *, const double *, int, double *, double *, \
                                                 cudaStream_t, R *, const double *, double);             \
    template fm_status launch_prior_hvp<R>(Ctx &, const R *, R *, cudaStream_t);                         \
    template fm_status launch_add_dc<R>(Ctx &, const R *, long long, R *, cudaStream_t);                \
    template fm_status launch_center<R>(Ctx &, const R *, R *, R *, cudaStream_t);
FM_INST(float)
FM_INST(double)

}  // namespace fm
