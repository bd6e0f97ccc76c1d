// Contraction on grids that are no drift scan of whole hour-angle cells: every distinct fringe
// (FringeGroups) summed once on the CUDA cores, with the phasors of the covering antenna subset
// formed in the kernels.
//
//   V_u(t) = sum_p w_p x_p E_i conj(E_j),  w = dOmega A,   xbar_p = sum_t w_p sum_u Re[conj(Q_u) E_i conj(E_j)]
//
// for the representative pair (i, j) of group u.  The pairs are sorted by i, so that w x E_i
// (forward) and Y_i = sum_j Q E_j (adjoint) stay in registers over a run and a (group, pixel) costs one
// shared-memory read and two packed complex multiply-adds.  Bound: instruction issue, split between the
// phasors (two-float phase and sincospif, about 45 instructions each) and those products.
//
// chi^2 + gradient against the per-baseline sums of k_simt.cu: 37 antennas, 64 channels, 12 LSTs, 128 x 160
// pixels in FP32 14.44 -> 2.42 ms; 7 antennas, 16 channels, 19 LSTs, 32 x 96 pixels in FP64 7.06 -> 1.54 ms.
//
// FP64 and FP32 handles whose groups are few enough that the phasors are formed at most four times
// (GD_MAX_U); larger arrays without redundancy run the tiled per-baseline sum of k_simt.cu.
#include <algorithm>
#include <cstdlib>
#include <type_traits>
#include <vector>

#include "fm_internal.cuh"
#include "phasor.cuh"

namespace fm {
namespace {

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ double2 fma2(double2 a, double2 b, double2 c)
{
    return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y));
}
__device__ __forceinline__ float2 mk2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ double2 mk2(double a, double b) { return make_double2(a, b); }

constexpr int GD_PC = 64;              // forward: pixels staged at a time, two a lane
constexpr int GD_NGW = 8;              // groups of a forward warp
constexpr int GD_TU = 8 * GD_NGW;      // groups of a forward CTA (8 warps)
constexpr int GD_AT = 128;             // adjoint threads
constexpr int GD_MAX_U = 256;          // groups (four forward tiles)

struct GdDev {
    int U, nant, ntile, nsplit;
    const int4 *ord;                   // [U] (i, j, u, 0) sorted by (i, j)
    const int *ant;                    // [nant] subset entry -> antenna
};

// phase slopes of one channel's subset antennas, in shared memory
template <typename R> struct Slopes;
template <> struct Slopes<float> {
    float4 a;                          // east hi, lo, north hi, lo
    float2 b;                          // up hi, lo
    float2 pad;
    __device__ __forceinline__ void load(const DevGeom &g, int f, int i)
    {
        const float *k = g.kap32 + ((size_t)f * g.A + i) * 6;
        a = make_float4(k[0], k[1], k[2], k[3]);
        b = make_float2(k[4], k[5]);
    }
};
template <> struct Slopes<double> {
    double k[4];
    __device__ __forceinline__ void load(const DevGeom &g, int f, int i)
    {
        const double *s = g.kap64 + ((size_t)f * g.A + i) * 3;
        k[0] = s[0]; k[1] = s[1]; k[2] = s[2];
    }
};

// direction of one pixel at one LST, in registers
template <typename R> struct Dir;
template <> struct Dir<float> {
    float s[6];
    __device__ __forceinline__ void load(const DevGeom &g, int t, int p)
    {
        const float2 *q = reinterpret_cast<const float2 *>(g.s32) + ((size_t)t * g.npix + p) * 3;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float2 v = __ldg(q + c);
            s[2 * c] = v.x;
            s[2 * c + 1] = v.y;
        }
    }
    // the arithmetic of phase_frac_2f; a flat array's up terms are exact zeros and left out
    __device__ __forceinline__ float2 phasor(const Slopes<float> &k, int flat) const
    {
        const float kk[6] = {k.a.x, k.a.y, k.a.z, k.a.w, k.b.x, k.b.y};
        float accf = 0.f, acce = 0.f;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (c == 2 && flat) break;
            const float p = __fmul_rn(kk[2 * c], s[2 * c]);
            const float e = __fmaf_rn(kk[2 * c], s[2 * c], -p);
            accf = __fadd_rn(accf, __fsub_rn(p, rintf(p)));
            acce = __fadd_rn(acce, __fadd_rn(e, __fmaf_rn(kk[2 * c], s[2 * c + 1], __fmul_rn(kk[2 * c + 1], s[2 * c]))));
        }
        float t = __fadd_rn(accf, acce);
        t = __fsub_rn(t, rintf(t));
        float sn, cs;
        sincospif(2.0f * t, &sn, &cs);
        return make_float2(cs, -sn);
    }
};
template <> struct Dir<double> {
    double s[3];
    __device__ __forceinline__ void load(const DevGeom &g, int t, int p)
    {
        const double *q = g.s64 + ((size_t)t * g.npix + p) * 3;
        s[0] = q[0]; s[1] = q[1]; s[2] = q[2];
    }
    __device__ __forceinline__ double2 phasor(const Slopes<double> &k, int) const
    {
        double ph = k.k[0] * s[0] + k.k[1] * s[1] + k.k[2] * s[2];
        ph -= rint(ph);
        double sn, cs;
        sincospi(2.0 * ph, &sn, &cs);
        return make_double2(cs, -sn);
    }
};

// the two pixels of a lane: neighbours in FP32 (one 16-byte read), 32 apart in FP64
template <typename R> __device__ __forceinline__ int lane_pix(int lane, int q)
{
    return std::is_same<R, float>::value ? 2 * lane + q : lane + 32 * q;
}
__device__ __forceinline__ void load_pair(const float2 *row, int lane, float2 (&v)[2])
{
    const float4 q = *reinterpret_cast<const float4 *>(row + 2 * lane);
    v[0] = make_float2(q.x, q.y);
    v[1] = make_float2(q.z, q.w);
}
__device__ __forceinline__ void load_pair(const double2 *row, int lane, double2 (&v)[2])
{
    v[0] = row[lane];
    v[1] = row[lane + 32];
}

// CTA = (channel, LST, tile of 64 groups, split of the pixels).  64 pixels at a time the phasors of the
// subset go to shared memory (thread = one pixel of 64, every fourth antenna); warp w then adds its 8
// groups' products over them, two pixels a lane; the lanes' sums are added at the end.  Per group
// s1 = sum a.x b, s2 = sum a.y b with a = w x E_i, b = E_j: V = (s1.x + s2.y, s2.x - s1.y).
template <typename R>
__global__ void __launch_bounds__(256) k_gd_fwd(DevGeom g, GdDev h, const R *__restrict__ x,
                                                typename V2<R>::t *__restrict__ part)
{
    using C2 = typename V2<R>::t;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C2 *sE = reinterpret_cast<C2 *>(smem_raw);                         // [nant][GD_PC]
    Slopes<R> *sK = reinterpret_cast<Slopes<R> *>(sE + (size_t)h.nant * GD_PC);   // [nant]
    R *sW = reinterpret_cast<R *>(sK + h.nant);                        // [GD_PC]
    int b = blockIdx.x;
    const int sp = b % h.nsplit;
    b /= h.nsplit;
    const int tile = b % h.ntile, ft = b / h.ntile, f = ft / g.T, t = ft % g.T;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int a = tid; a < h.nant; a += 256) sK[a].load(g, f, h.ant[a]);
    const int n0 = tile * GD_TU + warp * GD_NGW;
    int oi[GD_NGW], oj[GD_NGW];        // rows of the groups' pairs; past the end the first row, not stored
#pragma unroll
    for (int n = 0; n < GD_NGW; ++n) {
        const int4 o = n0 + n < h.U ? __ldg(h.ord + n0 + n) : make_int4(0, 0, 0, 0);
        oi[n] = o.x * GD_PC;
        oj[n] = o.y * GD_PC;
    }
    C2 s1[GD_NGW], s2[GD_NGW];
#pragma unroll
    for (int n = 0; n < GD_NGW; ++n) s1[n] = s2[n] = mk2(R(0), R(0));
    const int nch = (g.npix + GD_PC - 1) / GD_PC;
    const int c0 = (int)((long long)nch * sp / h.nsplit), c1 = (int)((long long)nch * (sp + 1) / h.nsplit);
    const R *xf = x + (size_t)f * g.npix;
    for (int c = c0; c < c1; ++c) {
        __syncthreads();
        {
            const int pl = tid & (GD_PC - 1), p = c * GD_PC + pl;
            const bool in = p < g.npix;
            Dir<R> dir;
            if (in) dir.load(g, t, p);
            for (int a = tid / GD_PC; a < h.nant; a += 256 / GD_PC)
                sE[a * GD_PC + pl] = in ? dir.phasor(sK[a], g.flat_array) : mk2(R(0), R(0));
            if (tid < GD_PC) sW[pl] = in ? pixel_weight<R>(g, f, t, p) * xf[p] : R(0);
        }
        __syncthreads();
        if (n0 < h.U) {
            const R w0 = sW[lane_pix<R>(lane, 0)], w1 = sW[lane_pix<R>(lane, 1)];
            int cur = -1;
            C2 ax[2], ay[2];
            ax[0] = ax[1] = ay[0] = ay[1] = mk2(R(0), R(0));
#pragma unroll
            for (int n = 0; n < GD_NGW; ++n) {
                if (oi[n] != cur) {    // the same for the whole warp
                    cur = oi[n];
                    C2 e[2];
                    load_pair(sE + cur, lane, e);
                    ax[0] = mk2(w0 * e[0].x, w0 * e[0].x);
                    ay[0] = mk2(w0 * e[0].y, w0 * e[0].y);
                    ax[1] = mk2(w1 * e[1].x, w1 * e[1].x);
                    ay[1] = mk2(w1 * e[1].y, w1 * e[1].y);
                }
                C2 v[2];
                load_pair(sE + oj[n], lane, v);
                s1[n] = fma2(ax[1], v[1], fma2(ax[0], v[0], s1[n]));
                s2[n] = fma2(ay[1], v[1], fma2(ay[0], v[0], s2[n]));
            }
        }
    }
#pragma unroll
    for (int n = 0; n < GD_NGW; ++n) {
        R re = s1[n].x + s2[n].y, im = s2[n].x - s1[n].y;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            re += __shfl_xor_sync(0xffffffffu, re, o);
            im += __shfl_xor_sync(0xffffffffu, im, o);
        }
        if (lane == 0 && n0 + n < h.U)
            part[((size_t)sp * g.F * g.T + ft) * h.U + __ldg(h.ord + n0 + n).z] = mk2(re, im);
    }
}

// CTA = (channel, tile of 256 (FP64: 128) pixels), one or two pixels a thread, over all LSTs: the
// thread's phasors in its own columns of shared memory, Q of the LST in the sorted order, and per run
// of equal i: Y = sum_j Q E_j from A = sum Q.x E_j, B = sum Q.y E_j: Y = (A.x - B.y, A.y + B.x).
template <typename R>
__global__ void __launch_bounds__(GD_AT) k_gd_adj(DevGeom g, GdDev h, const typename V2<R>::t *__restrict__ Q,
                                                  R *__restrict__ xbar)
{
    using C2 = typename V2<R>::t;
    constexpr int PP = std::is_same<R, float>::value ? 2 : 1, PT = PP * GD_AT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C2 *sE = reinterpret_cast<C2 *>(smem_raw);                         // [nant][PT]
    Slopes<R> *sK = reinterpret_cast<Slopes<R> *>(sE + (size_t)h.nant * PT);
    C2 *sQ = reinterpret_cast<C2 *>(sK + h.nant);                      // [U], sorted order
    int2 *sO = reinterpret_cast<int2 *>(sQ + h.U);                     // [U] rows of the pair
    const int f = blockIdx.y, tid = threadIdx.x, p0 = blockIdx.x * PT + PP * tid;
    for (int a = tid; a < h.nant; a += GD_AT) sK[a].load(g, f, h.ant[a]);
    for (int n = tid; n < h.U; n += GD_AT) {
        const int4 o = __ldg(h.ord + n);
        sO[n] = make_int2(o.x * PT, o.y * PT);
    }
    R xb[PP];
#pragma unroll
    for (int q = 0; q < PP; ++q) xb[q] = R(0);
    for (int t = 0; t < g.T; ++t) {
        __syncthreads();
        const C2 *qt = Q + ((size_t)f * g.T + t) * h.U;
        for (int n = tid; n < h.U; n += GD_AT) sQ[n] = qt[__ldg(h.ord + n).z];
        Dir<R> dir[PP];
        R w[PP];
#pragma unroll
        for (int q = 0; q < PP; ++q) {
            const int p = min(p0 + q, g.npix - 1);                     // past the end: not stored
            dir[q].load(g, t, p);
            w[q] = pixel_weight<R>(g, f, t, p);
        }
        for (int a = 0; a < h.nant; ++a) {
            const Slopes<R> k = sK[a];
            C2 e[PP];
#pragma unroll
            for (int q = 0; q < PP; ++q) e[q] = dir[q].phasor(k, g.flat_array);
            if constexpr (PP == 2)
                *reinterpret_cast<float4 *>(sE + a * PT + 2 * tid) = make_float4(e[0].x, e[0].y, e[1].x, e[1].y);
            else
                sE[a * PT + tid] = e[0];
        }
        __syncthreads();
        C2 A[PP], B[PP];
        R acc[PP];
#pragma unroll
        for (int q = 0; q < PP; ++q) {
            A[q] = B[q] = mk2(R(0), R(0));
            acc[q] = R(0);
        }
        auto row = [&](int off, C2 (&v)[PP]) {
            if constexpr (PP == 2) load_pair(sE + off, tid, v);
            else v[0] = sE[off + tid];
        };
        auto close = [&](int off) {                                    // Re(E_i conj(Y_i)) of a finished run
            C2 e[PP];
            row(off, e);
#pragma unroll
            for (int q = 0; q < PP; ++q) {
                acc[q] += e[q].x * (A[q].x - B[q].y) + e[q].y * (A[q].y + B[q].x);
                A[q] = B[q] = mk2(R(0), R(0));
            }
        };
        int cur = sO[0].x;
        for (int n = 0; n < h.U; ++n) {
            const int2 o = sO[n];
            if (o.x != cur) {
                close(cur);
                cur = o.x;
            }
            const C2 u = sQ[n];
            C2 e[PP];
            row(o.y, e);
#pragma unroll
            for (int q = 0; q < PP; ++q) {
                A[q] = fma2(mk2(u.x, u.x), e[q], A[q]);
                B[q] = fma2(mk2(u.y, u.y), e[q], B[q]);
            }
        }
        close(cur);
#pragma unroll
        for (int q = 0; q < PP; ++q) xb[q] += w[q] * acc[q];
    }
#pragma unroll
    for (int q = 0; q < PP; ++q)
        if (p0 + q < g.npix) xbar[(size_t)f * g.npix + p0 + q] = xb[q];
}

template <typename R> size_t gd_fwd_smem(const Ctx &c)
{
    return c.fg.nant * (sizeof(typename V2<R>::t) * GD_PC + sizeof(Slopes<R>)) + sizeof(R) * GD_PC;
}
template <typename R> size_t gd_adj_smem(const Ctx &c)
{
    const size_t pt = GD_AT * (std::is_same<R, float>::value ? 2 : 1);
    return c.fg.nant * (sizeof(typename V2<R>::t) * pt + sizeof(Slopes<R>)) +
           c.fg.U * (sizeof(typename V2<R>::t) + sizeof(int2));
}

GdDev gd_dev(const Ctx &c)
{
    GdDev h;
    h.U = c.fg.U; h.nant = c.fg.nant; h.ntile = (int)cdiv(c.fg.U, GD_TU); h.nsplit = c.gd.nsplit;
    h.ord = c.gd.ord; h.ant = c.fg.ant;
    return h;
}

template <typename R>
fm_status gd_fwd_launch(Ctx &c, const R *x, typename V2<R>::t *part, cudaStream_t st)
{
    const GdDev h = gd_dev(c);
    FM_CK(smem_opt_in(k_gd_fwd<R>));
    k_gd_fwd<R><<<(unsigned)((long long)c.F * c.T * h.ntile * h.nsplit), 256, gd_fwd_smem<R>(c), st>>>(c.g, h, x, part);
    FM_CK_LAUNCH();
    return FM_OK;
}

template <typename T>
fm_status gd_alloc(Ctx &c, T **p, size_t bytes)
{
    void *q = nullptr;
    cudaError_t e = cudaMalloc(&q, bytes > 0 ? bytes : 16);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMalloc (fringe sums)", __FILE__, __LINE__);
    c.allocs.push_back(q);
    *p = reinterpret_cast<T *>(q);
    return FM_OK;
}

}  // namespace

// On for handles whose grid has no drift-scan form and whose groups and antennas fit (both real types,
// since the monopole visibilities of an FP32 handle are summed in FP64).  FM_HA_GROUPS=0 leaves it off.
fm_status gd_setup(Ctx &c)
{
    GdState &s = c.gd;
    const FringeGroups &fg = c.fg;
    s.on = false;
    if (const char *e = getenv("FM_HA_GROUPS"))
        if (atoi(e) == 0) return FM_OK;
    // with c.mm: only the monopole's sum off the pixel grid, which has a buffer of its own (launch_vis_gd)
    if ((c.ha.on && !c.mm.on) || c.hs.on || (c.mm.on && fg.drift) || fg.U > GD_MAX_U) return FM_OK;
    const bool f64 = c.prec == FM_PREC_FP64_SIMT;
    if (c.prec >= FM_PREC_BF16X1) return FM_OK;
    if (std::max(gd_fwd_smem<double>(c), f64 ? gd_adj_smem<double>(c) : gd_adj_smem<float>(c)) > 200 * 1024) return FM_OK;
    const int nch = (int)cdiv(c.npix, GD_PC), ntile = (int)cdiv(fg.U, GD_TU);
    const long long ctas = (long long)c.F * c.T * ntile;
    // about eight waves of four CTAs an SM, at least four pixel chunks a CTA
    s.nsplit = (int)std::max<long long>(1, std::min<long long>(nch / 4, cdiv(4864, ctas)));
    if (ctas * s.nsplit > 0x7fffffffLL || c.F > 65535) return FM_OK;
    std::vector<int4> ord(fg.U);
    for (int u = 0; u < fg.U; ++u) ord[u] = make_int4(fg.rep_i[u], fg.rep_j[u], u, 0);
    std::sort(ord.begin(), ord.end(), [](const int4 &a, const int4 &b) { return a.x != b.x ? a.x < b.x : a.y < b.y; });
    FM_TRY(gd_alloc(c, &s.ord, sizeof(int4) * ord.size()));
    FM_CK(cudaMemcpy(s.ord, ord.data(), sizeof(int4) * ord.size(), cudaMemcpyHostToDevice));
    if (!c.mm.on) {
        const size_t v = (size_t)c.F * c.T * fg.U * 2 * c.rsz;
        FM_TRY(gd_alloc(c, &s.part, v * s.nsplit));
        FM_TRY(gd_alloc(c, &s.qsum, v));
    }
    s.on = true;
    return FM_OK;
}

template <typename R>
fm_status launch_vis_gd(Ctx &c, const R *x, R *vis, cudaStream_t st, const R *dc, long long dcs)
{
    using C2 = typename V2<R>::t;
    if (c.prec < FM_PREC_BF16X1) FM_TRY(simt_supports<R>(c, false));
    // the FP64 monopole visibilities of an FP32 handle: their partial sums need twice its buffer
    C2 *part = (C2 *)c.gd.part, *tmp = nullptr;
    if (sizeof(R) != c.rsz) {
        FM_CK(cudaMalloc(&tmp, sizeof(C2) * (size_t)c.F * c.T * c.fg.U * c.gd.nsplit));
        part = tmp;
    }
    fm_status s = profiled(c, 0, st, [&]() -> fm_status { return gd_fwd_launch<R>(c, x, part, st); });
    if (s == FM_OK) s = launch_group_finish<R>(c, c.gd.nsplit, part, vis, st, dc, dcs);
    if (tmp) {
        cudaStreamSynchronize(st);
        cudaFree(tmp);
    }
    return s;
}

template <typename R>
fm_status launch_adjoint_gd(Ctx &c, const R *omega, R *xbar, cudaStream_t st)
{
    using C2 = typename V2<R>::t;
    if (c.prec < FM_PREC_BF16X1) FM_TRY(simt_supports<R>(c, true));
    FM_TRY(launch_group_qsum<R>(c, omega, c.gd.qsum, st));
    return profiled(c, 1, st, [&]() -> fm_status {
        constexpr int PT = GD_AT * (std::is_same<R, float>::value ? 2 : 1);
        FM_CK(smem_opt_in(k_gd_adj<R>));
        k_gd_adj<R><<<dim3(cdiv(c.npix, PT), c.F), GD_AT, gd_adj_smem<R>(c), st>>>(c.g, gd_dev(c), (const C2 *)c.gd.qsum,
                                                                                 xbar);
        FM_CK_LAUNCH();
        return FM_OK;
    });
}

#define GD_INST(R)                                                                                  \
    template fm_status launch_vis_gd<R>(Ctx &, const R *, R *, cudaStream_t, const R *, long long); \
    template fm_status launch_adjoint_gd<R>(Ctx &, const R *, R *, cudaStream_t);
GD_INST(float)
GD_INST(double)

}  // namespace fm
