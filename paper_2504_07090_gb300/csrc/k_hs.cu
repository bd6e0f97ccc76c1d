// Fringe groups, drift-scan geometry, and the drift-scan form of the contraction on the CUDA
// cores for the FP64 and FP32 handles.
//
// Baselines with equal vectors up to sign share their fringe (Eq. rime_discrete), so each distinct
// one is summed once: 63 instead of 666 for the 37-antenna hexagon.  In a drift scan with LSTs
// spaced by k / q RA pixels the direction of pixel r at LST t depends only on the hour-angle cell
// n = t k + (R - 1 - r) q, so one table of antenna phasors per (channel, declination, cell), built
// once per handle in FP64, replaces the sincos of every (antenna, pixel, LST), and the sum becomes
// a real matrix product over cells,
//   V_u(t) = sum_d sum_n P_u(n, d) x(r(n, t), d),   P_u = E_i conj(E_j),  E = sqrt(dOmega A) fringe,
// whose sky operand is a strip read at an offset that shifts with t.  With q > 1 the LSTs fall into
// q classes (t k mod q) that use the cells n = t k mod q only: within a class LST s = (t - t0) / q
// and cell v = (n - t0 k) / q meet at pixel r = R - 1 - (v - k s), so nothing of a class's work is
// spent on empty cells.
//
// Bound: FP32 (FP64) multiply-adds.  Each thread keeps 2 G rows x 4 LSTs (forward) or 4 cells x 8
// LSTs (adjoint) in registers, so that a shared-memory wavefront feeds several FMAs; the forward's
// FP32 products run on (Re, Im) pairs with packed FMAs.
//
// chi^2 + gradient, against the per-baseline sums of k_simt.cu (which stay for LSTs off the pixel
// grid): 37 antennas, 64 channels, 60 LSTs, 128 x 192 pixels in FP32 79.1 -> 3.13 ms; 7 antennas,
// 16 channels, 20 LSTs, 32 x 96 pixels in FP64 10.08 -> 0.44 ms.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <type_traits>
#include <unordered_map>
#include <vector>

#include "fm_internal.cuh"

namespace fm {

template <typename T>
static fm_status hs_alloc(Ctx &c, T **p, size_t bytes)
{
    void *q = nullptr;
    cudaError_t e = cudaMalloc(&q, bytes > 0 ? bytes : 16);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMalloc (fringe groups)", __FILE__, __LINE__);
    c.allocs.push_back(q);
    *p = reinterpret_cast<T *>(q);
    return FM_OK;
}

// LST step = k / q RA pixels (q <= 4, k <= 32).  The split precisions and FP32 accept a step that
// is off by 1e-9; FP64 handles, whose phases reach 1e3 rad, only LSTs within 2e-14 rad of the grid.
bool drift_step(const Ctx &c, int &k, int &q)
{
    const double dra = (c.cfg.ra_max - c.cfg.ra_min) / c.R;
    k = q = 1;
    if (c.T == 1) return true;
    const bool f64 = c.prec == FM_PREC_FP64_SIMT;
    const double dl = f64 ? (c.lst[c.T - 1] - c.lst[0]) / (c.T - 1) : c.lst[1] - c.lst[0];
    if (!f64)
        for (int t = 1; t < c.T; ++t)
            if (std::fabs(c.lst[t] - c.lst[0] - t * dl) > 1e-9 * dra) return false;
    const double kr = dl / dra;
    for (q = 1; q <= 4; ++q) {
        k = (int)std::llround(kr * q);
        if (k < 1 || k > 32 || std::fabs(kr * q - k) > 1e-9 * k) continue;
        if (!f64) return true;
        bool ok = true;
        for (int t = 1; t < c.T && ok; ++t) ok = std::fabs(c.lst[t] - c.lst[0] - t * (k * dra / q)) <= 2e-14;
        return ok;
    }
    return false;
}

// Groups by the cell of 1 um their vectors fall into; a vector on the edge of cells is looked for in all of them.  (Every
// vector against every group took 19 ms for 4950 baselines, and grew with their square.)
class FringeCells {
public:
    explicit FringeCells(double tol) : tol_(tol) {}
    void add(const double *v, int u)
    {
        double q[3];
        for (int c = 0; c < 3; ++c) q[c] = cell(v[c]);
        map_[key(q)].push_back(u);
    }
    // f(u) for every group within tol of v, and perhaps others
    template <typename F> void around(const double *v, F f) const
    {
        double lo[3], hi[3], q[3];
        for (int c = 0; c < 3; ++c) {
            lo[c] = cell(v[c] - 2.0 * tol_);
            hi[c] = cell(v[c] + 2.0 * tol_);
        }
        for (int s = 0; s < 8; ++s) {
            bool again = false;
            for (int c = 0; c < 3; ++c) {
                q[c] = s >> c & 1 ? hi[c] : lo[c];
                again = again || (s >> c & 1 && hi[c] == lo[c]);
            }
            if (again) continue;
            const auto it = map_.find(key(q));
            if (it == map_.end()) continue;
            for (int u : it->second) f(u);
        }
    }

private:
    static double cell(double x) { return std::floor(x * 1e6) + 0.0; }      // no negative zero
    static uint64_t key(const double *q)
    {
        uint64_t h = 0;
        for (int c = 0; c < 3; ++c) {
            uint64_t b;
            std::memcpy(&b, q + c, sizeof b);
            h = (h ^ b) * 0x9e3779b97f4a7c15ull;
            h ^= h >> 32;
        }
        return h;
    }
    double tol_;
    std::unordered_map<uint64_t, std::vector<int>> map_;
};

// Groups, covering antenna subset (greedy: add the antenna that completes the most groups, ties
// broken by partial coverage; each group's representative is a member pair inside it) and the
// device tables.  FM_HA_GROUPS=0 keeps every baseline a group of its own; FM_HA=0 switches the
// drift-scan forms off.
fm_status fringe_setup(Ctx &c)
{
    FringeGroups &fg = c.fg;
    bool ha = true;
    if (const char *e = getenv("FM_HA"))
        if (atoi(e) == 0) ha = false;
    fg.drift = ha && drift_step(c, fg.k, fg.q);
    if (fg.drift) fg.nh = (c.R - 1) * fg.q + (c.T - 1) * fg.k + 1;

    // equal baseline vectors up to sign: to 1 nm (a phase of 3e-9 at 2 m wavelength), to 1 pm on FP64
    // handles
    const double tol = c.prec == FM_PREC_FP64_SIMT ? 1e-12 : 1e-9;
    bool group = true;
    if (const char *e = getenv("FM_HA_GROUPS"))
        if (atoi(e) == 0) group = false;
    std::vector<int> rep_i, rep_j, bmap(c.B), bi(c.B), bj(c.B);
    std::vector<double> rep_b;
    std::vector<std::vector<int>> members;
    FringeCells cells(tol);
    for (int i = 0, b = 0; i < c.A; ++i)
        for (int j = i + 1; j < c.A; ++j, ++b) {
            bi[b] = i;
            bj[b] = j;
            const double v[3] = {c.ant[3 * i] - c.ant[3 * j], c.ant[3 * i + 1] - c.ant[3 * j + 1],
                                 c.ant[3 * i + 2] - c.ant[3 * j + 2]};
            int found = -1, cj = 0;       // the first group whose vector is v, or -v
            for (int flip = 0; flip < 2 && group; ++flip) {
                const double w[3] = {flip ? -v[0] : v[0], flip ? -v[1] : v[1], flip ? -v[2] : v[2]};
                cells.around(w, [&](int u) {
                    const double *r = &rep_b[3 * u];
                    if ((found >= 0 && u >= found) ||
                        !(std::fmax(std::fabs(w[0] - r[0]), std::fmax(std::fabs(w[1] - r[1]), std::fabs(w[2] - r[2]))) < tol))
                        return;
                    found = u;
                    cj = flip;
                });
            }
            if (found < 0) {
                found = (int)rep_i.size();
                rep_i.push_back(i);
                rep_j.push_back(j);
                rep_b.insert(rep_b.end(), v, v + 3);
                members.emplace_back();
                cells.add(v, found);
            }
            bmap[b] = 2 * found + cj;
            members[found].push_back(2 * b + cj);
        }
    fg.U = (int)rep_i.size();

    // Antennas whose phasors the table holds: a small set S such that every group has a
    // member pair inside S (greedy: add the antenna that completes the most groups, ties
    // broken by partial coverage); each group's representative is then such a pair.
    std::vector<int> in_s(c.A, 0), uncovered(fg.U, 1);
    int n_unc = fg.U;
    if (fg.U == c.B) {                     // nothing is redundant: every antenna is needed
        for (int a = 0; a < c.A; ++a) in_s[a] = 1;
        n_unc = 0;
    }
    std::vector<long long> full(c.A), part(c.A);
    std::vector<int> full_of(c.A), part_of(c.A);        // the last group counted
    while (n_unc > 0) {
        // per antenna: groups it completes, and partly covers (less those that every antenna does: the groups with a
        // member of one antenna in S, which only the antenna that completes the first such member may not)
        std::fill(full.begin(), full.end(), 0);
        std::fill(part.begin(), part.end(), 0);
        std::fill(full_of.begin(), full_of.end(), -1);
        std::fill(part_of.begin(), part_of.end(), -1);
        for (int u = 0; u < fg.U; ++u) {
            if (!uncovered[u]) continue;
            const std::vector<int> &mu = members[u];
            size_t first = 0;
            while (first < mu.size() && !in_s[bi[mu[first] >> 1]] && !in_s[bj[mu[first] >> 1]]) ++first;
            for (size_t k = 0; k < first; ++k)
                for (int a : {bi[mu[k] >> 1], bj[mu[k] >> 1]})
                    if (part_of[a] != u) {
                        part_of[a] = u;
                        if (first == mu.size()) ++part[a];
                    }
            for (size_t k = first; k < mu.size(); ++k) {
                const int i = bi[mu[k] >> 1], j = bj[mu[k] >> 1], a = in_s[i] ? j : i;
                if ((!in_s[i] && !in_s[j]) || full_of[a] == u) continue;
                full_of[a] = u;
                ++full[a];
                if (k == first && part_of[a] != u) --part[a];
            }
        }
        int best = -1;
        for (int a = 0; a < c.A; ++a)
            if (!in_s[a] && (best < 0 || full[a] > full[best] || (full[a] == full[best] && part[a] > part[best]))) best = a;
        in_s[best] = 1;
        for (int u = 0; u < fg.U; ++u) {
            if (!uncovered[u]) continue;
            for (int m : members[u]) {
                const int b = m >> 1;
                if (in_s[bi[b]] && in_s[bj[b]]) { uncovered[u] = 0; --n_unc; break; }
            }
        }
    }
    std::vector<int> pos(c.A, -1);
    fg.ant_of.clear();
    for (int a = 0; a < c.A; ++a)
        if (in_s[a]) { pos[a] = (int)fg.ant_of.size(); fg.ant_of.push_back(a); }
    fg.nant = (int)fg.ant_of.size();
    // representatives inside S, member orientation relative to them
    for (int u = 0; u < fg.U; ++u) {
        int rb = -1;
        for (int m : members[u]) {
            const int b = m >> 1;
            if (in_s[bi[b]] && in_s[bj[b]]) { rb = m; break; }
        }
        const int rflip = rb & 1;   // representative reversed w.r.t. the group's first member
        rep_i[u] = pos[bi[rb >> 1]];
        rep_j[u] = pos[bj[rb >> 1]];
        for (int &m : members[u]) m ^= rflip;
    }
    for (int u = 0; u < fg.U; ++u)
        for (int m : members[u]) bmap[m >> 1] = 2 * u + (m & 1);

    fg.rep_i = rep_i;
    fg.rep_j = rep_j;
    std::vector<int2> huij(fg.U);
    std::vector<int> hoff(fg.U + 1, 0), hmem;
    hmem.reserve(c.B);
    for (int u = 0; u < fg.U; ++u) {
        huij[u] = make_int2(rep_i[u], rep_j[u]);
        hoff[u] = (int)hmem.size();
        for (int m : members[u]) hmem.push_back(m);
    }
    hoff[fg.U] = (int)hmem.size();
    auto put = [&](auto **dst, const auto &src) -> fm_status {
        const size_t n = sizeof(src[0]) * src.size();
        FM_TRY(hs_alloc(c, dst, n));
        FM_CK(cudaMemcpy(*dst, src.data(), n, cudaMemcpyHostToDevice));
        return FM_OK;
    };
    std::vector<int2> hpair(c.B), hgm(c.B);
    for (int b = 0; b < c.B; ++b) hpair[b] = make_int2(bi[b] | (bj[b] << 16), bmap[b]);
    for (int m = 0; m < c.B; ++m) hgm[m] = make_int2(hmem[m], hpair[hmem[m] >> 1].x);
    FM_TRY(put(&fg.pairs, hpair));
    FM_TRY(put(&fg.gmem, hgm));
    FM_TRY(put(&fg.uij, huij));
    FM_TRY(put(&fg.ant, fg.ant_of));
    FM_TRY(put(&fg.bmap, bmap));
    FM_TRY(put(&fg.moff, hoff));
    return put(&fg.mem, hmem);
}

namespace {

template <typename R> struct C2of;
template <> struct C2of<float> { using t = float2; };
template <> struct C2of<double> { using t = double2; };

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ double2 fma2(double2 a, double2 b, double2 c)
{
    return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y));
}
__device__ __forceinline__ float2 mk2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ double2 mk2(double a, double b) { return make_double2(a, b); }

// n complex (n = 1, 2 or 4) from shared memory, 16 bytes at a time where the type allows it
template <int N> __device__ __forceinline__ void load_c(const float2 *p, float2 (&v)[N])
{
    if constexpr (N == 1) {
        v[0] = p[0];
    } else {
#pragma unroll
        for (int i = 0; i < N; i += 2) {
            const float4 q = *reinterpret_cast<const float4 *>(p + i);
            v[i] = make_float2(q.x, q.y);
            v[i + 1] = make_float2(q.z, q.w);
        }
    }
}
template <int N> __device__ __forceinline__ void load_c(const double2 *p, double2 (&v)[N])
{
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = p[i];
}

constexpr int HS_NC = 32;              // forward: cells staged at a time
constexpr int HA_CELLS = 256;          // adjoint: cells, LSTs and groups of a tile
constexpr int HA_LSTS = 32;
constexpr int HA_UG = 16;
constexpr int HA_LD = HA_CELLS + 4;

struct HsDev {
    int F, D, T, R, U, k, q, nant, row;
    int TU, TL, KS, nut, ntt, nsplit;
    int t0[4], off[4], n[4];           // LST classes
    const int2 *uij;
};

// ------------------------------------------------------------ per-handle phasor table
// E[f][d][a][off_c + v] = sqrt(dOmega_d A) exp(-2 pi i nu r_a . s / c) at the cell n = t0_c k + q v
// of class c, hour angle LST_0 - (ra_min + ((R - 1) q - n + q / 2) dRA / q); zero below the horizon.
struct HsTabArgs {
    double lst0, ra_min, dra, dec_min, ddec, lat, dew, dns;
    const double *kap64, *bcoef64, *domega64, *freq;
    const int *ant;
    int A_all, airy;
};

template <typename R>
__global__ void __launch_bounds__(256) k_hs_table(HsDev h, HsTabArgs a, typename C2of<R>::t *__restrict__ E)
{
    const long long total = (long long)h.F * h.D * h.row;
    double sl, cl;
    sincos(a.lat, &sl, &cl);
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int col = (int)(e % h.row);
        const long long fd = e / h.row;
        const int d = (int)(fd % h.D), f = (int)(fd / h.D);
        int c = 0;
        while (c + 1 < h.q && h.n[c + 1] > 0 && col >= h.off[c + 1]) ++c;
        const int v = col - h.off[c];
        double amp = 0.0, sE = 0.0, sN = 0.0, sU = 0.0;
        if (v < h.R + (h.n[c] - 1) * h.k) {
            const int n = h.t0[c] * h.k + h.q * v;
            const double H = a.lst0 - (a.ra_min + ((double)((h.R - 1) * h.q - n) + 0.5 * h.q) * (a.dra / h.q));
            const double dec = a.dec_min + (d + 0.5) * a.ddec;
            double sd, cd, sh, ch;
            sincos(dec, &sd, &cd);
            sincos(H, &sh, &ch);
            sE = -cd * sh;
            sN = cl * sd - sl * cd * ch;
            sU = sl * sd + cl * cd * ch;
            if (sU > 0.0) {
                const double za = acos(sU > 1.0 ? 1.0 : sU);
                amp = sqrt(a.domega64[d] * (a.airy ? airy_power(a.freq[f], sE, sN, sU, a.dew, a.dns)
                                                   : exp(a.bcoef64[f] * za * za)));
            }
        }
        for (int i = 0; i < h.nant; ++i) {
            double sn = 0.0, cs = 0.0;
            if (amp > 0.0) {
                const double *kp = a.kap64 + ((size_t)f * a.A_all + a.ant[i]) * 3;
                double ph = kp[0] * sE + kp[1] * sN + kp[2] * sU;
                ph -= rint(ph);
                sincospi(2.0 * ph, &sn, &cs);
            }
            E[((size_t)fd * h.nant + i) * h.row + col] = mk2((R)(amp * cs), (R)(-amp * sn));
        }
    }
}

// ------------------------------------------------------------ forward
// CTA = (channel, group tile of TU, LST tile of 4 TL of one class, split sp of the declinations).
// Per declination the reversed sky strip with zero margins goes to shared memory; 32 cells at a time
// the responses P of the tile's groups are formed there from the phasor table, and thread
// (rt, lt, ks) adds P x over the cells = ks mod KS for its G groups and LSTs lt + TL j.  A
// declination's sum is formed before it joins the total (FP32: the rounding error grows with R + D / nsplit
// terms, not with their product).  The splits' partial sums are added in order by k_group_finish.
template <typename R, int G>
__global__ void __launch_bounds__(256) k_hs_fwd(HsDev h, const typename C2of<R>::t *__restrict__ E,
                                                const R *__restrict__ x, typename C2of<R>::t *__restrict__ part)
{
    using C2 = typename C2of<R>::t;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int ST = 4 * h.TL, ldp = h.TU + 2, pad = h.k * (ST - 1);
    C2 *sP = reinterpret_cast<C2 *>(smem_raw);                 // [HS_NC][ldp]
    R *sX = reinterpret_cast<R *>(sP + HS_NC * ldp);           // [R + 2 pad]
    int2 *sIJ = reinterpret_cast<int2 *>(smem_raw + ((sizeof(C2) * HS_NC * ldp + sizeof(R) * (h.R + 2 * pad) + 15) & ~15));
    int b = blockIdx.x;
    const int sp = b % h.nsplit;
    b /= h.nsplit;
    const int tile = b % h.ntt, cls = (b / h.ntt) % h.q;
    b /= h.ntt * h.q;
    const int ut = b % h.nut, f = b / h.nut;
    const int S0 = tile * ST, ns = min(ST, h.n[cls] - S0);
    if (ns <= 0) return;
    const int u0 = ut * h.TU, nu = min(h.TU, h.U - u0);
    const int tid = threadIdx.x, TR = h.TU / G;
    const int rt = tid % TR, lt = (tid / TR) % h.TL, ks = tid / (TR * h.TL);
    for (int e = tid; e < nu; e += 256) {
        const int2 ij = h.uij[u0 + e];
        sIJ[e] = make_int2(ij.x * h.row, ij.y * h.row);
    }
    for (int e = tid; e < pad; e += 256) sX[e] = sX[pad + h.R + e] = R(0);
    for (int e = tid; e < HS_NC * ldp; e += 256) sP[e] = mk2(R(0), R(0));    // rows past nu stay zero
    C2 tot[G][4];
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
        for (int j = 0; j < 4; ++j) tot[g][j] = mk2(R(0), R(0));
    const int nv = h.R + (ns - 1) * h.k;
    const int d0 = (int)((long long)h.D * sp / h.nsplit), d1 = (int)((long long)h.D * (sp + 1) / h.nsplit);
    const C2 *Ec = E + h.off[cls] + h.k * S0;
    for (int d = d0; d < d1; ++d) {
        const size_t fd = (size_t)f * h.D + d;
        const C2 *Ed = Ec + fd * h.nant * h.row;
        __syncthreads();
        for (int e = tid; e < h.R; e += 256) sX[pad + h.R - 1 - e] = x[fd * h.R + e];
        C2 acc[G][4];
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[g][j] = mk2(R(0), R(0));
        for (int v0 = 0; v0 < nv; v0 += HS_NC) {
            const int nc = min(HS_NC, nv - v0);
            if (v0) __syncthreads();
            {
                const int v = tid % HS_NC;
                if (v < nc)
#pragma unroll 4
                    for (int u = tid / HS_NC; u < nu; u += 256 / HS_NC) {
                        const C2 a = __ldg(Ed + sIJ[u].x + v0 + v), c = __ldg(Ed + sIJ[u].y + v0 + v);
                        sP[v * ldp + u] = mk2(a.x * c.x + a.y * c.y, a.y * c.x - a.x * c.y);
                    }
            }
            __syncthreads();
            if (ks < h.KS) {
                const R *xs = sX + pad + v0 - h.k * lt;
                const int xj = h.k * h.TL;
#pragma unroll 2
                for (int v = ks; v < nc; v += h.KS) {
                    C2 p[G];
                    R y[4];
                    load_c<G>(sP + v * ldp + rt * G, p);
#pragma unroll
                    for (int j = 0; j < 4; ++j) y[j] = xs[v - j * xj];
#pragma unroll
                    for (int g = 0; g < G; ++g)
#pragma unroll
                        for (int j = 0; j < 4; ++j) acc[g][j] = fma2(p[g], mk2(y[j], y[j]), acc[g][j]);
                }
            }
        }
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
            for (int j = 0; j < 4; ++j) tot[g][j] = mk2(tot[g][j].x + acc[g][j].x, tot[g][j].y + acc[g][j].y);
    }
    // the KS cell classes' sums, added in order
    __syncthreads();
    C2 *red = reinterpret_cast<C2 *>(smem_raw);                // [KS][ST][TU]
    if (ks < h.KS)
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
            for (int j = 0; j < 4; ++j) red[((size_t)ks * ST + lt + h.TL * j) * h.TU + rt * G + g] = tot[g][j];
    __syncthreads();
    for (int e = tid; e < ns * nu; e += 256) {
        const int s = e / nu, u = e % nu;
        C2 r = red[s * h.TU + u];
        for (int kq = 1; kq < h.KS; ++kq) {
            const C2 w = red[((size_t)kq * ST + s) * h.TU + u];
            r.x += w.x;
            r.y += w.y;
        }
        const int t = h.t0[cls] + h.q * (S0 + s);
        part[(((size_t)sp * h.F + f) * h.T + t) * h.U + u0 + u] = r;
    }
}

// V of every member of a group: the splits' partial sums in order, conjugated for reversed
// members, plus the monopole dc[f dcs] Udc[f][t][b]
template <typename R, bool PAIR>
__global__ void __launch_bounds__(128) k_group_finish(int F, int T, int U, int nsplit, int B, const typename C2of<R>::t *__restrict__ part,
                                                   const int *__restrict__ moff, const int *__restrict__ mem,
                                                   const R *__restrict__ dc, long long dcs,
                                                   const float *__restrict__ Udc, R *__restrict__ vis)
{
    using C2 = typename C2of<R>::t;
    const long long n = (long long)F * T * U;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const int u = (int)(e % U);
        const long long ft = e / U;
        C2 s = mk2(R(0), R(0));
        for (int k0 = 0; k0 < nsplit; k0 += 8) {       // in order, eight loads ahead
            C2 w[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) w[k] = k0 + k < nsplit ? part[(size_t)(k0 + k) * n + e] : mk2(R(0), R(0));
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                s.x += w[k].x;
                s.y += w[k].y;
            }
        }
        const R cf = dc ? dc[(ft / T) * dcs] : R(0);
        for (int m = moff[u]; m < moff[u + 1]; ++m) {
            const int code = mem[m];
            const size_t o = 2 * ((size_t)ft * B + (code >> 1));
            C2 v = mk2(s.x, (code & 1) ? -s.y : s.y);
            if (dc) {
                v.x += cf * (R)Udc[o];
                v.y += cf * (R)Udc[o + 1];
            }
            put_pair(vis + o, v, PAIR);
        }
    }
}

// ------------------------------------------------------------ adjoint
// Q[f][t][u]: the members' residual weights summed (conjugated for reversed members)
template <typename R>
__global__ void __launch_bounds__(256) k_group_qsum(int F, int T, int U, int B, const R *__restrict__ omega,
                                                 const int *__restrict__ moff, const int *__restrict__ mem,
                                                 typename C2of<R>::t *__restrict__ Q)
{
    using C2 = typename C2of<R>::t;
    const long long n = (long long)F * T * U;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const int u = (int)(e % U);
        const long long ft = e / U;
        C2 s = mk2(R(0), R(0));
        for (int m = moff[u]; m < moff[u + 1]; ++m) {
            const int code = mem[m];
            const C2 w = *reinterpret_cast<const C2 *>(omega + 2 * ((size_t)ft * B + (code >> 1)));
            s.x += w.x;
            s.y += (code & 1) ? -w.y : w.y;
        }
        Q[e] = s;
    }
}

// xbar(r, d) = sum_t sum_u Re[conj(Q_u(t)) P_u(n(r, t), d)].  CTA = (channel, declination).  Per tile
// of 32 LSTs of a class and 256 cells, 16 groups at a time, P (formed from the table) and Q are
// staged and thread (ct, lt) keeps X[cell][LST] of 4 cells x 8 LSTs in registers; the tile then goes to
// shared memory and the thread of pixel r adds its diagonal v = R - 1 - r + k s in LST order.
template <typename R>
__global__ void __launch_bounds__(256) k_hs_adj(HsDev h, const typename C2of<R>::t *__restrict__ E,
                                                const typename C2of<R>::t *__restrict__ Q, R *__restrict__ xbar)
{
    using C2 = typename C2of<R>::t;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    R *sP = reinterpret_cast<R *>(smem_raw);                   // [2 HA_UG][HA_LD], then X [HA_LSTS][HA_LD]
    R *sQ = sP + HA_LSTS * HA_LD;                              // [2 HA_UG][HA_LSTS]
    R *sxb = sQ + 2 * HA_UG * HA_LSTS;                         // [R]
    static_assert(2 * HA_UG == HA_LSTS, "the two uses of sP");
    const int f = blockIdx.x / h.D, tid = threadIdx.x;
    const int ct = tid & 63, lt = tid >> 6;
    const C2 *Ed = E + (size_t)blockIdx.x * h.nant * h.row;
    for (int r = tid; r < h.R; r += 256) sxb[r] = R(0);
    for (int cls = 0; cls < h.q; ++cls) {
        const int ncls = h.n[cls], tcls = h.t0[cls], off = h.off[cls];
        for (int S0 = 0; S0 < ncls; S0 += HA_LSTS) {
            const int ns = min(HA_LSTS, ncls - S0), nv = h.R + (ns - 1) * h.k;
            for (int c0 = 0; c0 < nv; c0 += HA_CELLS) {
                const int nc = min(HA_CELLS, nv - c0);
                const C2 *Ec = Ed + off + h.k * S0 + c0;
                C2 acc[4][4];
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[i][j] = mk2(R(0), R(0));
                const bool work = 4 * ct < nc && 8 * lt < ns;
                for (int g0 = 0; g0 < h.U; g0 += HA_UG) {
                    const int ng = min(HA_UG, h.U - g0);
                    __syncthreads();
                    for (int u = 0; u < ng; ++u) {
                        const int2 ij = __ldg(h.uij + g0 + u);
                        C2 p = mk2(R(0), R(0));
                        if (tid < nc) {
                            const C2 a = __ldg(Ec + (size_t)ij.x * h.row + tid), b = __ldg(Ec + (size_t)ij.y * h.row + tid);
                            p = mk2(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
                        }
                        sP[(2 * u) * HA_LD + tid] = p.x;
                        sP[(2 * u + 1) * HA_LD + tid] = p.y;
                    }
                    for (int e = tid; e < ng * HA_LSTS; e += 256) {
                        const int u = e % ng, s = e / ng;
                        C2 w = mk2(R(0), R(0));
                        if (s < ns) w = Q[((size_t)f * h.T + tcls + h.q * (S0 + s)) * h.U + g0 + u];
                        sQ[(2 * u) * HA_LSTS + s] = w.x;
                        sQ[(2 * u + 1) * HA_LSTS + s] = w.y;
                    }
                    __syncthreads();
                    if (work)
#pragma unroll 2
                        for (int rho = 0; rho < 2 * ng; ++rho) {
                            C2 a2[2], w[4];
                            load_c<2>(reinterpret_cast<const C2 *>(sP + rho * HA_LD + 4 * ct), a2);
                            load_c<4>(reinterpret_cast<const C2 *>(sQ + rho * HA_LSTS + 8 * lt), w);
                            const R a[4] = {a2[0].x, a2[0].y, a2[1].x, a2[1].y};
#pragma unroll
                            for (int i = 0; i < 4; ++i)
#pragma unroll
                                for (int j = 0; j < 4; ++j) acc[i][j] = fma2(mk2(a[i], a[i]), w[j], acc[i][j]);
                        }
                }
                __syncthreads();
                if (work)
#pragma unroll
                    for (int j = 0; j < 4; ++j)
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            sP[(8 * lt + 2 * j) * HA_LD + 4 * ct + i] = acc[i][j].x;
                            sP[(8 * lt + 2 * j + 1) * HA_LD + 4 * ct + i] = acc[i][j].y;
                        }
                __syncthreads();
                for (int r = tid; r < h.R; r += 256) {
                    // LSTs whose cell R - 1 - r + k s lies in [c0, c0 + nc)
                    R v = R(0);
                    const int base = h.R - 1 - r - c0;
                    int s = base >= 0 ? 0 : (-base + h.k - 1) / h.k;
                    for (; s < ns && base + h.k * s < nc; ++s) v += sP[s * HA_LD + base + h.k * s];
                    sxb[r] += v;
                }
            }
        }
    }
    for (int r = tid; r < h.R; r += 256) xbar[(size_t)blockIdx.x * h.R + r] = sxb[r];
}

HsDev hs_dev(const Ctx &c)
{
    const HsState &s = c.hs;
    HsDev h;
    h.F = c.F; h.D = c.D; h.T = c.T; h.R = c.R; h.U = c.fg.U; h.k = c.fg.k; h.q = c.fg.q; h.nant = c.fg.nant;
    h.row = s.row;
    h.TU = s.TU; h.TL = s.TL; h.KS = s.KS; h.nut = s.nut; h.ntt = s.ntt; h.nsplit = s.nsplit;
    for (int i = 0; i < 4; ++i) { h.t0[i] = s.cls_t0[i]; h.off[i] = s.cls_off[i]; h.n[i] = s.cls_n[i]; }
    h.uij = c.fg.uij;
    return h;
}

template <typename R>
size_t fwd_smem(const Ctx &c, int TU, int TL, int KS)
{
    const size_t tiles = ((sizeof(R) * (2 * (size_t)HS_NC * (TU + 2) + c.R + 2 * (size_t)c.fg.k * (4 * TL - 1)) + 15) & ~(size_t)15) +
                         sizeof(int2) * TU;
    return std::max(tiles, sizeof(R) * 2 * (size_t)KS * 4 * TL * TU);
}

template <typename R>
size_t adj_smem(const Ctx &c) { return sizeof(R) * ((size_t)HA_LSTS * HA_LD + 2 * HA_UG * HA_LSTS + c.R); }

template <typename R>
fm_status hs_setup_t(Ctx &c)
{
    HsState &s = c.hs;
    const FringeGroups &fg = c.fg;
    int nmax = 0;
    s.row = 0;
    for (int t0 = 0; t0 < fg.q; ++t0) {
        const int n = t0 < c.T ? (c.T - t0 + fg.q - 1) / fg.q : 0;
        s.cls_t0[t0] = t0;
        s.cls_n[t0] = n;
        s.cls_off[t0] = s.row;
        if (n) s.row += (c.R + (n - 1) * fg.k + 3) & ~3;
        nmax = std::max(nmax, n);
    }
    // groups per thread and per tile: at most 16 row threads; 64 groups with 4 a thread
    s.G = fg.U >= 24 ? 4 : fg.U >= 12 ? 2 : 1;
    s.nut = (int)cdiv(fg.U, 16 * s.G);
    s.TU = (int)cdiv(cdiv(fg.U, s.nut), s.G) * s.G;
    const int TR = s.TU / s.G;
    // LSTs per tile: a tile of ST LSTs sums R + (ST - 1) k cells for every LST and forms each response
    // once, at the price of `form` LSTs' products
    const double form = std::is_same<R, double>::value ? 2.0 : 6.0;
    double best = 0.0;
    s.TL = 0;
    for (int tl = 1; tl <= 16 && TR * tl <= 256; ++tl) {
        const int st = 4 * tl, ks = std::min(256 / (TR * tl), HS_NC);
        if (fwd_smem<R>(c, s.TU, tl, ks) > 110 * 1024) continue;
        const double cost = (double)cdiv(nmax, st) * (c.R + (double)(std::min(st, nmax) - 1) * fg.k) * (st + form);
        if (s.TL == 0 || cost < best) { best = cost; s.TL = tl; }
    }
    if (s.TL == 0 || adj_smem<R>(c) > 200 * 1024) return FM_OK;
    s.KS = std::min(256 / (TR * s.TL), HS_NC);
    s.ntt = (int)cdiv(nmax, 4 * s.TL);
    const long long ctas = (long long)c.F * s.nut * s.ntt * fg.q;
    // about eight waves of two CTAs an SM, at least two declinations a CTA where there are that many CTAs
    s.nsplit = (int)std::max<long long>(1, std::min<long long>(c.D, cdiv(2432, ctas)));
    if (ctas * s.nsplit > 0x7fffffffLL || (long long)c.F * c.D > 0x7fffffffLL) return FM_OK;

    const size_t e_n = (size_t)c.F * c.D * fg.nant * s.row, v_n = (size_t)c.F * c.T * fg.U;
    size_t fr = 0, tot = 0;
    FM_CK(cudaMemGetInfo(&fr, &tot));
    if (sizeof(R) * 2 * (e_n + v_n * (s.nsplit + 1)) > fr / 2) return FM_OK;
    FM_TRY(hs_alloc(c, &s.E, sizeof(R) * 2 * e_n));
    FM_TRY(hs_alloc(c, &s.part, sizeof(R) * 2 * v_n * s.nsplit));
    FM_TRY(hs_alloc(c, &s.qsum, sizeof(R) * 2 * v_n));
    HsTabArgs a;
    a.lst0 = c.lst[0]; a.ra_min = c.cfg.ra_min; a.dra = (c.cfg.ra_max - c.cfg.ra_min) / c.R;
    a.dec_min = c.cfg.dec_min; a.ddec = (c.cfg.dec_max - c.cfg.dec_min) / c.D; a.lat = c.cfg.latitude_rad;
    a.dew = c.g.dish_ew; a.dns = c.g.dish_ns;
    a.kap64 = c.g.kap64; a.bcoef64 = c.g.bcoef64; a.domega64 = c.g.domega64; a.freq = c.g.freq64;
    a.ant = fg.ant; a.A_all = c.A; a.airy = c.g.beam32 != nullptr;
    k_hs_table<R><<<2048, 256>>>(hs_dev(c), a, (typename C2of<R>::t *)s.E);
    FM_CK_LAUNCH();
    FM_CK(cudaDeviceSynchronize());
    s.on = true;
    return FM_OK;
}

template <typename R, int G>
fm_status hs_fwd_launch(Ctx &c, const HsDev &h, const R *x, cudaStream_t st)
{
    using C2 = typename C2of<R>::t;
    FM_CK(smem_opt_in(k_hs_fwd<R, G>));
    k_hs_fwd<R, G><<<(unsigned)((long long)h.F * h.nut * h.q * h.ntt * h.nsplit), 256,
                     fwd_smem<R>(c, h.TU, h.TL, h.KS), st>>>(h, (const C2 *)c.hs.E, x, (C2 *)c.hs.part);
    FM_CK_LAUNCH();
    return FM_OK;
}

}  // namespace

fm_status hs_setup(Ctx &c)
{
    c.hs.on = false;
    if (c.prec >= FM_PREC_BF16X1 || c.ha.on || !c.fg.drift) return FM_OK;
    return c.prec == FM_PREC_FP64_SIMT ? hs_setup_t<double>(c) : hs_setup_t<float>(c);
}

static unsigned group_blocks(const Ctx &c)
{
    return (unsigned)std::min<long long>(cdiv((long long)c.F * c.T * c.fg.U, 256), 152 * 8);
}

template <typename R>
fm_status launch_group_finish(Ctx &c, int nsplit, const void *part, R *vis, cudaStream_t st, const R *dc, long long dcs)
{
    using C2 = typename C2of<R>::t;
    auto *kern = pair_aligned<C2>(vis) ? k_group_finish<R, true> : k_group_finish<R, false>;
    kern<<<2 * group_blocks(c), 128, 0, st>>>(c.F, c.T, c.fg.U, nsplit, c.B, (const C2 *)part, c.fg.moff, c.fg.mem, dc, dcs,
                                              c.dc_u, vis);
    FM_CK_LAUNCH();
    return FM_OK;
}

template <typename R>
fm_status launch_group_qsum(Ctx &c, const R *omega, void *q, cudaStream_t st)
{
    k_group_qsum<R><<<group_blocks(c), 256, 0, st>>>(c.F, c.T, c.fg.U, c.B, omega, c.fg.moff, c.fg.mem,
                                                     (typename C2of<R>::t *)q);
    FM_CK_LAUNCH();
    return FM_OK;
}

template <typename R>
fm_status launch_vis_hs(Ctx &c, const R *x, R *vis, cudaStream_t st, const R *dc, long long dcs)
{
    FM_TRY(simt_supports<R>(c, false));
    const HsDev h = hs_dev(c);
    FM_TRY(profiled(c, 0, st, [&]() -> fm_status {
        return c.hs.G == 4   ? hs_fwd_launch<R, 4>(c, h, x, st)
               : c.hs.G == 2 ? hs_fwd_launch<R, 2>(c, h, x, st)
                             : hs_fwd_launch<R, 1>(c, h, x, st);
    }));
    return launch_group_finish<R>(c, h.nsplit, c.hs.part, vis, st, dc, dcs);
}

template <typename R>
fm_status launch_adjoint_hs(Ctx &c, const R *omega, R *xbar, cudaStream_t st)
{
    using C2 = typename C2of<R>::t;
    FM_TRY(simt_supports<R>(c, true));
    const HsDev h = hs_dev(c);
    FM_TRY(launch_group_qsum<R>(c, omega, c.hs.qsum, st));
    return profiled(c, 1, st, [&]() -> fm_status {
        FM_CK(smem_opt_in(k_hs_adj<R>));
        k_hs_adj<R><<<(unsigned)(c.F * c.D), 256, adj_smem<R>(c), st>>>(h, (const C2 *)c.hs.E, (const C2 *)c.hs.qsum,
                                                                        xbar);
        FM_CK_LAUNCH();
        return FM_OK;
    });
}

#define HS_INST(R)                                                                                         \
    template fm_status launch_group_finish<R>(Ctx &, int, const void *, R *, cudaStream_t, const R *, long long); \
    template fm_status launch_group_qsum<R>(Ctx &, const R *, void *, cudaStream_t);                       \
    template fm_status launch_vis_hs<R>(Ctx &, const R *, R *, cudaStream_t, const R *, long long);        \
    template fm_status launch_adjoint_hs<R>(Ctx &, const R *, R *, cudaStream_t);
HS_INST(float)
HS_INST(double)

}  // namespace fm
