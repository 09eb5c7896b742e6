// rism_adjoint.cu -- reverse mode of the initialization grids.
//
// L = sum_s sum_r [G_u,s(r) u_s(r) + G_c,s(r) c_s(r) + G_h,s(r) h_s(r)] with u,
// c, h as defined in rism3d.h (Coulomb + truncated LJ, eq. (dcf-r),
// eq. (tcf-r)).  The paper has no gradient; these are the derivatives of
// those definitions.  Pair terms are recomputed, never stored.
//
// Site contraction first (per grid point, FP64 inputs):
//   W1 = k_e sum_s q_s G_u,s          (Coulomb part of u)
//   Wc = -beta k_e sum_s q_s G_c,s    (c)
//   Wh = -(beta k_e/(2 eps_r)) sum_s q_s G_h,s   (h)
// The long-range kernels split exactly as in the forward pass:
//   erf(x)/d = 1/d - erfc(x)/d,
//   phi_h(d) = 2 e^{a^2} e^{-kappa d}/d - Sh(d),
//   Sh(d) = e^{a^2}[e^{-kappa d} erfc(x-a) + e^{kappa d} erfc(x+a)]/d,
// so the far adjoint needs A1 = W1 + Wc (coefficient of 1/d) and
// Ak = 2 e^{a^2} Wh (coefficient of e^{-kappa d}/d) for every (point, atom)
// pair, and the near adjoint adds the erfc corrections within r_short and
// the LJ terms within the cut-offs.
//
//   k_adj_weights: W fields (float4 per point: A1, Ak, Wc, Wh; FP32)
//   k_adj_far:     atoms as targets (2 per thread), grid rows streamed through
//                  shared memory by bulk TMA copies; partials per row chunk
//   k_adj_sites, k_adj_near: warps of an atom over the grid points of its spheres
//   k_adj_final:   fixed-order sum of the partials, output in FP64
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>
#include <vector>

#include "rism_adjoint.h"
#include "rism_tree.h"

namespace rism {
namespace {

constexpr int kAT = 128;     // threads per far-adjoint CTA
constexpr int kAPT = 2;      // atoms per thread
constexpr int kRowT = 64;    // grid points per shared-memory tile (a row segment)
constexpr int kNearT = 256;  // threads per near-adjoint CTA

// A double as a float pair on the integer and FP32 pipes (the FP64 pipe of this part is slow): hi its leading 24 bits,
// lo the next 24.  The rare values outside FP32's normal range (with room for lo) go through the FP64 pipe.
static __device__ __noinline__ float2 split_slow(double v) {
    const float h = (float)v;
    const float l = (float)(v - (double)h);
    return make_float2(h, isfinite(l) ? l : 0.f);  // an infinite or NaN v stays in hi
}
__device__ __forceinline__ float2 split_d(double v) {
    const uint32_t hw = (uint32_t)__double2hiint(v), lw = (uint32_t)__double2loint(v);
    const uint32_t e = (hw >> 20) & 0x7ffu;
    if (e - 930u > 200u) return (hw << 1 | lw) == 0u ? make_float2(0.f, 0.f) : split_slow(v);
    const uint32_t sign = hw & 0x80000000u, ef = (e - 896u) << 23;
    const float hi = __uint_as_float(sign | ef | ((hw & 0xfffffu) << 3) | (lw >> 29));
    // the low 29 bits m: 2^(e - 52) m, its leading 23 bits written under the exponent of 2^(e - 23) and that taken off
    const float one = __uint_as_float(sign | (ef - (23u << 23)));
    const float lo = __uint_as_float(sign | (ef - (23u << 23)) | ((lw & 0x1fffffffu) >> 6)) - one;
    return make_float2(hi, lo);
}

// Site-contraction coefficients as float pairs: k_e q_s, -beta k_e q_s, -(beta k_e/(2 eps_r)) q_s, and 2 e^{a^2}.
struct WeightCoef {
    float h[3][kMaxSites], l[3][kMaxSites];
    float e2h, e2l;
};

// Bound by memory: 64 bytes read and 32 written per point and four sites of two cotangents (55,000 atoms' grid, 3.8 GB:
// 0.68 ms; the same sums on the FP64 pipe 1.66 ms).
template <int NS>
__device__ __forceinline__ void weight_sum(const float2 (&g)[NS], const float* ch, const float* cl, int S, float& h,
                                           float& l) {
    h = l = 0.f;
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        if (s >= S) break;
        const float p = ch[s] * g[s].x;
        ff_add(h, l, p);
        l += fmaf(ch[s], g[s].x, -p) + (ch[s] * g[s].y + cl[s] * g[s].x);
    }
}
template <int NS>
__global__ void __launch_bounds__(256) k_adj_weights(int64_t M, int S, const double* __restrict__ gu,
                                                     const double* __restrict__ gc, const double* __restrict__ gh,
                                                     const __grid_constant__ WeightCoef k, float4* w, float4* gu4) {
    for (int64_t f = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; f < M; f += (int64_t)gridDim.x * blockDim.x) {
        float h[3] = {0.f, 0.f, 0.f}, l[3] = {0.f, 0.f, 0.f};
        const double* in[3] = {gu, gc, gh};
        double raw[3][NS];  // every load first
#pragma unroll
        for (int q = 0; q < 3; ++q)
#pragma unroll
            for (int s = 0; s < NS; ++s) raw[q][s] = in[q] && s < S ? __ldcs(in[q] + s * M + f) : 0.0;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            if (!in[q]) continue;
            float2 g[NS];
#pragma unroll
            for (int s = 0; s < NS; ++s) g[s] = split_d(raw[q][s]);
            weight_sum<NS>(g, k.h[q], k.l[q], S, h[q], l[q]);
            if (q == 0) {
                float v[8] = {};
#pragma unroll
                for (int s = 0; s < NS; ++s) v[s] = g[s].x + g[s].y;
                gu4[f] = make_float4(v[0], v[1], v[2], v[3]);
                if (NS > 4) gu4[M + f] = make_float4(v[4], v[5], v[6], v[7]);
            }
        }
        float a, e;
        two_sum(h[0], h[1], a, e);
        const float pk = k.e2h * h[2];
        // an infinite sum's low part is not a number: the high part stands alone
        auto both = [](float hi, float lo) { return isfinite(hi) ? hi + lo : hi; };
        w[f] = make_float4(both(a, e + l[0] + l[1]), both(pk, fmaf(k.e2h, h[2], -pk) + (k.e2h * l[2] + k.e2l * h[2])),
                           both(h[1], l[1]), both(h[2], l[2]));
    }
}

struct FarAdjArgs {
    int nx, ny, nz;
    int n;
    int seg_per_row, nseg;   // row segments of kRowT points
    int chunks;              // grid chunks (partials per atom)
    float kap_g;             // kappa in 1/grid units
    float kap2;              // -kappa h log2(e): e^{-kappa d} = 2^(kap2 d_grid)
    const SrcF* srcf;
    const float4* w;
    double* part;            // [chunks][n][4]: dq, Gx, Gy, Gz (grid units)
    DevErr* err;
    long long wlim;
};

// Atoms as targets, grid points as sources.  Row segments of kRowT points are
// contiguous in the W array, so one bulk copy brings a tile; y and z are
// constant along it and x advances by one grid unit per point.
template <bool DH>
__global__ void __launch_bounds__(kAT) k_adj_far(FarAdjArgs a) {
    __shared__ __align__(16) float4 tile[2][kRowT];
    __shared__ __align__(8) uint64_t bar[2];
    const int tid = threadIdx.x;
    const int chunk = blockIdx.y;
    const int s0 = (int)((int64_t)a.nseg * chunk / a.chunks), s1 = (int)((int64_t)a.nseg * (chunk + 1) / a.chunks);
    float xh[kAPT], yh[kAPT], zh[kAPT], xl[kAPT], yl[kAPT], zl[kAPT];
    float dqh[kAPT], dql[kAPT], gxh[kAPT], gxl[kAPT], gyh[kAPT], gyl[kAPT], gzh[kAPT], gzl[kAPT];
    int atom[kAPT];
#pragma unroll
    for (int u = 0; u < kAPT; ++u) {
        atom[u] = (blockIdx.x * kAPT + u) * kAT + tid;
        const SrcF s = atom[u] < a.n ? a.srcf[atom[u]] : SrcF{1e30f, 1e30f, 1e30f, 0.f, 0.f, 0.f, 0.f, 0.f};
        xh[u] = s.xh; yh[u] = s.yh; zh[u] = s.zh;
        xl[u] = s.xl; yl[u] = s.yl; zl[u] = s.zl;
        dqh[u] = dql[u] = gxh[u] = gxl[u] = gyh[u] = gyl[u] = gzh[u] = gzl[u] = 0.f;
    }
    if (tid == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        mbar_fence_init();
    }
    __syncthreads();
    const int nt = s1 - s0;
    auto seg_len = [&](int sg) {
        const int within = sg % a.seg_per_row;
        return min(kRowT, a.nx - within * kRowT);
    };
    auto issue = [&](int t) {
        const int sg = s0 + t;
        const int row = sg / a.seg_per_row, within = sg % a.seg_per_row;
        const int len = seg_len(sg);
        const uint32_t bytes = len * sizeof(float4);
        mbar_expect_tx(&bar[t & 1], bytes);
        bulk_g2s(tile[t & 1], a.w + (int64_t)row * a.nx + within * kRowT, bytes, &bar[t & 1]);
    };
    if (tid == 0) {
        if (nt > 0) issue(0);
        if (nt > 1) issue(1);
    }
    for (int t = 0; t < nt; ++t) {
        const bool ok = mbar_wait_bounded(&bar[t & 1], (t >> 1) & 1, a.wlim);
        if (__syncthreads_or(!ok)) {
            if (tid == 0) {
                report_error(a.err, DEV_TIMEOUT, WHERE_ADJOINT);
                for (int u2 = t; u2 < min(t + 2, nt); ++u2) mbar_wait_bounded(&bar[u2 & 1], (u2 >> 1) & 1, a.wlim);
            }
            return;
        }
        const int sg = s0 + t;
        const int row = sg / a.seg_per_row, within = sg % a.seg_per_row;
        const int len = seg_len(sg);
        const float fy = (float)(row % a.ny), fz = (float)(row / a.ny);
        const float fx0 = (float)(within * kRowT);
        const float4* W = tile[t & 1];
        float dy[kAPT], dz[kAPT], dyz2[kAPT], pq[kAPT], px[kAPT], pyz[kAPT];
#pragma unroll
        for (int u = 0; u < kAPT; ++u) {
            dy[u] = (fy - yh[u]) - yl[u];
            dz[u] = (fz - zh[u]) - zl[u];
            dyz2[u] = fmaf(dy[u], dy[u], dz[u] * dz[u]);
            pq[u] = px[u] = pyz[u] = 0.f;
        }
        float fx = fx0;
        for (int p = 0; p < len; ++p, fx += 1.0f) {
            const float4 wv = W[p];
#pragma unroll
            for (int u = 0; u < kAPT; ++u) {
                const float dx = (fx - xh[u]) - xl[u];
                const float d2 = fmaf(dx, dx, dyz2[u]);
                const float rr = rsqrt_approx(d2);
                const float ri = d2 > 0.f ? rr : 0.f;
                const float ri2 = ri * ri;
                float t1 = wv.x * ri, tg = t1;
                if (DH) {
                    const float d = d2 * ri;
                    const float tk = wv.y * ri * ex2_approx(a.kap2 * d);
                    t1 += tk;
                    tg = fmaf(tk, a.kap_g * d, t1);
                }
                pq[u] += t1;
                const float rad = tg * ri2;
                px[u] = fmaf(dx, rad, px[u]);
                pyz[u] += rad;  // (dy, dz) are constant along the row
            }
        }
#pragma unroll
        for (int u = 0; u < kAPT; ++u) {
            ff_add(dqh[u], dql[u], pq[u]);
            ff_add(gxh[u], gxl[u], px[u]);
            ff_add(gyh[u], gyl[u], dy[u] * pyz[u]);
            ff_add(gzh[u], gzl[u], dz[u] * pyz[u]);
        }
        __syncthreads();
        if (tid == 0 && t + 2 < nt) issue(t + 2);
    }
#pragma unroll
    for (int u = 0; u < kAPT; ++u) {
        if (atom[u] >= a.n) continue;
        double* o = a.part + ((int64_t)chunk * a.n + atom[u]) * 4;
        o[0] = (double)dqh[u] + (double)dql[u];
        o[1] = (double)gxh[u] + (double)gxl[u];
        o[2] = (double)gyh[u] + (double)gyl[u];
        o[3] = (double)gzh[u] + (double)gzl[u];
    }
}

struct NearAdjArgs {
    GridD g;
    int n, S, smax;
    const SrcF* srcf;
    const LJf* ljf;          // [n][smax] grid units
    const float2* site;      // [n][smax] d ln(sigma_is)/d sigma_i, d ln(eps_is)/d eps_i
    const float4* w;
    const float4* gu4;       // [ceil(S/4)][M]: G_u of the sites in FP32, four per record (nullable)
    const uint32_t* order;   // position -> atom (Morton order from the tree, for cache reuse); null: identity
    const float4* tab;       // [kAdjTab][4]: cubic pieces of C0, C1, H0, H1
    float tab_inv;           // kAdjTab / r_short (grid units)
    float rs, rs2;           // r_short (grid units)
    float xs, aa;            // h / eta and kappa eta / 2, where the functions are called
    int wpa;                 // warps per atom: 1, 2, 4 or 8
    double* out;             // [n][9]: dq, Gx, Gy, Gz (grid units as in the far part), dLJ/dR (3), dsigma, deps
};

struct SiteLJ {
    double sig[kMaxSites], eps[kMaxSites];
};

// The mixing derivatives of every (atom, site) pair, in FP64.
__global__ void k_adj_sites(int n, int S, int smax, const double* __restrict__ raw, SiteLJ lj, float2* site) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= (int64_t)n * smax) return;
    const int64_t i = t / smax;
    const int s = (int)(t - i * smax);
    float2 v = make_float2(0.f, 0.f);
    if (s < S) {
        const double sig = 0.5 * (raw[6 * i + 4] + lj.sig[s]);
        const double eps = sqrt(raw[6 * i + 5] * lj.eps[s]);
        v.x = sig > 0.0 ? (float)(0.5 / sig) : 0.f;                                       // dsigma_is/dsigma_i / sigma_is
        v.y = eps > 0.0 ? (float)(lj.eps[s] / (2.0 * eps * eps)) : 0.f;         // (deps_is/deps_i) / eps_is
    }
    site[t] = v;
}

// The short-range kernels of the reverse mode in d over [0, r_short], kAdjTab cubic Hermite pieces each (built in FP64):
// with x = d/eta, C0 = erfc(x) and H0 = e^{-x^2}[erfcx(x-a) + erfcx(x+a)] the potentials are Sc = C0/d and Sh = H0/d, and
// with C1 = C0 - d C0', H1 = H0 - d H0' their slopes are -C1/d^2 and -H1/d^2.  Evaluated in FP32 the pieces are within 7e-8
// (C) and 1.2e-7 (H at a = 0) to 5.5e-7 (a = 1) of the functions, which evaluated in FP32 are within 1.1e-7 and 2.7e-7 to
// 1.0e-6; but the error of a piece grows with the fourth power of a times its width (H1 at a = 2: 1.1e-4 against 3.4e-5),
// so a stronger screening than kAdjPieceA takes the functions.
constexpr int kAdjTab = 256;
constexpr double kAdjPieceA = 1.0;

// C0, C1, H0, H1 at d = x eta by the functions themselves.
__device__ __forceinline__ float4 near_functions(float x, float a) {
    const float ex = __expf(-x * x), em = erfcxf(x - a), ep = erfcxf(x + a), c0 = erfcf(x), h0 = ex * (em + ep);
    const float tsp = 1.12837917f;  // 2/sqrt(pi)
    return make_float4(c0, fmaf(x * tsp, ex, c0), h0, h0 - x * (2.f * a * ex * (ep - em) - 2.f * tsp * ex));
}

struct FFs {
    float h, l;
};
__device__ __forceinline__ void ffs_add(FFs& a, FFs b) {
    float s, e;
    two_sum(a.h, b.h, s, e);
    a.h = s;
    a.l += b.l + e;
}
__device__ __forceinline__ FFs ffs_mul(float c, FFs x) {
    const float p = c * x.h;
    return FFs{p, fmaf(c, x.h, -p) + c * x.l};
}

// A tile of 8 x 4 grid columns (one per lane) of the box [lo, hi] around an atom, cut to the sphere r2 = r^2.
struct ColTile {
    float fx, fy;        // the column's grid indices
    float dx, dy, dxy2;  // dxy2 infinite outside the grid or the sphere: such a column has no term
    int64_t at;          // first point (a lane outside reads a neighbour's column)
    int k0, k1;          // z range of the warp
};
__device__ __forceinline__ ColTile col_tile(const GridD& g, const SrcF& sf, const int (&lo)[3], const int (&hi)[3],
                                            float r2, int t, int ntx, int lane) {
    ColTile c;
    const int ii = lo[0] + (t % ntx) * 8 + (lane & 7), jj = lo[1] + (t / ntx) * 4 + (lane >> 3);
    c.fx = (float)ii;
    c.fy = (float)jj;
    c.dx = (c.fx - sf.xh) - sf.xl;
    c.dy = (c.fy - sf.yh) - sf.yl;
    c.dxy2 = fmaf(c.dx, c.dx, c.dy * c.dy);
    const bool in = ii <= hi[0] && jj <= hi[1] && c.dxy2 < r2;
    if (!in) c.dxy2 = INFINITY;
    // the chord of the column (one grid unit of margin; the pair test decides)
    const float hz = in ? (isfinite(r2) ? sqrtf(r2 - c.dxy2) + 1.0f : 1e6f) : 0.f;
    const int a0 = in ? max(lo[2], (int)floorf(fmaxf(sf.zh - hz, -1e6f))) : INT_MAX;
    const int a1 = in ? min(hi[2], (int)ceilf(fminf(sf.zh + hz, 1e6f))) : -1;
    c.k0 = __reduce_min_sync(0xffffffffu, a0);
    c.k1 = __reduce_max_sync(0xffffffffu, a1);
    if (c.k0 == INT_MAX) c.k0 = 0;  // k1 = -1: empty
    c.at = ((int64_t)c.k0 * g.ny + min(jj, hi[1])) * g.nx + min(ii, hi[0]);
    return c;
}

// d^2 of a near point less its rounded value d2: (px, py, pz) is the part of the high difference that (dx, dy, dz) took,
// so px - xl is what the rounding of dx left (exact for the nearest points).
__device__ __forceinline__ float dist2_rest(float dx, float dy, float dz, float px, float py, float pz, const SrcF& sf,
                                            float d2) {
    const float x2 = dx * dx, y2 = dy * dy, z2 = dz * dz;
    float s1, e1, s2, e2;
    two_sum(x2, y2, s1, e1);
    two_sum(s1, z2, s2, e2);
    const float e = fmaf(dx, dx, -x2) + fmaf(dy, dy, -y2) + fmaf(dz, dz, -z2);
    const float low = fmaf(dx, px - sf.xl, fmaf(dy, py - sf.yl, dz * (pz - sf.zl)));
    return (s2 - d2) + (e1 + e2 + e + 2.f * low);
}

// The box of grid points within r (grid units, possibly infinite) of the atom; false when it is empty.
__device__ __forceinline__ bool point_box(const GridD& g, const SrcF& sf, float r, int (&lo)[3], int (&hi)[3]) {
    const float c[3] = {sf.xh, sf.yh, sf.zh};
    const int nn[3] = {g.nx, g.ny, g.nz};
    bool any = true;
    for (int d = 0; d < 3; ++d) {
        lo[d] = (int)fminf(fmaxf(ceilf(c[d] - r - 0.01f), 0.f), 1e6f);
        hi[d] = (int)fmaxf(fminf(floorf(c[d] + r + 0.01f), (float)(nn[d] - 1)), -1.f);
        any = any && lo[d] <= hi[d];
    }
    return any;
}

constexpr int kFold = 64;
// wpa warps per atom over the grid columns of its spheres: the erfc corrections (dq, G) within r_short, then the LJ
// terms within the largest cut-off of the atom's sites.  A lane owns a column of a tile and goes down its chord, so x
// and y offsets are fixed and the x, y forces take the column's sum once.  Per site the sums of G_u/d^12 and G_u/d^6
// are kept (two sites per two-wide instruction); sigma and eps gradients follow from them at the end.  FP32 sums of at
// most kFold points of a column, folded into float pairs, so that rounding does not grow with the length of a column (all
// of nz without a cut-off); a chord within a cut-off is mostly one fold.  UNI: one cut-off for all of an atom's sites.
// FN: the short-range kernels by their functions instead of the pieces.
// Bound by issue and the latency of the cotangent loads (two CTAs per SM at 121 registers; three at 80 spill and are
// slower).  2,000 atoms on 128^3: 0.34 ms (1.02 ms with one CTA per atom that called erfc, erfcx and, in every thread,
// the FP64 mixing derivatives); 55,000 atoms on 320x320x384, u and c: 7.7 ms (21.2).
template <int NR, bool UNI, bool FN>
__global__ void __launch_bounds__(kNearT) k_adj_near(const __grid_constant__ NearAdjArgs a) {
    __shared__ float4 tab[kAdjTab][4];
    __shared__ FFs red[kNearT / 32][9];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const GridD& g = a.g;
    const int64_t plane = (int64_t)g.nx * g.ny, M = plane * g.nz;
    if (!FN)
        for (int k = threadIdx.x; k < 4 * kAdjTab; k += kNearT) tab[k >> 2][k & 3] = a.tab[k];
    __syncthreads();
    const int per = (kNearT / 32) / a.wpa, sub = w % a.wpa;  // atoms per CTA pass; this warp's share of its atom
    for (int p0 = blockIdx.x * per; p0 < a.n; p0 += gridDim.x * per) {
        const int pos = p0 + w / a.wpa;
        const bool live = pos < a.n;
        const int i = live ? (a.order ? (int)a.order[pos] : pos) : 0;
        FFs v[9];
#pragma unroll
        for (int q = 0; q < 9; ++q) v[q] = FFs{0.f, 0.f};
        const SrcF sf = a.srcf[i];
        int lo[3], hi[3];
        if (live && point_box(g, sf, a.rs, lo, hi)) {
            const int ntx = (hi[0] - lo[0]) / 8 + 1, nt = ntx * ((hi[1] - lo[1]) / 4 + 1);
            for (int t = sub; t < nt; t += a.wpa) {
                const ColTile c = col_tile(g, sf, lo, hi, a.rs2, t, ntx, lane);
                const float4* pw = a.w + c.at;
                float fk = (float)c.k0;
                for (int kb = c.k0; kb <= c.k1; kb += kFold) {
                    const int ke = min(c.k1, kb + kFold - 1);
                    float dq = 0.f, rs = 0.f, rz = 0.f;
#pragma unroll 4
                    for (int kk = kb; kk <= ke; ++kk, pw += plane, fk += 1.f) {
                        const float2 W = __ldg(reinterpret_cast<const float2*>(pw) + 1);  // Wc, Wh
                        const float dz = (fk - sf.zh) - sf.zl;
                        const float d2 = fmaf(dz, dz, c.dxy2);
                        const bool ok = d2 < a.rs2 && d2 > 0.f;
                        const float dd = ok ? d2 : 1.f;
                        const float ri = rsqrt_approx(dd);
                        const float wc = ok ? W.x : 0.f, wh = ok ? W.y : 0.f;
                        float f0, f1;
                        if (FN) {
                            const float4 k = near_functions(dd * ri * a.xs, a.aa);
                            // without a cotangent of h nothing of its kernel enters (it overflows at extreme screening)
                            f0 = fmaf(wc, k.x, wh != 0.f ? wh * k.z : 0.f);
                            f1 = fmaf(wc, k.y, wh != 0.f ? wh * k.w : 0.f);
                        } else {
                            const float u = dd * ri * a.tab_inv;
                            // segment of u: adding 1.5 2^23 leaves round(u - 1/2) in the low bits of the sum
                            const float sh = (u - 0.5f) + 12582912.0f;
                            const int it = min(__float_as_int(sh) - 0x4B400000, kAdjTab - 1);
                            const float tt = u - fminf(sh - 12582912.0f, (float)(kAdjTab - 1));
                            auto piece = [&](int f) {
                                const float4 k = tab[it][f];
                                return fmaf(fmaf(fmaf(k.w, tt, k.z), tt, k.y), tt, k.x);
                            };
                            f0 = fmaf(wc, piece(0), wh * piece(2));
                            f1 = fmaf(wc, piece(1), wh * piece(3));
                        }
                        dq = fmaf(-f0, ri, dq);
                        const float rad = f1 * ri * ri * ri;
                        rs += rad;
                        rz = fmaf(dz, rad, rz);
                    }
                    ff_add(v[0].h, v[0].l, dq);
                    ff_add(v[1].h, v[1].l, c.dxy2 < INFINITY ? c.dx * rs : 0.f);
                    ff_add(v[2].h, v[2].l, c.dxy2 < INFINITY ? c.dy * rs : 0.f);
                    ff_add(v[3].h, v[3].l, rz);
                }
            }
        }
        if (live && a.gu4) {
            f32x2 A[2 * NR], B[2 * NR];
            float rc[4 * NR], rmax = 0.f;
#pragma unroll
            for (int s = 0; s < 2 * NR; ++s) {
                float x[2] = {0.f, 0.f}, y[2] = {0.f, 0.f};
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const int q = 2 * s + k;
                    rc[q] = 0.f;
                    if (q < a.S) {
                        const LJf l = a.ljf[(int64_t)i * a.smax + q];
                        x[k] = l.A;
                        y[k] = l.B;
                        rc[q] = l.rc2;
                    }
                    rmax = fmaxf(rmax, rc[q]);
                }
                A[s] = pk2(x[0], x[1]);
                B[s] = pk2(y[0], y[1]);
            }
            FFs x12[4 * NR], x6[4 * NR];
#pragma unroll
            for (int q = 0; q < 4 * NR; ++q) x12[q] = x6[q] = FFs{0.f, 0.f};
            const bool any = point_box(g, sf, sqrtf(rmax), lo, hi);
            const int ntx = any ? (hi[0] - lo[0]) / 8 + 1 : 1, nt = any ? ntx * ((hi[1] - lo[1]) / 4 + 1) : 0;
            for (int t = sub; t < nt; t += a.wpa) {
                const ColTile c = col_tile(g, sf, lo, hi, rmax, t, ntx, lane);
                const float4* pg = a.gu4 + c.at;
                float fk = (float)c.k0;
                for (int kb = c.k0; kb <= c.k1; kb += kFold) {
                    const int ke = min(c.k1, kb + kFold - 1);
                    f32x2 s12[2 * NR], s6[2 * NR];
#pragma unroll
                    for (int s = 0; s < 2 * NR; ++s) s12[s] = s6[s] = 0ull;
                    float fs = 0.f, fz = 0.f;
#pragma unroll 4
                    for (int kk = kb; kk <= ke; ++kk, pg += plane, fk += 1.f) {
                        ulonglong2 gv[NR];  // loaded before the tests: the loads of the unrolled points run together
#pragma unroll
                        for (int q = 0; q < NR; ++q) gv[q] = __ldg(reinterpret_cast<const ulonglong2*>(pg + q * M));
                        const float dz = (fk - sf.zh) - sf.zl;
                        const float d2 = fmaf(dz, dz, c.dxy2);
                        // a point outside the cut-off, or on the atom, has no term whatever its cotangent is
                        const bool ok = d2 < rmax && d2 > 0.f;
                        float r2 = rcp_approx(ok ? d2 : 1.f);
                        // the nearest points carry the sums, and their error counts seven times: there 1/d^2 takes what
                        // the rounding of d^2 and of the reciprocal left
                        if (__any_sync(0xffffffffu, ok && d2 < 4.f)) {
                            const float e = dist2_rest(c.dx, c.dy, dz, (c.fx - sf.xh) - c.dx, (c.fy - sf.yh) - c.dy,
                                                       (fk - sf.zh) - dz, sf, d2);
                            r2 = fmaf(r2, fmaf(-d2, r2, 1.f) - e * r2, r2);
                        }
                        if (!ok) r2 = 0.f;
                        f32x2 G[2 * NR];
#pragma unroll
                        for (int q = 0; q < NR; ++q) {
                            G[2 * q] = ok ? gv[q].x : 0ull;
                            G[2 * q + 1] = ok ? gv[q].y : 0ull;
                        }
                        if (!UNI) {
#pragma unroll
                            for (int s = 0; s < 2 * NR; ++s) {
                                const float2 q = up2(G[s]);
                                G[s] = pk2(d2 < rc[2 * s] ? q.x : 0.f, d2 < rc[2 * s + 1] ? q.y : 0.f);
                            }
                        }
                        const float r6 = r2 * r2 * r2, r12 = r6 * r6;
                        const f32x2 R6 = pk2(r6, r6), R12 = pk2(r12, r12);
                        f32x2 T12 = mul2(A[0], G[0]), T6 = mul2(B[0], G[0]);
#pragma unroll
                        for (int s = 1; s < 2 * NR; ++s) {
                            T12 = fma2(A[s], G[s], T12);
                            T6 = fma2(B[s], G[s], T6);
                        }
#pragma unroll
                        for (int s = 0; s < 2 * NR; ++s) {
                            s12[s] = fma2(G[s], R12, s12[s]);
                            s6[s] = fma2(G[s], R6, s6[s]);
                        }
                        const float2 p12 = up2(T12), p6 = up2(T6);
                        // dLJ/dd / d, grid units
                        const float lrad = fmaf(-12.f * (p12.x + p12.y), r6, 6.f * (p6.x + p6.y)) * (r6 * r2);
                        fs += lrad;
                        fz = fmaf(dz, lrad, fz);
                    }
#pragma unroll
                    for (int s = 0; s < 2 * NR; ++s) {
                        const float2 t12 = up2(s12[s]), t6 = up2(s6[s]);
                        ff_add(x12[2 * s].h, x12[2 * s].l, t12.x);
                        ff_add(x12[2 * s + 1].h, x12[2 * s + 1].l, t12.y);
                        ff_add(x6[2 * s].h, x6[2 * s].l, t6.x);
                        ff_add(x6[2 * s + 1].h, x6[2 * s + 1].l, t6.y);
                    }
                    ff_add(v[4].h, v[4].l, c.dxy2 < INFINITY ? c.dx * fs : 0.f);
                    ff_add(v[5].h, v[5].l, c.dxy2 < INFINITY ? c.dy * fs : 0.f);
                    ff_add(v[6].h, v[6].l, fz);
                }
            }
#pragma unroll
            for (int q = 0; q < 4 * NR; ++q) {
                if (q >= a.S) break;
                const float2 m = a.site[(int64_t)i * a.smax + q];
                const float2 ab = make_float2(up2(A[q / 2]).x, up2(A[q / 2]).y), bb = up2(B[q / 2]);
                const float Aq = q & 1 ? ab.y : ab.x, Bq = q & 1 ? bb.y : bb.x;
                ffs_add(v[7], ffs_mul(12.f * Aq * m.x, x12[q]));
                ffs_add(v[7], ffs_mul(-6.f * Bq * m.x, x6[q]));
                ffs_add(v[8], ffs_mul(Aq * m.y, x12[q]));
                ffs_add(v[8], ffs_mul(-Bq * m.y, x6[q]));
            }
        }
#pragma unroll
        for (int q = 0; q < 9; ++q)
            for (int o = 16; o > 0; o >>= 1)
                ffs_add(v[q], FFs{__shfl_xor_sync(0xffffffffu, v[q].h, o), __shfl_xor_sync(0xffffffffu, v[q].l, o)});
        if (a.wpa > 1) {  // the warps of an atom, in warp order
            __syncthreads();
            if (lane == 0)
#pragma unroll
                for (int q = 0; q < 9; ++q) red[w][q] = v[q];
            __syncthreads();
            if (live && sub == 0 && lane < 9) {
                FFs r = red[w][lane];
                for (int k = 1; k < a.wpa; ++k) ffs_add(r, red[w + k][lane]);
                a.out[(int64_t)i * 9 + lane] = (double)r.h + (double)r.l;
            }
        } else if (live) {
            FFs r = v[0];
#pragma unroll
            for (int q = 1; q < 9; ++q)
                if (lane == q) r = v[q];
            if (lane < 9) a.out[(int64_t)i * 9 + lane] = (double)r.h + (double)r.l;
        }
    }
}

template <bool FN>
void near_launch(const NearAdjArgs& a, int S, bool uni, int ctas, cudaStream_t st) {
    if (S <= 4) {
        if (uni) k_adj_near<1, true, FN><<<ctas, kNearT, 0, st>>>(a);
        else k_adj_near<1, false, FN><<<ctas, kNearT, 0, st>>>(a);
    } else {
        if (uni) k_adj_near<2, true, FN><<<ctas, kNearT, 0, st>>>(a);
        else k_adj_near<2, false, FN><<<ctas, kNearT, 0, st>>>(a);
    }
}

struct FinalArgs {
    int n, chunks;
    double h;
    const double* raw;       // [n][6]
    const double* part;      // [chunks][n][4]
    const double* near;      // [n][9]
    double *d_xyz, *d_q, *d_sigma, *d_eps;
};

// dL/dq = (dq_far + dq_near)/h; dL/dR = -q (G_far + G_near)/h^2 - dLJ/dR;
// signs: d(1/d)/dR_i = (r - R_i)/d^3 and (r - R_i) = h (grid index - U).
__global__ void k_adj_final(FinalArgs a) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.n) return;
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    for (int c = 0; c < a.chunks; ++c)
        for (int k = 0; k < 4; ++k) s[k] += a.part[((int64_t)c * a.n + i) * 4 + k];
    const double* nr = a.near + (int64_t)i * 9;
    const double q = a.raw[6 * i + 3];
    const double ih = 1.0 / a.h, ih2 = ih * ih;
    if (a.d_q) a.d_q[i] = (s[0] + nr[0]) * ih;
    if (a.d_xyz) {
        // far: sum (r-R) * (A1/d + ...)/d^2 -> q * that / h^2 (grid units: r-R = h dvec, 1/d^3 = 1/(h^3 d_g^3));
        // near erfc terms carry their own radial factor (dphi/dd / d, grid units) with dL/dR = -q (r-R) * rad
        for (int k = 0; k < 3; ++k)
            a.d_xyz[3 * i + k] = q * s[1 + k] * ih2 - q * nr[1 + k] * ih2 - nr[4 + k] * ih;
    }
    if (a.d_sigma) a.d_sigma[i] = nr[7];
    if (a.d_eps) a.d_eps[i] = nr[8];
}

}  // namespace

struct AdjointState {
    float4* w = nullptr;
    int64_t cap_w = 0;
    float4* gu4 = nullptr;
    int64_t cap_gu4 = 0;
    double* part = nullptr;
    int64_t cap_part = 0;
    double* near = nullptr;
    int64_t cap_near = 0;
    float2* site = nullptr;  // mixing derivatives per (atom, site)
    int64_t cap_site = 0;
    float4* tab = nullptr;   // short-range kernels (k_adj_near)
    double tab_key[4] = {0.0, 0.0, 0.0, -1.0};
};

AdjointState* adjoint_create() { return new AdjointState(); }

void adjoint_destroy(AdjointState* s) {
    if (!s) return;
    cudaFree(s->w);
    cudaFree(s->gu4);
    cudaFree(s->part);
    cudaFree(s->near);
    cudaFree(s->site);
    cudaFree(s->tab);
    delete s;
}

static rism_status aerr(std::string& err, cudaError_t e, const char* what) {
    err = std::string(what) + ": " + cudaGetErrorString(e);
    return e == cudaErrorMemoryAllocation ? RISM_E_NOMEM : RISM_E_CUDA;
}

// The cubic pieces of k_adj_near for the current smearing, screening, spacing and short-range radius.
static cudaError_t near_table(AdjointState* s, const GridD& g, const Phys& ph, cudaStream_t st) {
    const double key[4] = {ph.eta, g.h, ph.a, ph.rs};
    if (s->tab && std::memcmp(key, s->tab_key, sizeof key) == 0) return cudaSuccess;
    cudaError_t e;
    if ((e = alloc_once(s->tab, 4 * kAdjTab)) != cudaSuccess) return e;
    const double a = ph.a, dx = ph.rs / ph.eta / kAdjTab, tsp = 2.0 / std::sqrt(M_PI);
    // values and slopes in x at the nodes; H0'' = 4 a^2 H0 + (8 x/sqrt(pi)) e^{-x^2}
    auto node = [&](int k, double (&f)[4], double (&d)[4]) {
        const double x = k * dx, ex = std::exp(-x * x);
        const double em = std::exp(a * a - 2.0 * a * x) * std::erfc(x - a), ep = std::exp(a * a + 2.0 * a * x) * std::erfc(x + a);
        f[0] = std::erfc(x);
        d[0] = -tsp * ex;
        f[2] = em + ep;
        d[2] = 2.0 * a * (ep - em) - 2.0 * tsp * ex;
        f[1] = f[0] - x * d[0];
        d[1] = -2.0 * tsp * x * x * ex;
        f[3] = f[2] - x * d[2];
        d[3] = -x * (4.0 * a * a * f[2] + 4.0 * tsp * x * ex);
    };
    std::vector<float4> tab(4 * kAdjTab);
    for (int k = 0; k < kAdjTab; ++k) {
        double f0[4], d0[4], f1[4], d1[4];
        node(k, f0, d0);
        node(k + 1, f1, d1);
        for (int q = 0; q < 4; ++q)
            tab[4 * k + q] = make_float4((float)f0[q], (float)(d0[q] * dx),
                                         (float)(3.0 * (f1[q] - f0[q]) - dx * (2.0 * d0[q] + d1[q])),
                                         (float)(2.0 * (f0[q] - f1[q]) + dx * (d0[q] + d1[q])));
    }
    if ((e = upload(s->tab, tab.data(), sizeof(float4) * tab.size(), st)) != cudaSuccess) return e;
    std::memcpy(s->tab_key, key, sizeof key);
    return cudaSuccess;
}

rism_status adjoint_run(AdjointState* s, TreeState* tree, const DevTables& t, const GridD& g, const Phys& ph_,
                        const rism_options& o, const double* raw_dev, const double* sig_s, const double* eps_s,
                        const double* g_u, const double* g_c, const double* g_h, double* d_xyz, double* d_q,
                        double* d_sigma, double* d_eps, cudaStream_t st, std::string& err) {
    if (o.precision != RISM_PREC_FP32) {
        err = "the adjoint is implemented with FP32 pair terms (precision RISM_PREC_FP32)";
        return RISM_E_UNSUPPORTED;
    }
    // the short-range kernels end at (5 + a) eta for FP32 (3e-12 of the whole): a wider r_short does not stretch the pieces
    Phys ph = ph_;
    const bool pieces = ph.a <= kAdjPieceA;
    if (pieces) ph.rs = std::min(ph.rs, (5.0 + ph.a) * ph.eta);
    const int n = (int)t.n;
    if (n == 0) return RISM_OK;
    const int64_t M = (int64_t)g.nx * g.ny * g.nz;
    cudaError_t e;
    if ((e = grow(s->cap_w, M, buf(s->w, M))) != cudaSuccess) return aerr(err, e, "adjoint weights");
    const int seg_per_row = (g.nx + kRowT - 1) / kRowT;
    const int nseg = seg_per_row * g.ny * g.nz;
    const int ablocks = (n + kAT * kAPT - 1) / (kAT * kAPT);
    // enough CTAs to fill the GPU several times; at most one per row segment
    int chunks = (4 * sm_count() + ablocks - 1) / ablocks;
    chunks = max(1, min(chunks, min(nseg, 256)));
    const int tchunks = tree && o.method == RISM_METHOD_TREECODE ? tree_adjoint_chunks(n) : 0;
    const int64_t need_part = (int64_t)max(chunks, tchunks) * n * 4;
    if ((e = grow(s->cap_part, need_part, buf(s->part, need_part))) != cudaSuccess) return aerr(err, e, "adjoint partials");
    const int64_t need_near = (int64_t)n * 9, need_site = (int64_t)n * t.smax;
    if ((e = grow(s->cap_near, need_near, buf(s->near, need_near))) != cudaSuccess) return aerr(err, e, "adjoint near");
    if ((e = grow(s->cap_site, need_site, buf(s->site, need_site))) != cudaSuccess)
        return aerr(err, e, "adjoint site table");
    const int64_t need_gu4 = g_u ? M * ((ph.S + 3) / 4) : 0;
    if (g_u && (e = grow(s->cap_gu4, need_gu4, buf(s->gu4, need_gu4))) != cudaSuccess) return aerr(err, e, "adjoint G_u");
    WeightCoef wc;
    const double cf[3] = {ph.k_e, -ph.beta * ph.k_e, -ph.beta * ph.k_e / (2.0 * ph.eps_r)};
    for (int q = 0; q < 3; ++q)
        for (int k = 0; k < kMaxSites; ++k) {
            const double v = cf[q] * ph.qs[k];
            wc.h[q][k] = (float)v;
            wc.l[q][k] = (float)(v - (double)wc.h[q][k]);
        }
    wc.e2h = (float)(2.0 * ph.ea2);
    wc.e2l = (float)(2.0 * ph.ea2 - (double)wc.e2h);
    if (ph.S <= 2) k_adj_weights<2><<<8 * sm_count(), 256, 0, st>>>(M, ph.S, g_u, g_c, g_h, wc, s->w, s->gu4);
    else if (ph.S <= 4) k_adj_weights<4><<<8 * sm_count(), 256, 0, st>>>(M, ph.S, g_u, g_c, g_h, wc, s->w, s->gu4);
    else k_adj_weights<8><<<8 * sm_count(), 256, 0, st>>>(M, ph.S, g_u, g_c, g_h, wc, s->w, s->gu4);
    FarAdjArgs fa;
    fa.nx = g.nx;
    fa.ny = g.ny;
    fa.nz = g.nz;
    fa.n = n;
    fa.seg_per_row = seg_per_row;
    fa.nseg = nseg;
    fa.chunks = chunks;
    fa.kap_g = (float)(ph.kappa * g.h);
    fa.kap2 = (float)(-ph.kappa * g.h * 1.4426950408889634);
    fa.srcf = t.srcf;
    fa.w = s->w;
    fa.part = s->part;
    fa.err = t.err;
    fa.wlim = o.wait_limit;
    const bool dh = g_h && ph.kappa > 0.0;
    bool tree_far = false;
    if (tree && o.method == RISM_METHOD_TREECODE) {
        rism_status r = tree_adjoint_far(tree, t, g, ph, o, s->w, dh, s->part, tchunks, st, err, tree_far);
        if (r != RISM_OK) return r;
    }
    if (tree_far) {
        chunks = tchunks;  // written in original atom order
    } else {
        dim3 grid(ablocks, chunks);
        if (dh) k_adj_far<true><<<grid, kAT, 0, st>>>(fa);
        else k_adj_far<false><<<grid, kAT, 0, st>>>(fa);
    }
    if (pieces && (e = near_table(s, g, ph, st)) != cudaSuccess) return aerr(err, e, "adjoint kernel table");
    SiteLJ lj;
    for (int k = 0; k < kMaxSites; ++k) {
        lj.sig[k] = k < ph.S ? sig_s[k] : 0.0;
        lj.eps[k] = k < ph.S ? eps_s[k] : 0.0;
    }
    k_adj_sites<<<(int)(((int64_t)n * t.smax + 127) / 128), 128, 0, st>>>(n, ph.S, t.smax, raw_dev, lj, s->site);
    NearAdjArgs na;
    na.g = g;
    na.n = n;
    na.S = ph.S;
    na.smax = t.smax;
    na.srcf = t.srcf;
    na.ljf = t.ljf;
    na.site = s->site;
    na.w = s->w;
    na.gu4 = g_u ? s->gu4 : nullptr;
    na.order = (tree && o.method == RISM_METHOD_TREECODE) ? tree_atom_order(tree) : nullptr;
    na.tab = s->tab;
    na.tab_inv = (float)(kAdjTab / (ph.rs / g.h));
    na.xs = (float)(g.h / ph.eta);
    na.aa = (float)ph.a;
    na.rs = (float)(ph.rs / g.h);
    na.rs2 = (float)((ph.rs / g.h) * (ph.rs / g.h));
    na.out = s->near;
    // enough warps for 64 per SM: few atoms get several warps each
    na.wpa = 1;
    while (na.wpa < kNearT / 32 && (int64_t)n * na.wpa < 64 * (int64_t)sm_count()) na.wpa *= 2;
    const int nctas = (int)std::min<int64_t>(((int64_t)n * na.wpa + kNearT / 32 - 1) / (kNearT / 32), 4 * sm_count());
    const bool uni = o.lj_mode != RISM_LJ_TOL;
    if (pieces) near_launch<false>(na, ph.S, uni, nctas, st);
    else near_launch<true>(na, ph.S, uni, nctas, st);
    FinalArgs fin{n, chunks, g.h, raw_dev, s->part, s->near, d_xyz, d_q, d_sigma, d_eps};
    k_adj_final<<<(n + 255) / 256, 256, 0, st>>>(fin);
    if ((e = cudaGetLastError()) != cudaSuccess) return aerr(err, e, "adjoint kernels");
    return RISM_OK;
}

}  // namespace rism
