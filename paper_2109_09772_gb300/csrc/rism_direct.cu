// rism_direct.cu -- solute/solvent setup and the direct-sum evaluation kernels.
//
// The direct kernels evaluate, for every grid point of a CTA tile and every
// atom, the pair terms of the generic pair sum of Sec. 2.3, eq. (pot):
//   Phi1  = sum q/d                 (Coulomb, and the long-range part of eq. (dcf-r))
//   Phik  = sum q e^{-kappa d}/d    (long-range part of eq. (tcf-r))
//   Sc    = sum_{d<rs} q erfc(d/eta)/d
//   Sh    = sum_{d<rs} q e^{-x^2}[erfcx(x-a)+erfcx(x+a)]/d,  x = d/eta, a = kappa eta/2
//   LJ_s  = sum_{d<rc_is} A_is/d^12 - B_is/d^6                (Sec. 2.6)
// and assemble u = k_e q_s Phi1 + LJ_s, c = -beta k_e q_s (Phi1 - Sc),
// h = -(beta k_e q_s/(2 eps_r)) (2 e^{a^2} Phik - Sh).  The split
// erf = 1 - erfc and e^{a^2}[e^{-kd}erfc(a-x) - e^{kd}erfc(a+x)] =
// 2 e^{a^2} e^{-kd} - e^{-x^2}[erfcx(x-a) + erfcx(x+a)] is exact; the
// remainders Sc, Sh fall below 1e-16 relative beyond rs ~ 6 eta, which is the
// exact form of the far-field simplification eq. (tcfexp) of Sec. 2.4.2.
//
// Data movement: atoms are streamed through shared memory in tiles of T by
// bulk TMA copies (cp.async.bulk + mbarrier, double-buffered, bounded waits).
// A warp owns a compact block of 2P x 4 x 4 points, a thread P consecutive x
// points of it, and reads each atom (FP32: each pair of atoms) as a
// shared-memory broadcast.
#include <cmath>
#include <vector>

#include "rism_kernels.h"

namespace rism {

// ------------------------------------------------------------------ setup
__device__ double lj_u(double A, double B, double r) {
    double r2 = 1.0 / (r * r);
    double r6 = r2 * r2 * r2;
    return r6 * (A * r6 - B);
}

// Largest r with |A/r^12 - B/r^6| = tol (Sec. 2.6 per-pair cut-off), bisection.
__device__ double rcut_from_tol(double A, double B, double tol) {
    if (A <= 0.0 || B <= 0.0) return 0.0;
    double sig6 = A / B;                     // sigma^6
    double rmin = cbrt(sqrt(2.0 * sig6));    // 2^(1/6) sigma
    double eps = B * B / (4.0 * A);          // well depth
    double lo, hi;
    if (tol < eps) {
        lo = rmin;
        hi = rmin;
        for (int k = 0; k < 64 && fabs(lj_u(A, B, hi)) > tol; ++k) hi *= 2.0;
        for (int it = 0; it < 200; ++it) {
            double mid = 0.5 * (lo + hi);
            if (mid <= lo || mid >= hi) break;
            if (fabs(lj_u(A, B, mid)) > tol) lo = mid; else hi = mid;
        }
        return hi;
    }
    double sig = cbrt(sqrt(sig6));
    lo = 0.5 * sig;
    for (int k = 0; k < 64 && lj_u(A, B, lo) < tol; ++k) lo *= 0.5;
    hi = sig;
    for (int it = 0; it < 200; ++it) {
        double mid = 0.5 * (lo + hi);
        if (mid <= lo || mid >= hi) break;
        if (lj_u(A, B, mid) > tol) lo = mid; else hi = mid;
    }
    return hi;
}

struct SetupArgs {
    const double* raw;
    int64_t n;
    int S, smax;
    double sig_s[kMaxSites], eps_s[kMaxSites];
    int lj_mode;
    double lj_rcut, lj_tol;
    GridD g;
};

// One thread per (atom, site slot): the pair's Lorentz-Berthelot LJ terms (FP64 and FP32 grid units); the
// thread of slot 0 also writes the atom's position records.
__global__ void k_setup(SetupArgs a, Geo* geo, SrcF* srcf, LJd* ljd, LJf* ljf) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= a.n * a.smax) return;
    const int64_t i = t / a.smax;
    const int s = (int)(t - i * a.smax);
    const double* r = a.raw + 6 * i;
    if (s == 0) {
        const double x = r[0], y = r[1], z = r[2], q = r[3];
        geo[i] = Geo{x, y, z, q};
        const double ih = 1.0 / a.g.h;
        srcf[i] = make_srcf((x - a.g.ox) * ih, (y - a.g.oy) * ih, (z - a.g.oz) * ih, q);
    }
    LJd d{0.0, 0.0, 0.0, 0.0};
    LJf f{0.f, 0.f, 0.f, 0.f};
    if (s < a.S) {
        const double sg = r[4], ep = r[5];
        const double h2 = a.g.h * a.g.h, h6 = h2 * h2 * h2;
        double sig = 0.5 * (sg + a.sig_s[s]);      // Lorentz
        double eps = sqrt(ep * a.eps_s[s]);        // Berthelot
        double s2 = sig * sig, s6 = s2 * s2 * s2;
        double A = 4.0 * eps * s6 * s6, B = 4.0 * eps * s6;
        double rc2;
        if (a.lj_mode == RISM_LJ_RCUT) rc2 = a.lj_rcut * a.lj_rcut;
        else if (a.lj_mode == RISM_LJ_TOL) { double rc = rcut_from_tol(A, B, a.lj_tol); rc2 = rc * rc; }
        else rc2 = INFINITY;
        d = LJd{A, B, rc2, 0.0};
        f = LJf{(float)(A / (h6 * h6)), (float)(B / h6), (float)(rc2 / h2), 0.f};
    }
    ljd[t] = d;
    ljf[t] = f;
}

cudaError_t launch_setup(const double* raw, int64_t n, int S, int smax, const double* sig_s, const double* eps_s,
                         int lj_mode, double lj_rcut, double lj_tol, const GridD& g, DevTables& t,
                         cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    SetupArgs a;
    a.raw = raw;
    a.n = n;
    a.S = S;
    a.smax = smax;
    for (int s = 0; s < kMaxSites; ++s) {
        a.sig_s[s] = s < S ? sig_s[s] : 0.0;
        a.eps_s[s] = s < S ? eps_s[s] : 0.0;
    }
    a.lj_mode = lj_mode;
    a.lj_rcut = lj_rcut;
    a.lj_tol = lj_tol;
    a.g = g;
    const int nb = (int)((n * smax + 127) / 128);
    k_setup<<<nb, 128, 0, st>>>(a, t.geo, t.srcf, t.ljd, t.ljf);
    return cudaGetLastError();
}

// I_s = sum_i 4 pi (A/(9 rc^9) - B/(3 rc^3)); one CTA per site, fixed-order reduction.
constexpr int kTailThreads = 1024;
__global__ void __launch_bounds__(kTailThreads) k_lj_tail(const LJd* lj, int64_t n, int smax, double* out) {
    constexpr int NT = kTailThreads;
    __shared__ double red[NT];
    int s = blockIdx.x;
    double acc = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += NT) {
        LJd p = lj[i * smax + s];
        if (isfinite(p.rc2) && p.rc2 > 0.0) {
            // 4 pi (A / (9 rc^9) - B / (3 rc^3)) with r3 = rc^-3 from one reciprocal square root
            const double ri = rsqrt(p.rc2), r3 = ri * ri * ri;
            acc += 4.0 * M_PI * r3 * (p.A * (1.0 / 9.0) * r3 * r3 - p.B * (1.0 / 3.0));
        }
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int w = NT / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[s] = red[0];
}

cudaError_t launch_lj_tail(const DevTables& t, int S, double* dev_out, cudaStream_t st) {
    k_lj_tail<<<S, kTailThreads, 0, st>>>(t.ljd, t.n, t.smax, dev_out);
    return cudaGetLastError();
}

// In grid units; F_h = e^{a^2-2ax} erfc(x-a) + e^{a^2+2ax} erfc(x+a), x = d h / eta, a = kappa eta / 2, with the
// derivatives dF_c/dx = -2/sqrt(pi) e^{-x^2} and dF_h/dx = -2a e^{a^2-2ax} erfc(x-a) + 2a e^{a^2+2ax} erfc(x+a) -
// 4/sqrt(pi) e^{-x^2}; built in FP64.
void short_range_table(const Phys& ph, double h, float4* tab) {
    const double sx = h / ph.eta, a = ph.a, D = ph.rs / h / kNTab;
    const double tsp = 2.0 / std::sqrt(3.14159265358979323846);
    std::vector<double> fc(kNTab + 1), gc(kNTab + 1), fh(kNTab + 1), gh(kNTab + 1);
    for (int k = 0; k <= kNTab; ++k) {
        const double x = k * D * sx, ex = std::exp(-x * x);
        const double em = std::exp(a * a - 2.0 * a * x), ep = std::exp(a * a + 2.0 * a * x);
        const double cm = std::erfc(x - a), cp = std::erfc(x + a);
        fc[k] = std::erfc(x);
        gc[k] = -tsp * ex * sx * D;  // derivative per segment length
        fh[k] = em * cm + ep * cp;
        gh[k] = (-2.0 * a * em * cm + 2.0 * a * ep * cp - 2.0 * tsp * ex) * sx * D;
    }
    for (int k = 0; k < kNTab; ++k) {
        auto c2 = [&](const std::vector<double>& f, const std::vector<double>& g) {
            return (float)(3.0 * (f[k + 1] - f[k]) - 2.0 * g[k] - g[k + 1]);
        };
        auto c3 = [&](const std::vector<double>& f, const std::vector<double>& g) {
            return (float)(2.0 * (f[k] - f[k + 1]) + g[k] + g[k + 1]);
        };
        tab[2 * k] = make_float4((float)fc[k], (float)fh[k], (float)gc[k], (float)gh[k]);
        tab[2 * k + 1] = make_float4(c2(fc, gc), c2(fh, gh), c3(fc, gc), c3(fh, gh));
    }
}

// Taylor pieces: in t = (u - middle) with u = d kTab64 / r_short, |t| <= 1/2.  With E = e^{-x^2} and H_k the Hermite
// polynomials, E^(k) = (-1)^k H_k E; F_c' = -(2/sqrt(pi)) E; and F_h = G- + G+ with G-+ = e^{a^2 -+ 2ax} erfc(x -+ a),
// G-+' = -+ 2a G-+ - (2/sqrt(pi)) E, differentiated term by term.  Eight terms leave less than 1e-16 (the segments are
// 0.0234 eta wide at r_short = 6 eta): absolute, where the library's functions are good to an ulp of their value.  What
// they are subtracted from (q/d and its screened form) has that absolute error already.
void short_range_table64(const Phys& ph, double* tab) {
    const double a = ph.a, dx = ph.rs / ph.eta / kTab64, tsp = 2.0 / std::sqrt(3.14159265358979323846);
    for (int s = 0; s < kTab64; ++s) {
        const double x = (s + 0.5) * dx;
        double E[kTerm64], hm = 0.0, h = 1.0;  // E^(k)
        for (int k = 0; k < kTerm64; ++k) {
            E[k] = (k & 1 ? -h : h) * std::exp(-x * x);
            const double nx = 2.0 * x * h - 2.0 * k * hm;
            hm = h;
            h = nx;
        }
        double gm = std::exp(a * a - 2.0 * a * x) * std::erfc(x - a), gp = std::exp(a * a + 2.0 * a * x) * std::erfc(x + a);
        double c = std::erfc(x), f = 1.0;  // f = dx^k / k!
        for (int k = 0; k < kTerm64; ++k) {
            tab[s * kTerm64 + k] = c * f;
            tab[(kTab64 + s) * kTerm64 + k] = (gm + gp) * f;
            c = -tsp * E[k];
            gm = -2.0 * a * gm - tsp * E[k];
            gp = 2.0 * a * gp - tsp * E[k];
            f *= dx / (k + 1);
        }
    }
    for (int j = 0; j < 256; ++j) {  // 2^(j/256) as a double and what its rounding left (long double's extra digits)
        const long double v = std::exp2((long double)j / 256.0L);
        double* o = tab + 2 * kTab64 * kTerm64 + 2 * j;
        o[0] = (double)v;
        o[1] = (double)(v - (long double)o[0]);
    }
}

// ------------------------------------------------------- common epilogue
template <int P>
__device__ __forceinline__ void store_strip(double* base, int i0, int nx, const double (&v)[P], bool vec_ok) {
    if (P % 2 == 0 && vec_ok && i0 + P <= nx) {
#pragma unroll
        for (int p = 0; p + 1 < P; p += 2)
            __stcs(reinterpret_cast<double2*>(base + i0 + p), make_double2(v[p], v[p + 1]));
    } else {
#pragma unroll
        for (int p = 0; p < P; ++p)
            if (i0 + p < nx) __stcs(base + i0 + p, v[p]);
    }
}

constexpr int kDirectT = 64;  // atoms per tile (two ballots)

// ------------------------------------------------------------ FP64 direct
// The FP64 pipe of this part is slow (1.7 multiply-adds per clock per SM), so what need not run on it does not:
// comparisons of non-negative doubles order their bit patterns on the integer pipe.
__device__ __forceinline__ bool lt_bits(double a, double b) { return __double_as_longlong(a) < __double_as_longlong(b); }

// 1/sqrt(d2) (0 for d2 = 0): the single-precision approximation of the leading bits, moved to and from FP32 by their bit
// patterns, and one step of Halley's iteration: with h = 1 - d2 y^2, y + y h (1/2 + 3/8 h) leaves 5/16 h^3, below 2^-64;
// five FP64 operations.  Exponents outside FP32's range take the library function.
__device__ __noinline__ double rsqrt64_slow(double d2) { return d2 > 0.0 ? rsqrt(d2) : 0.0; }
__device__ __forceinline__ double rsqrt64(double d2) {
    const uint32_t hi = (uint32_t)__double2hiint(d2), lo = (uint32_t)__double2loint(d2);
    if ((hi >> 20) - 910u > 220u) return rsqrt64_slow(d2);
    const uint32_t f = __float_as_uint(rsqrt_approx(__uint_as_float(((hi - 0x38000000u) << 3) | (lo >> 29))));
    const double y = __hiloint2double((int)((f >> 3) + 0x38000000u), (int)(f << 29));
    const double h = fma(-(d2 * y), y, 1.0);
    return fma(y * h, fma(h, 0.375, 0.5), y);
}

constexpr double kRound64 = 6755399441055744.0;  // 1.5 2^52: adding it leaves round(v) in the low word

// F at u = d kTab64 / r_short (below kTab64) from a table of short_range_table64.
__device__ __forceinline__ double piece64(const double* tab, double u) {
    const double m = (u - 0.5) + kRound64;  // the segment: round(u - 1/2)
    const int it = min(__double2loint(m), kTab64 - 1);
    const double t = (u - 0.5) - (it == __double2loint(m) ? m - kRound64 : (double)(kTab64 - 1));
    const double2* c = reinterpret_cast<const double2*>(tab + it * kTerm64);
    const double2 c67 = c[3], c45 = c[2], c23 = c[1], c01 = c[0];
    return fma(fma(fma(fma(fma(fma(fma(c67.y, t, c67.x), t, c45.y), t, c45.x), t, c23.y), t, c23.x), t, c01.y), t, c01.x);
}

// e^{-kappa d} from c = -256 kappa log2(e): with N = round(c d) and f = c d - N, 2^(N/256) as a pair from the table and
// the powers of two, e^{f ln2/256} from four terms (below 4e-17); ten FP64 operations with the distance.
__device__ __forceinline__ double exp64(const double2* pow2, double d, double c) {
    const double m = fma(d, c, kRound64);
    const int n = __double2loint(m);
    const double f = fma(d, c, -(m - kRound64));
    constexpr double L = 0.69314718055994530942 / 256.0;
    const double p = fma(fma(fma(L * L * L * L / 24.0, f, L * L * L / 6.0), f, L * L / 2.0), f, L);
    const double2 t = pow2[n & 255];
    const double e = t.x + fma(t.x, f * p, t.y);
    return n < -261000 || d * c < -1e9 ? 0.0 : __hiloint2double(__double2hiint(e) + (n >> 8) * (1 << 20), __double2loint(e));
}

// Launch shape: four warps of 8 x 4 x 4 points (P = 4) or 2 x 4 x 4 (P = 1), two by two along x and y; T atoms per tile.
// A warp's points are compact so that few warps take an atom's erfc remainders for the sake of a few of their points.
// Bound by the FP64 pipe.  200 atoms on 64^3, two sites, no cut-off: 2.4 ms (4.2 ms with the library's reciprocal
// square root and erfc, a division per pair, comparisons in FP64 and warps of 32 x 4 x 1 points).
template <int SM, int P, int T, bool DU, bool DH>
__global__ void __launch_bounds__(128) k_direct64(GridD g, Phys ph, const Geo* __restrict__ geo,
                                                  const LJd* __restrict__ lj, int64_t n,
                                                  const double* __restrict__ sr, Outputs o, DevErr* err,
                                                  long long wlim, int dbg) {
    extern __shared__ __align__(16) unsigned char smem[];
    Geo* sgeo = reinterpret_cast<Geo*>(smem);
    LJd* slj = reinterpret_cast<LJd*>(smem + 2 * T * sizeof(Geo));
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + 2 * T * sizeof(Geo) + 2 * T * SM * sizeof(LJd));
    double* tab = reinterpret_cast<double*>(bar + 2);  // [kLen64]
    const double2* pow2 = reinterpret_cast<const double2*>(tab + 2 * kTab64 * kTerm64);

    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    if (sr)
        for (int q = tid; q < kLen64; q += 128) tab[q] = sr[q];
    const double srinv = kTab64 / ph.rs, kexp = -256.0 * 1.4426950408889634074 * ph.kappa;
    const int i0 = (blockIdx.x * 2 + (w & 1)) * 2 * P + (lane & 1) * P;
    const int j = (blockIdx.y * 2 + (w >> 1)) * 4 + ((lane >> 1) & 3), k = blockIdx.z * 4 + (lane >> 3);
    double gx[P];
#pragma unroll
    for (int p = 0; p < P; ++p) gx[p] = g.ox + g.h * (double)(i0 + p);
    const double gy = g.oy + g.h * (double)j, gz = g.oz + g.h * (double)k;
    const double rs2 = ph.rs * ph.rs, ieta = 1.0 / ph.eta, a = ph.a, kap = ph.kappa;
    const bool DC = o.c != nullptr;

    double f1[P], fk[P], sc[P], sh[P], lj_[P][SM];
#pragma unroll
    for (int p = 0; p < P; ++p) {
        f1[p] = fk[p] = sc[p] = sh[p] = 0.0;
#pragma unroll
        for (int s = 0; s < SM; ++s) lj_[p][s] = 0.0;
    }
    unsigned hit = 0u;

    const int ntiles = (int)((n + T - 1) / T);
    if (tid == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        mbar_fence_init();
    }
    __syncthreads();
    auto issue = [&](int t) {
        int st = t & 1;
        int cnt = (int)min((int64_t)T, n - (int64_t)t * T);
        uint32_t b1 = cnt * sizeof(Geo), b2 = cnt * SM * sizeof(LJd);
        mbar_expect_tx(&bar[st], b1 + b2);
        bulk_g2s(sgeo + st * T, geo + (int64_t)t * T, b1, &bar[st]);
        bulk_g2s(slj + st * T * SM, lj + (int64_t)t * T * SM, b2, &bar[st]);
    };
    if (tid == 0) {
        // debug hook: without the first copy its wait can only run out
        if (ntiles > 0 && !(dbg & 1)) issue(0);
        if (ntiles > 1) issue(1);
    }
    for (int t = 0; t < ntiles; ++t) {
        const int st = t & 1;
        bool ok = mbar_wait_bounded(&bar[st], (t >> 1) & 1, wlim);
        if (__syncthreads_or(!ok)) {
            if (tid == 0) {
                report_error(err, DEV_TIMEOUT, WHERE_DIRECT);
                // drain the copies still in flight (bounded) before the CTA exits
                for (int u2 = t; u2 < min(t + 2, ntiles); ++u2) mbar_wait_bounded(&bar[u2 & 1], (u2 >> 1) & 1, wlim);
            }
            return;
        }
        const int cnt = (int)min((int64_t)T, n - (int64_t)t * T);
        const Geo* G = sgeo + st * T;
        const LJd* L = slj + st * T * SM;
        for (int aa = 0; aa < cnt; ++aa) {
            const Geo A = G[aa];
            const double dy = gy - A.y, dz = gz - A.z;
            const double dyz2 = dy * dy + dz * dz;
#pragma unroll
            for (int p = 0; p < P; ++p) {
                const double dx = gx[p] - A.x;
                const double d2 = fma(dx, dx, dyz2);
                const double ri = rsqrt64(d2);
                const double qr = A.q * ri;
                f1[p] += qr;
                const double d = d2 * ri;
                if (DH) fk[p] += qr * (sr ? exp64(pow2, d, kexp) : exp(-kap * d));
                if (lt_bits(d2, rs2)) {
                    if (__double_as_longlong(d2) != 0ll && sr) {
                        if (DC) sc[p] += qr * piece64(tab, d * srinv);
                        if (DH) sh[p] += qr * piece64(tab + kTab64 * kTerm64, d * srinv);
                    } else if (__double_as_longlong(d2) != 0ll) {
                        const double x = d * ieta;
                        if (DC) sc[p] += qr * erfc(x);
                        if (DH) sh[p] += qr * exp(-x * x) * (erfcx(x - a) + erfcx(x + a));
                    } else {
                        hit |= 1u << p;
                        if (DC) sc[p] -= A.q * ph.phi_c0;
                        if (DH) sh[p] -= A.q * ph.phi_h0;
                    }
                }
                if (DU) {
                    long long rc = 0ll;  // the largest cut-off of the atom's sites
#pragma unroll
                    for (int s = 0; s < SM; ++s) rc = max(rc, __double_as_longlong(L[aa * SM + s].rc2));
                    if (__double_as_longlong(d2) < rc) {
                        // 1/d^2 from the square of the reciprocal root with the residual made up: three operations
                        const double y2 = ri * ri, r2i = fma(y2, fma(-d2, y2, 1.0), y2);
                        const double r6 = r2i * r2i * r2i;
#pragma unroll
                        for (int s = 0; s < SM; ++s) {
                            const LJd l = L[aa * SM + s];
                            if (lt_bits(d2, l.rc2)) lj_[p][s] += r6 * (l.A * r6 - l.B);
                        }
                    }
                }
            }
        }
        __syncthreads();
        if (tid == 0 && t + 2 < ntiles) issue(t + 2);
    }
    if (j >= g.ny || k >= g.nz || i0 >= g.nx) return;
    const int64_t plane = (int64_t)g.nx * g.ny * g.nz;
    const int64_t row = ((int64_t)k * g.ny + j) * g.nx;
    const bool vec_ok = P > 1 && (g.nx & 1) == 0;
    const double cu0 = ph.k_e, cc0 = -ph.beta * ph.k_e, ch0 = -ph.beta * ph.k_e / (2.0 * ph.eps_r);
#pragma unroll
    for (int s = 0; s < SM; ++s) {
        if (s >= ph.S) break;
        const double qs = ph.qs[s];
        double v[P];
        if (DU) {
#pragma unroll
            for (int p = 0; p < P; ++p) v[p] = (hit >> p & 1u) ? INFINITY : cu0 * qs * f1[p] + lj_[p][s];
            store_strip<P>(o.u + s * plane + row, i0, g.nx, v, vec_ok);
        }
        if (DC) {
#pragma unroll
            for (int p = 0; p < P; ++p) v[p] = cc0 * qs * (f1[p] - sc[p]);
            store_strip<P>(o.c + s * plane + row, i0, g.nx, v, vec_ok);
        }
        if (DH) {
#pragma unroll
            for (int p = 0; p < P; ++p) v[p] = ch0 * qs * (2.0 * ph.ea2 * fk[p] - sh[p]);
            store_strip<P>(o.h + s * plane + row, i0, g.nx, v, vec_ok);
        }
    }
}

// ------------------------------------------------------------ FP32 direct
// Pair terms in FP32 from float-float grid-unit source positions (SrcF): the
// grid coordinates are exact integers, so dx = (i - xh) - xl is exact to half
// an ulp of dx for every nearby atom.  Per-tile FP32 partial sums are folded
// into float-float totals (TwoSum), which carry ~48 bits.
//
// A warp owns a block of 2P x 4 x 4 points (P consecutive x points per lane), a CTA two by two of them.  Per tile of
// atoms a warp takes the long-range sums of all of them, two sources per instruction, and then only the atoms within
// the short-range radius or their largest LJ cut-off of its block, listed by ballots, for the LJ terms and the erfc
// remainders (a few in a hundred of a solute's atoms).

// Sources 2l and 2l + 1 of a tile, field by field (two-wide operands); an odd count is padded with a zero charge 10^6
// grid units away, whose terms are exactly zero.
struct DirRec {
    float4 x;  // xh0, xh1, xl0, xl1
    float4 y, z;
    float4 q;  // q0, q1, 0, 0
};

// The long-range sums of one tile at P points: per pair dx = (x - x_hi) - x_lo, d2, r = rsqrt(d2), q r, and with DH
// the screening factor by ex2.  ON: some source of the tile sits on a lattice point; d2 = 0 adds nothing here.
template <int P, bool DH, bool ON>
__device__ __forceinline__ void direct_far(const DirRec* rec, int np, const f32x2 (&GX)[P], f32x2 FY, f32x2 FZ, f32x2 K2,
                                           f32x2 (&P1)[P], f32x2 (&PK)[P]) {
#pragma unroll 2
    for (int l = 0; l < np; ++l) {
        const ulonglong2 X = *reinterpret_cast<const ulonglong2*>(&rec[l].x);
        const ulonglong2 Y = *reinterpret_cast<const ulonglong2*>(&rec[l].y);
        const ulonglong2 Z = *reinterpret_cast<const ulonglong2*>(&rec[l].z);
        const f32x2 Q = *reinterpret_cast<const f32x2*>(&rec[l].q);
        const f32x2 DY = sub2(sub2(FY, Y.x), Y.y);
        const f32x2 DZ = sub2(sub2(FZ, Z.x), Z.y);
        const f32x2 DYZ = fma2(DY, DY, mul2(DZ, DZ));
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const f32x2 DX = sub2(sub2(GX[p], X.x), X.y);
            const f32x2 D2 = fma2(DX, DX, DYZ);
            const float2 d2 = up2(D2);
            float r0 = rsqrt_approx(d2.x), r1 = rsqrt_approx(d2.y);
            if (ON) {
                r0 = d2.x > 0.f ? r0 : 0.f;
                r1 = d2.y > 0.f ? r1 : 0.f;
            }
            const f32x2 RI = pk2(r0, r1);
            const f32x2 QR = mul2(Q, RI);
            P1[p] = add2(P1[p], QR);
            if (DH) {
                const float2 e = up2(mul2(K2, mul2(D2, RI)));
                PK[p] = fma2(QR, pk2(ex2_approx(e.x), ex2_approx(e.y)), PK[p]);
            }
        }
    }
}

// Bound by the special-function pipe (a reciprocal square root and an exponential per pair).  2,000 atoms on 128^3, 4
// sites: 2.1 ms, of which the long-range sums are 1.25 ms at the pipe's rate; 5.8 ms when every pair also took a
// reciprocal, its sites' cut-off tests and a divergent branch to the remainders, in scalar instructions.
template <int SM, int P, bool DU, bool DH>
__global__ void __launch_bounds__(128, SM > 4 ? 2 : (P > 2 ? 3 : 4))
    k_direct32(GridD g, Phys ph, const SrcF* __restrict__ srcf, const LJf* __restrict__ lj, int64_t n,
               const float4* __restrict__ sr, float sr_inv, Outputs o, DevErr* err, long long wlim, int dbg) {
    constexpr int T = kDirectT;
    extern __shared__ __align__(16) unsigned char smem[];
    SrcF* ssrc = reinterpret_cast<SrcF*>(smem);                                   // [2][T]
    LJf* slj = reinterpret_cast<LJf*>(smem + 2 * T * sizeof(SrcF));               // [2][T][SM]
    DirRec* rec = reinterpret_cast<DirRec*>(slj + 2 * T * SM);                    // [T / 2]
    uint64_t* bar = reinterpret_cast<uint64_t*>(rec + T / 2);                     // [2]
    int* list = reinterpret_cast<int*>(bar + 2);                                   // [4][T]
    float4* tab = reinterpret_cast<float4*>(list + 4 * T);                         // [2 kNTab]

    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int bx = (blockIdx.x * 2 + (w & 1)) * 2 * P, by = (blockIdx.y * 2 + (w >> 1)) * 4, bz = blockIdx.z * 4;
    const int i0 = bx + (lane & 1) * P, j = by + ((lane >> 1) & 3), k = bz + (lane >> 3);
    f32x2 GX[P];
    float gx[P];
#pragma unroll
    for (int p = 0; p < P; ++p) {
        gx[p] = (float)(i0 + p);
        GX[p] = pk2(gx[p], gx[p]);
    }
    const float fy = (float)j, fz = (float)k;
    const f32x2 FY = pk2(fy, fy), FZ = pk2(fz, fz);
    const float wlo[3] = {(float)bx, (float)by, (float)bz};
    const float whi[3] = {(float)(bx + 2 * P - 1), (float)(by + 3), (float)(bz + 3)};
    const float rs2 = (float)((ph.rs / g.h) * (ph.rs / g.h));
    const float xs = (float)(g.h / ph.eta);                            // x = d_grid * xs
    const float kap2 = (float)(-ph.kappa * g.h * 1.4426950408889634);  // e^{-kappa d} = 2^(kap2 d_grid)
    const f32x2 K2 = pk2(kap2, kap2);
    const float a = (float)ph.a;
    const float c0h = (float)(ph.phi_c0 * g.h), h0h = (float)(ph.phi_h0 * g.h);
    const bool DC = o.c != nullptr;

    float f1h[P], f1l[P], fkh[P], fkl[P], sch[P], scl[P], shh[P], shl[P], ljh[P][SM], ljl[P][SM];
#pragma unroll
    for (int p = 0; p < P; ++p) {
        f1h[p] = f1l[p] = fkh[p] = fkl[p] = sch[p] = scl[p] = shh[p] = shl[p] = 0.f;
#pragma unroll
        for (int s = 0; s < SM; ++s) ljh[p][s] = ljl[p][s] = 0.f;
    }
    unsigned hit = 0u;

    const int ntiles = (int)((n + T - 1) / T);
    if (sr)
        for (int q = tid; q < 2 * kNTab; q += 128) tab[q] = sr[q];
    if (tid == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        mbar_fence_init();
    }
    __syncthreads();
    auto issue = [&](int t) {
        int st = t & 1;
        int cnt = (int)min((int64_t)T, n - (int64_t)t * T);
        uint32_t b1 = cnt * sizeof(SrcF), b2 = cnt * SM * sizeof(LJf);
        mbar_expect_tx(&bar[st], b1 + b2);
        bulk_g2s(ssrc + st * T, srcf + (int64_t)t * T, b1, &bar[st]);
        bulk_g2s(slj + st * T * SM, lj + (int64_t)t * T * SM, b2, &bar[st]);
    };
    if (tid == 0) {
        // debug hook: without the first copy its wait can only run out
        if (ntiles > 0 && !(dbg & 1)) issue(0);
        if (ntiles > 1) issue(1);
    }
    for (int t = 0; t < ntiles; ++t) {
        const int st = t & 1;
        bool ok = mbar_wait_bounded(&bar[st], (t >> 1) & 1, wlim);
        if (__syncthreads_or(!ok)) {
            if (tid == 0) {
                report_error(err, DEV_TIMEOUT, WHERE_DIRECT);
                for (int u2 = t; u2 < min(t + 2, ntiles); ++u2) mbar_wait_bounded(&bar[u2 & 1], (u2 >> 1) & 1, wlim);
            }
            return;
        }
        const int cnt = (int)min((int64_t)T, n - (int64_t)t * T);
        const SrcF* Sx = ssrc + st * T;
        const LJf* L = slj + st * T * SM;
        if (tid < T / 2) {  // the pair records of the tile
            const int s0 = 2 * tid, s1 = s0 + 1;
            float4 a0 = make_float4(1e6f, 1e6f, 1e6f, 0.f), a1 = make_float4(0.f, 0.f, 0.f, 0.f), b0 = a0, b1 = a1;
            if (s0 < cnt) {
                a0 = *reinterpret_cast<const float4*>(&Sx[s0].xh);
                a1 = *reinterpret_cast<const float4*>(&Sx[s0].xl);
            }
            if (s1 < cnt) {
                b0 = *reinterpret_cast<const float4*>(&Sx[s1].xh);
                b1 = *reinterpret_cast<const float4*>(&Sx[s1].xl);
            }
            rec[tid].x = make_float4(a0.x, b0.x, a1.x, b1.x);
            rec[tid].y = make_float4(a0.y, b0.y, a1.y, b1.y);
            rec[tid].z = make_float4(a0.z, b0.z, a1.z, b1.z);
            rec[tid].q = make_float4(a0.w, b0.w, 0.f, 0.f);
        }
        // the atoms that reach the warp's block: within r_short or the largest cut-off of their sites (0.01 grid units
        // of slack for the position rounded to its high part)
        auto reach = [&](int i) {
            if (i >= cnt) return false;
            const float4 c = *reinterpret_cast<const float4*>(&Sx[i].xh);
            float r2 = rs2;
            if (DU)
#pragma unroll
                for (int s = 0; s < SM; ++s) r2 = fmaxf(r2, L[i * SM + s].rc2);
            const float qx = fmaxf(0.f, fmaxf(wlo[0] - c.x, c.x - whi[0]));
            const float qy = fmaxf(0.f, fmaxf(wlo[1] - c.y, c.y - whi[1]));
            const float qz = fmaxf(0.f, fmaxf(wlo[2] - c.z, c.z - whi[2]));
            const float lim = sqrtf(r2) + 0.01f;
            return fmaf(qx, qx, fmaf(qy, qy, qz * qz)) < lim * lim;
        };
        const bool k0 = reach(lane), k1 = reach(lane + 32);
        const bool mine = (lane < cnt && Sx[lane].on_grid != 0.f) || (lane + 32 < cnt && Sx[lane + 32].on_grid != 0.f);
        const bool on = __any_sync(0xffffffffu, mine);
        const unsigned m0 = __ballot_sync(0xffffffffu, k0), m1 = __ballot_sync(0xffffffffu, k1);
        const unsigned lt = (1u << lane) - 1u;
        int* wl = list + w * T;
        const int near = __popc(m0) + __popc(m1);
        if (k0) wl[__popc(m0 & lt)] = lane;
        if (k1) wl[__popc(m0) + __popc(m1 & lt)] = lane + 32;
        __syncthreads();  // the records and the list
        {
            f32x2 P1[P], PK[P];
#pragma unroll
            for (int p = 0; p < P; ++p) P1[p] = PK[p] = 0ull;
            const int np = (cnt + 1) >> 1;
            if (on) direct_far<P, DH, true>(rec, np, GX, FY, FZ, K2, P1, PK);
            else direct_far<P, DH, false>(rec, np, GX, FY, FZ, K2, P1, PK);
#pragma unroll
            for (int p = 0; p < P; ++p) {
                const float2 s1 = up2(P1[p]);
                ff_add(f1h[p], f1l[p], s1.x + s1.y);
                if (DH) {
                    const float2 sk = up2(PK[p]);
                    ff_add(fkh[p], fkl[p], sk.x + sk.y);
                }
            }
        }
        if (near > 0) {
            f32x2 plj[P / 2][SM];  // two points per register pair
#pragma unroll
            for (int p = 0; p < P / 2; ++p)
#pragma unroll
                for (int s = 0; s < SM; ++s) plj[p][s] = 0ull;
            for (int q = 0; q < near; ++q) {
                const int aa = wl[q];
                const float4 g0 = *reinterpret_cast<const float4*>(&Sx[aa].xh);
                const float4 g1 = *reinterpret_cast<const float4*>(&Sx[aa].xl);
                const float dy = (fy - g0.y) - g1.y;
                const float dz = (fz - g0.z) - g1.z;
                const float dyz2 = fmaf(dy, dy, dz * dz);
                float d2[P];
#pragma unroll
                for (int p = 0; p < P; ++p) {
                    const float dx = (gx[p] - g0.x) - g1.x;
                    d2[p] = fmaf(dx, dx, dyz2);
                }
                if (DU) {
#pragma unroll
                    for (int p = 0; p < P / 2; ++p) {
                        const float r0 = rcp_approx(d2[2 * p]), r1 = rcp_approx(d2[2 * p + 1]);
                        const float a6 = r0 * r0 * r0, b6 = r1 * r1 * r1;
#pragma unroll
                        for (int s = 0; s < SM; ++s) {
                            const float4 l = *reinterpret_cast<const float4*>(&L[aa * SM + s]);
                            // a point outside the cut-off adds +0
                            const f32x2 R6 = pk2(d2[2 * p] < l.z ? a6 : 0.f, d2[2 * p + 1] < l.z ? b6 : 0.f);
                            plj[p][s] = fma2(R6, fma2(pk2(l.x, l.x), R6, pk2(-l.y, -l.y)), plj[p][s]);
                        }
                    }
                }
                float dmin = d2[0];
#pragma unroll
                for (int p = 1; p < P; ++p) dmin = fminf(dmin, d2[p]);
                if (dmin < rs2) {
#pragma unroll
                    for (int p = 0; p < P; ++p) {
                        if (d2[p] >= rs2) continue;
                        if (d2[p] > 0.f) {
                            const float ri = rsqrt_approx(d2[p]), qr = g0.w * ri;
                            if (sr) {
                                const float2 f = up2(short_range(tab, d2[p] * ri * sr_inv));
                                if (DC) ff_add(sch[p], scl[p], qr * f.x);
                                if (DH) ff_add(shh[p], shl[p], qr * f.y);
                            } else {
                                const float x = d2[p] * ri * xs;
                                if (DC) ff_add(sch[p], scl[p], qr * erfcf(x));
                                if (DH) ff_add(shh[p], shl[p], qr * (__expf(-x * x) * (erfcxf(x - a) + erfcxf(x + a))));
                            }
                        } else {
                            hit |= 1u << p;
                            if (DC) ff_add(sch[p], scl[p], -(g0.w * c0h));
                            if (DH) ff_add(shh[p], shl[p], -(g0.w * h0h));
                        }
                    }
                }
            }
            if (DU)
#pragma unroll
                for (int p = 0; p < P / 2; ++p)
#pragma unroll
                    for (int s = 0; s < SM; ++s) {
                        const float2 v = up2(plj[p][s]);
                        ff_add(ljh[2 * p][s], ljl[2 * p][s], v.x);
                        ff_add(ljh[2 * p + 1][s], ljl[2 * p + 1][s], v.y);
                    }
        }
        __syncthreads();
        if (tid == 0 && t + 2 < ntiles) issue(t + 2);
    }
    if (j >= g.ny || k >= g.nz || i0 >= g.nx) return;
    const int64_t plane = (int64_t)g.nx * g.ny * g.nz;
    const int64_t row = ((int64_t)k * g.ny + j) * g.nx;
    const bool vec_ok = (g.nx & 1) == 0;
    const double ih = 1.0 / g.h;
    const double cu0 = ph.k_e * ih, cc0 = -ph.beta * ph.k_e * ih, ch0 = -ph.beta * ph.k_e / (2.0 * ph.eps_r) * ih;
    double F1[P], FK[P], SC[P], SH[P];
#pragma unroll
    for (int p = 0; p < P; ++p) {
        F1[p] = (double)f1h[p] + (double)f1l[p];
        FK[p] = (double)fkh[p] + (double)fkl[p];
        SC[p] = (double)sch[p] + (double)scl[p];
        SH[p] = (double)shh[p] + (double)shl[p];
    }
#pragma unroll
    for (int s = 0; s < SM; ++s) {
        if (s >= ph.S) break;
        const double qs = ph.qs[s];
        double v[P];
        if (DU) {
#pragma unroll
            for (int p = 0; p < P; ++p)
                v[p] = (hit >> p & 1u) ? INFINITY : cu0 * qs * F1[p] + ((double)ljh[p][s] + (double)ljl[p][s]);
            store_strip<P>(o.u + s * plane + row, i0, g.nx, v, vec_ok);
        }
        if (DC) {
#pragma unroll
            for (int p = 0; p < P; ++p) v[p] = cc0 * qs * (F1[p] - SC[p]);
            store_strip<P>(o.c + s * plane + row, i0, g.nx, v, vec_ok);
        }
        if (DH) {
#pragma unroll
            for (int p = 0; p < P; ++p) v[p] = ch0 * qs * (2.0 * ph.ea2 * FK[p] - SH[p]);
            store_strip<P>(o.h + s * plane + row, i0, g.nx, v, vec_ok);
        }
    }
}

// ---------------------------------------------------------------- launch
namespace {
template <int SM, int P, bool DU, bool DH>
cudaError_t run_direct32(const GridD& g, const Phys& ph, const DevTables& t, Outputs o, long long wl, int dbg,
                         cudaStream_t st) {
    const size_t sm = 2 * kDirectT * sizeof(SrcF) + 2 * kDirectT * SM * sizeof(LJf) + (kDirectT / 2) * sizeof(DirRec) +
                      2 * sizeof(uint64_t) + 4 * kDirectT * sizeof(int) + 2 * kNTab * sizeof(float4);
    const dim3 grid((g.nx + 4 * P - 1) / (4 * P), (g.ny + 7) / 8, (g.nz + 3) / 4);
    raise_dyn_smem(k_direct32<SM, P, DU, DH>, sm);
    k_direct32<SM, P, DU, DH><<<grid, 128, sm, st>>>(g, ph, t.srcf, t.ljf, t.n, t.sr, t.sr_inv, o, t.err, wl, dbg);
    return cudaGetLastError();
}

template <int SM, int P, bool DU, bool DH>
cudaError_t run_direct64(const GridD& g, const Phys& ph, const DevTables& t, Outputs o, long long wl, int dbg,
                         cudaStream_t st) {
    const size_t sm = 2 * kDirectT * sizeof(Geo) + 2 * kDirectT * SM * sizeof(LJd) + 2 * sizeof(uint64_t) +
                      kLen64 * sizeof(double);
    const dim3 grid((g.nx + 4 * P - 1) / (4 * P), (g.ny + 7) / 8, (g.nz + 3) / 4);
    auto kern = k_direct64<SM, P, kDirectT, DU, DH>;
    raise_dyn_smem(kern, sm);
    kern<<<grid, 128, sm, st>>>(g, ph, t.geo, t.ljd, t.n, t.sr64, o, t.err, wl, dbg);
    return cudaGetLastError();
}

template <int SM, bool DU, bool DH>
cudaError_t run_direct(const GridD& g, const Phys& ph, const DevTables& t, int prec, Outputs o, long long wl,
                       int dbg, cudaStream_t st) {
    const int64_t ctas = (int64_t)((g.nx + 15) / 16) * ((g.ny + 7) / 8) * ((g.nz + 3) / 4);  // four points per lane
    if (prec == RISM_PREC_FP64) {
        // one point per lane where four would be fewer than three waves of CTAs (200 atoms, two sites, one against four
        // points: 32^3, 64 CTAs, 0.45 / 0.90 ms; 56^3, 392 CTAs, 1.79 / 1.94; 64^3, 512 CTAs, 2.46 / 2.41; 80^3 4.39 / 4.08)
        if (ctas >= 3 * (int64_t)sm_count()) return run_direct64<SM, 4, DU, DH>(g, ph, t, o, wl, dbg, st);
        return run_direct64<SM, 1, DU, DH>(g, ph, t, o, wl, dbg, st);
    }
    // four points per lane share an atom's y and z terms, but only where that still leaves a few waves of CTAs (2,000
    // atoms, 128^3, 4,096 CTAs: 2.30 against 2.61 ms; 500 atoms, 64^3, 512 CTAs: 0.47 against 0.39)
    if (ctas >= 12 * (int64_t)sm_count()) return run_direct32<SM, 4, DU, DH>(g, ph, t, o, wl, dbg, st);
    return run_direct32<SM, 2, DU, DH>(g, ph, t, o, wl, dbg, st);
}

template <int SM>
cudaError_t run_direct_sm(const GridD& g, const Phys& ph, const DevTables& t, int prec, Outputs o, long long wl,
                          int dbg, cudaStream_t st) {
    const bool du = o.u != nullptr, dh = o.h != nullptr;
    if (du && dh) return run_direct<SM, true, true>(g, ph, t, prec, o, wl, dbg, st);
    if (du) return run_direct<SM, true, false>(g, ph, t, prec, o, wl, dbg, st);
    if (dh) return run_direct<SM, false, true>(g, ph, t, prec, o, wl, dbg, st);
    return run_direct<SM, false, false>(g, ph, t, prec, o, wl, dbg, st);
}
}  // namespace

int direct_variant_count() { return 1; }

cudaError_t launch_direct(const GridD& g, const Phys& ph_, const DevTables& t, int precision, Outputs o,
                          long long wait_limit, int variant, int dbg, cudaStream_t st) {
    (void)variant;
    Phys ph = ph_;
    if (t.sr || t.sr64) ph.rs = short_reach(ph, precision == RISM_PREC_FP64);
    switch (t.smax) {
        case 2: return run_direct_sm<2>(g, ph, t, precision, o, wait_limit, dbg, st);
        case 4: return run_direct_sm<4>(g, ph, t, precision, o, wait_limit, dbg, st);
        case 8: return run_direct_sm<8>(g, ph, t, precision, o, wait_limit, dbg, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace rism
