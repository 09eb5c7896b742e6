// rism_kspace.cu -- reciprocal-space long-range asymptotics on the grid's reciprocal lattice.
//
// Eq. (dcf-k) and eq. (tcf-k) (Sec. 2.2), times the Coulomb constant of the unit reading:
//   c_s(k) = -(4 pi beta k_e q_s / k^2) e^{-k^2 eta^2/4} S(k)
//   h_s(k) = -(4 pi beta k_e q_s / (eps_r (k^2 + kappa^2))) e^{-k^2 eta^2/4} S(k),
//   S(k)   = sum_a Q_a e^{i k.(R_a - o)},
// o the grid origin, k = 2 pi (m_x/(n_x h), m_y/(n_y h), m_z/(n_z h)) on the half spectrum of a real-to-complex
// transform ([n_z][n_y][n_x/2 + 1], m_x = j_x, m = j or j - n along y and z), c(0) = 0.  With the frequency
// cut-off of Sec. 2.5 only k^2 <= k_cut^2 is summed (the rest is 0).
//
// The structure factor is a contraction over the atoms.  With the cosine (c) and sine (s) of each coordinate's
// phase, the eight real sums sum_a Q_a {c,s}_x {c,s}_y {c,s}_z of non-negative (m_x, m_y, m_z) give S at all four
// sign choices of (m_y, m_z):
//   Re S = ccc - t u css - t ssc - u scs,   Im S = scc - t u sss + t csc + u ccs,   t = sign m_y, u = sign m_z,
// so they are one real matrix product over the atoms,
//   rows (m_x, {c,s}) x columns (m_y, m_z, {cc,cs,sc,ss}),
// with half the multiplications of the complex form, and it runs on the tensor cores (tcgen05, kind::f16, FP32
// accumulators in TMEM).
//
// Precision: a tensor-core accumulator truncates, so FP32-class sums need more than the plain product of split
// operands.  Each FP32 operand v, scaled to |v| <= 256, is split into v1 + v2 + v3: v1 an integer, v2 a multiple
// of 2^-12 with |v2| <= 1/2, v3 the rest, each exact in FP16 (v3 to 2^-25).  The products v1 w1 are integers up to
// 2^16 whose sums stay below 2^24 over a block of atoms (the block length comes from the charges, see
// kspace_charge_plan): they accumulate without any rounding in one TMEM accumulator.  The other five products
// (v1 w2, v2 w1, v2 w2, v1 w3, v3 w1) are smaller by 2^-9 or more and share a second accumulator, whose truncation
// is 2^-9 of an FP32 rounding per step.  What is left out (v2 w3, v3 w2, v3 w3) is 2e-8 of the sum.
//
//   k_ktab: phase tables (the phase m x / n is reduced modulo one cycle exactly -- integer part of x modulo n in
//           integer arithmetic, the rest as an error-free product and float-float sum; sincospi of the rounded
//           half-cycle count plus the first-order term of what the rounding left): the x table as the three FP16
//           slices in the layout the tensor cores read, the y and the (charge-weighted) z table in FP32; its first
//           CTA also lays out the (m_y, m_z) pairs, those inside the cut-off first.
//   k_ksum: persistent, one CTA per SM, items of 64 m_x x up to 64 (m_y, m_z) pairs.  Per 32 atoms one bulk TMA
//           copy brings the x slices (24 KB); eight builder warps form the column operands Q y z in FP32, slice
//           them and store them; one thread issues the 12 products.  The builder warps also read the accumulators
//           back: the four sign choices, the k-dependent factors, every site's c and h as FP64 complex values
//           (each rounded once to FP32, widened on the integer pipe).
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "rism_kspace.h"

namespace rism {
namespace {

constexpr int kKA = 32;            // atoms per chunk (one pipeline stage)
constexpr int kKM = 64;            // m_x per item: 128 rows (c and s of each in adjacent rows)
constexpr int kKP = 64;            // (m_y, m_z) pairs per item at most: 256 columns
constexpr int kKStages = 3;
constexpr int kKBuild = 8;         // builder warps
constexpr int kKThreads = 32 * (kKBuild + 2);
// Operands in shared memory: per slice, groups of 8 atoms of 16-byte records (8 FP16) of every row.
constexpr uint32_t kKGroupA = 128 * 16, kKSliceA = (kKA / 8) * kKGroupA;  // bytes of the row operand
constexpr uint32_t kKBytesA = 3 * kKSliceA;
constexpr uint32_t kKBytesB = 3 * (kKA / 8) * 4 * kKP * 16;
constexpr int kKLo = 256;          // TMEM column of the second accumulator
constexpr float kKScale = 256.f;   // operands are scaled to |v| <= 256
constexpr int kKBlock = 64;        // chunks per accumulation block at most
constexpr size_t kKFlush = sizeof(float2) * 128 * 4 * kKP;  // bytes of one CTA's running sums

// The blocked tables.  xs: FP16 slices [mt][npad/32][slice][atom/8][row][8] (rows 2i, 2i+1: c and s of m_x =
// 64 t + i), one chunk of one m_x tile contiguous.  yt, zt: [npad/8][4][m] of (c_a, c_a+1, s_a, s_a+1), so the
// consecutive m of a warp's lanes are consecutive float4; z carries the charge and the operand scale.
struct KTables {
    uint4* xs;
    float4 *yt, *zt;
    double *kx2, *ky2, *kz2;  // squared wave numbers of m >= 0
    int *list, *cnt;          // pair order (cut-off only): pairs that more m_x tiles need first; cnt[t]: pairs of tile t
    float2* flush;            // [CTAs][4 kKP][128] running sums of solutes longer than a block
    int npad, mt, nxh, nym, nzm, np;  // np = nym nzm pairs
};

// e^{i 2 pi m x / na} for x = xh + xl grid units (float-float), 0 <= m < 2^16.
__device__ __forceinline__ float2 lattice_phase(float xh, float xl, int m, int na) {
    const float fi = floorf(xh), nf = (float)na;
    const float ff = xh - fi;                       // exact: [0, 1)
    int ir = (int)(fi >= 0.f && fi < nf ? fi : fmodf(fi, nf));  // integer part modulo na (fmodf is exact)
    if (ir < 0) ir += na;
    const uint32_t r0 = ((uint32_t)m * (uint32_t)ir) % (uint32_t)na;  // m, ir < 2^16
    const float fm = (float)m;
    const float p2 = fm * ff;                       // m * frac(xh), with its rounding error e2
    const float e2 = fmaf(fm, ff, -p2);
    const float p3 = fm * xl;                       // the low part: a tiny correction
    float s, e1;
    two_sum((float)r0, p2, s, e1);                  // s + e1 = r0 + p2 exactly
    const float lo = e1 + e2 + p3;
    const float qn = rintf(s / nf);
    const float r2 = 2.0f * fmaf(-qn, nf, s);       // exact: |r2| <= na and a multiple of ulp(2 s)
    const float q = __fdiv_rn(r2, nf);              // half cycles, and what the division leaves
    const float w = 3.14159265358979f * ((fmaf(-q, nf, r2) + 2.0f * lo) / nf);
    float sn, cs;
    sincospif(q, &sn, &cs);
    return make_float2(fmaf(-w, sn, cs), fmaf(w, cs, sn));
}

// (2 pi m / (n h))^2, rounded operation by operation as the FP64 definition orders it.
__device__ __forceinline__ double lattice_q2(int m, int n, double h) {
    const double k = __ddiv_rn(__dmul_rn(__dmul_rn(2.0, M_PI), (double)m), __dmul_rn((double)n, h));
    return __dmul_rn(k, k);
}

// The three slices of a pair of operands |v| <= 256 (consecutive atoms in the low and high halves).
__device__ __forceinline__ uint32_t half2_of(f32x2 v) {
    const float2 f = up2(v);
    const __half2 h = __floats2half2_rn(f.x, f.y);
    return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ void slice3(f32x2 v, uint32_t& h1, uint32_t& h2, uint32_t& h3) {
    // adding and subtracting 1.5 2^23 ulp rounds to a multiple of ulp: 1 and 2^-12
    const f32x2 M1 = pk2(12582912.f, 12582912.f), M2 = pk2(3072.f, 3072.f);
    const f32x2 v1 = sub2(add2(v, M1), M1), r = sub2(v, v1);
    const f32x2 v2 = sub2(add2(r, M2), M2);
    h1 = half2_of(v1);
    h2 = half2_of(v2);
    h3 = half2_of(sub2(r, v2));
}

struct KTabArgs {
    KTables tb;
    const SrcF* srcf;
    int n, nx, ny, nz;
    double h, kc2;
    float zscale;  // operand scale of the charge-weighted table: 256 / (power of two >= max |Q|)
};

// CTA 0: the squared wave numbers and, with a cut-off, the pair order: a counting sort by the number of m_x
// tiles a pair needs, most first (the order inside a class is arbitrary; every pair's sums are its own).
__device__ void pair_plan(const KTabArgs& a) {
    const KTables& tb = a.tb;
    for (int m = threadIdx.x; m < tb.nxh; m += blockDim.x) tb.kx2[m] = lattice_q2(m, a.nx, a.h);
    for (int m = threadIdx.x; m < tb.nym; m += blockDim.x) tb.ky2[m] = lattice_q2(m, a.ny, a.h);
    for (int m = threadIdx.x; m < tb.nzm; m += blockDim.x) tb.kz2[m] = lattice_q2(m, a.nz, a.h);
    if (!(a.kc2 > 0.0)) return;
    constexpr int kMaxT = 65536 / 2 / kKM + 2;
    __shared__ int at[kMaxT];  // [class]: count, then next position
    for (int t = threadIdx.x; t <= tb.mt; t += blockDim.x) at[t] = 0;
    __syncthreads();
    auto cls = [&](int p) {  // m_x tiles with an entry inside the sphere
        const double y2 = tb.ky2[p % tb.nym], z2 = tb.kz2[p / tb.nym];
        int t = 0;
        while (t < tb.mt && __dadd_rn(__dadd_rn(tb.kx2[t * kKM], y2), z2) <= a.kc2) ++t;
        return t;
    };
    for (int p = threadIdx.x; p < tb.np; p += blockDim.x) atomicAdd(&at[cls(p)], 1);
    __syncthreads();
    if (threadIdx.x == 0) {
        int acc = 0;
        for (int t = tb.mt; t >= 0; --t) {
            const int c = at[t];
            at[t] = acc;
            acc += c;
            if (t > 0) tb.cnt[t - 1] = acc;  // pairs that need tile t - 1: the classes above it
        }
    }
    __syncthreads();
    for (int p = threadIdx.x; p < tb.np; p += blockDim.x) tb.list[atomicAdd(&at[cls(p)], 1)] = p;
}

__global__ void __launch_bounds__(256) k_ktab(KTabArgs a) {
    const KTables& tb = a.tb;
    if (blockIdx.x == 0) {
        pair_plan(a);
        return;
    }
    const int64_t nx8 = (int64_t)tb.mt * kKM * (tb.npad / 8), nyz = (int64_t)(tb.nym + tb.nzm) * (tb.npad / 2);
    const int64_t stride = (int64_t)(gridDim.x - 1) * blockDim.x;
    for (int64_t t = (int64_t)(blockIdx.x - 1) * blockDim.x + threadIdx.x; t < nx8 + nyz; t += stride) {
        if (t < nx8) {
            // one m_x, eight atoms: six 16-byte records, rows c and s of each slice
            const int i = (int)(t % kKM), g = (int)((t / kKM) % (tb.npad / 8)), mt = (int)(t / kKM / (tb.npad / 8));
            const int m = mt * kKM + i;
            uint32_t c[3][4], s[3][4];
            for (int j = 0; j < 4; ++j) {
                float2 e[2];
                for (int k = 0; k < 2; ++k) {
                    const int at = 8 * g + 2 * j + k;
                    e[k] = make_float2(0.f, 0.f);
                    if (at < a.n && m < tb.nxh) e[k] = lattice_phase(a.srcf[at].xh, a.srcf[at].xl, m, a.nx);
                }
                slice3(pk2(e[0].x * kKScale, e[1].x * kKScale), c[0][j], c[1][j], c[2][j]);
                slice3(pk2(e[0].y * kKScale, e[1].y * kKScale), s[0][j], s[1][j], s[2][j]);
            }
            uint4* o = tb.xs + ((int64_t)mt * (tb.npad / kKA) + g / 4) * (kKBytesA / 16) + (g % 4) * (kKGroupA / 16) + 2 * i;
            for (int l = 0; l < 3; ++l) {
                o[l * (kKSliceA / 16)] = make_uint4(c[l][0], c[l][1], c[l][2], c[l][3]);
                o[l * (kKSliceA / 16) + 1] = make_uint4(s[l][0], s[l][1], s[l][2], s[l][3]);
            }
        } else {
            // one m_y or m_z, two atoms
            const int64_t u = t - nx8;
            const int w = tb.nym + tb.nzm, j = (int)(u % w), h2 = (int)(u / w);  // h2: atom pair
            const bool y = j < tb.nym;
            const int m = y ? j : j - tb.nym;
            float2 e[2];
            for (int k = 0; k < 2; ++k) {
                const int at = 2 * h2 + k;
                e[k] = make_float2(0.f, 0.f);
                if (at >= a.n) continue;
                const SrcF f = a.srcf[at];
                if (y) {
                    e[k] = lattice_phase(f.yh, f.yl, m, a.ny);
                } else {
                    const float q = f.q * a.zscale;  // a power of two: exact
                    e[k] = lattice_phase(f.zh, f.zl, m, a.nz);
                    e[k].x *= q;
                    e[k].y *= q;
                }
            }
            (y ? tb.yt : tb.zt)[(int64_t)h2 * (y ? tb.nym : tb.nzm) + m] = make_float4(e[0].x, e[1].x, e[0].y, e[1].y);
        }
    }
}

struct KSumArgs {
    KTables tb;
    int nx, ny, nz, S;
    int pt;                  // pairs per item, a multiple of 8
    int block;               // chunks per accumulation block
    double kc2;              // kc2 <= 0: no cut-off
    float fc0, fh0;          // -4 pi beta k_e and -4 pi beta k_e / eps_r
    float oscale;            // 1 / (scales of the two operands), a power of two
    float eta2q;             // eta^2 / 4
    float kap2;              // kappa^2 (0: h not requested / undefined)
    float qs[kMaxSites];
    double* c;               // [S][nz][ny][nxh] complex (re, im), or null
    double* hk;              // same, or null
    DevErr* err;
    long long wlim;
};

// ---- tcgen05
// Shared-memory operand descriptor, K-major without swizzle: 8-row x 16-byte core matrices, `lead` bytes between
// core matrices along K and 128 bytes between them along the rows.
__device__ __forceinline__ uint64_t umma_desc(uint32_t addr, uint32_t lead) {
    return (uint64_t)((addr >> 4) & 0x3fff) | (uint64_t)((lead >> 4) & 0x3fff) << 16 | (uint64_t)(128 >> 4) << 32 |
           (uint64_t)1 << 46;
}
// One lane of the issuing warp, elected so that the compiler knows the branch runs one thread: with a lane picked by
// its index the operands of an MMA count as divergent, and issuing one took 100 clocks instead of under 50 (an MMA
// of 128 x 224 x 16 takes 112).
__device__ __forceinline__ bool elect_one() {
    uint32_t e;
    asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(e));
    return e != 0;
}
__device__ __forceinline__ void umma_f16(uint32_t d, uint64_t da, uint64_t db, uint32_t idesc, bool acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d), "l"(da), "l"(db), "r"(idesc), "r"((uint32_t)acc)
        : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void tmem_ld2(uint32_t addr, float (&v)[2]) {
    uint32_t r[2];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr) : "memory");
    v[0] = __uint_as_float(r[0]);
    v[1] = __uint_as_float(r[1]);
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void bar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

struct KSmem {
    uint64_t full[kKStages], empty[kKStages], acc_full, acc_free;
    uint32_t tmem;
};

// One work item: pairs [p0, p0 + n) of m_x tile t; zero: entries beyond the cut-off, nothing is summed.
struct KItem {
    int t, p0, n;
    bool zero;
};
__device__ __forceinline__ bool item_at(const KSumArgs& a, int i, KItem& it) {
    const KTables& tb = a.tb;
    for (int z = 0; z < (a.kc2 > 0.0 ? 2 : 1); ++z)
        for (int t = 0; t < tb.mt; ++t) {
            const int c = a.kc2 > 0.0 ? tb.cnt[t] : tb.np;
            const int lo = z ? c : 0, hi = z ? tb.np : c, w = z ? kKP : a.pt, k = (hi - lo + w - 1) / w;
            if (i < k) {
                it = KItem{t, lo + i * w, min(w, hi - lo - i * w), z != 0};
                return true;
            }
            i -= k;
        }
    return false;
}

struct FF {
    float h, l;
};
__device__ __forceinline__ FF ff_sum(FF a, FF b, float s) {  // a + s b, s = +-1
    float h, e;
    two_sum(a.h, s * b.h, h, e);
    return FF{h, e + (a.l + s * b.l)};
}

// The entries of one pair at all sign choices, for m_x = jx: the lane of the c row writes u = +, of the s row u = -.
__device__ __forceinline__ void write_pair(const KSumArgs& a, int pair, int jx, bool odd, double kx2, bool summed,
                                           const FF (&own)[4], const FF (&oth)[4]) {
    const KTables& tb = a.tb;
    const int my = pair % tb.nym, mz = pair / tb.nym;
    if (jx >= tb.nxh || (odd ? mz < 1 : mz > (a.nz - 1) / 2)) return;
    const int jz = odd ? a.nz - mz : mz;
    const double k2d = __dadd_rn(__dadd_rn(kx2, tb.ky2[my]), tb.kz2[mz]);
    const bool keep = summed && (!(a.kc2 > 0.0) || k2d <= a.kc2);
    float fc = 0.f, fh = 0.f;
    if (keep) {
        const float k2 = (float)k2d;
        const float g = expf(-k2 * a.eta2q);
        fc = k2 > 0.f ? a.fc0 * g / k2 : 0.f;
        fh = a.kap2 > 0.f ? a.fh0 * g / (k2 + a.kap2) : 0.f;
    }
    const float u = odd ? -1.f : 1.f;
    const FF* C = odd ? oth : own;
    const FF* Sn = odd ? own : oth;
    // t-even and t-odd parts: Re = (ccc - u scs) - t (u css + ssc), Im = (scc + u ccs) + t (csc - u sss)
    const FF re0 = ff_sum(C[0], Sn[1], -u), re1 = ff_sum(Sn[2], C[3], u);
    const FF im0 = ff_sum(Sn[0], C[1], u), im1 = ff_sum(C[2], Sn[3], -u);
    const int64_t plane = (int64_t)a.ny * tb.nxh, site = plane * a.nz;
#pragma unroll
    for (int neg = 0; neg < 2; ++neg) {
        if (neg ? my < 1 : my > (a.ny - 1) / 2) continue;
        const FF re = ff_sum(re0, re1, neg ? 1.f : -1.f), im = ff_sum(im0, im1, neg ? -1.f : 1.f);
        const float sre = keep ? (re.h + re.l) * a.oscale : 0.f, sim = keep ? (im.h + im.l) * a.oscale : 0.f;
        const int64_t o = (int64_t)jz * plane + (int64_t)(neg ? a.ny - my : my) * tb.nxh + jx;
        for (int s = 0; s < a.S; ++s) {
            if (a.c) {
                const float f = a.qs[s] * fc;
                __stcs(reinterpret_cast<double2*>(a.c) + s * site + o, make_double2(f2d_alu(f * sre), f2d_alu(f * sim)));
            }
            if (a.hk) {
                const float f = a.qs[s] * fh;
                __stcs(reinterpret_cast<double2*>(a.hk) + s * site + o, make_double2(f2d_alu(f * sre), f2d_alu(f * sim)));
            }
        }
    }
}

__device__ __forceinline__ int pair_at(const KSumArgs& a, int p) { return a.kc2 > 0.0 ? a.tb.list[p] : p; }

// Read-back of one block of an item by the builder warps (quad: TMEM lanes; part: every other two pairs): added to the
// CTA's running sums of earlier blocks (more), which it becomes, or written to the outputs (last).  Two pairs at a
// time: with four, registers spill in the builders' loop.
__device__ __forceinline__ void read_back(const KSumArgs& a, const KItem& it, uint32_t tmem, int quad, int part, bool more,
                                       bool last) {
    const KTables& tb = a.tb;
    const int lane = threadIdx.x & 31, row = quad * 32 + lane, jx = it.t * kKM + row / 2;
    const double kx2 = tb.kx2[min(jx, tb.nxh - 1)];
    float2* fl = tb.flush ? tb.flush + (size_t)blockIdx.x * (kKFlush / sizeof(float2)) + row : nullptr;
    auto earlier = [&](int p, float2 (&o)[4][2]) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int k = 0; k < 2; ++k) o[q][k] = fl[(q * a.pt + p + k) * 128];
    };
    float2 next[4][2];
    if (more) earlier(2 * part, next);
    for (int p = 2 * part; p < a.pt; p += kKBuild / 2) {
        float x[4][2], y[4][2];
        float2 old[4][2];
        FF v[4][2];
        __syncwarp();  // the whole warp reads TMEM together
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t at = tmem + ((uint32_t)(quad * 32) << 16) + q * a.pt + p;
            tmem_ld2(at, x[q]);
            tmem_ld2(at + kKLo, y[q]);
#pragma unroll
            for (int k = 0; k < 2; ++k) old[q][k] = next[q][k];
        }
        if (more && p + kKBuild / 2 < a.pt) earlier(p + kKBuild / 2, next);  // ahead of this pass's stores
        tmem_wait_ld();
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                two_sum(x[q][k], y[q][k], v[q][k].h, v[q][k].l);
                if (more) v[q][k] = ff_sum(FF{old[q][k].x, old[q][k].y}, v[q][k], 1.f);
                if (!last) fl[(q * a.pt + p + k) * 128] = make_float2(v[q][k].h, v[q][k].l);
            }
        if (!last) continue;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            FF own[4], oth[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                own[q] = v[q][k];
                oth[q].h = __shfl_xor_sync(0xffffffffu, own[q].h, 1);
                oth[q].l = __shfl_xor_sync(0xffffffffu, own[q].l, 1);
            }
            if (p + k < it.n) write_pair(a, pair_at(a, it.p0 + p + k), jx, lane & 1, kx2, true, own, oth);
        }
    }
}

__device__ __forceinline__ void zero_fill(const KSumArgs& a, const KItem& it, int quad, int part) {
    const int row = quad * 32 + (threadIdx.x & 31), jx = it.t * kKM + row / 2;
    const FF none[4] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
    for (int p = part; p < it.n; p += kKBuild / 4)
        write_pair(a, pair_at(a, it.p0 + p), jx, row & 1, 0.0, false, none, none);
}

// What bounds it (13,600 atoms, 224x192x160, the whole half spectrum: 256 rows x 31,428 columns x 13,600 atoms x six
// products, 1.3e12 FP16 operations): 0.95 ms.  The items are 56 pairs wide there (224 columns), two to a CTA, 425
// chunks each: at 1,860 clocks a chunk 0.76 ms, of which the tensor cores need 1,344 (12 MMAs of 128 x 224 x 16, 112
// clocks each: 0.55 ms) and the builders about as long.  The rest, 0.19 ms, is the read-back: the running sums of an
// item's blocks and the outputs (444 MB).  The form it replaces, complex FP32 multiply-adds on the FMA pipe over twice
// the columns, took 10.1 ms.  Narrower items read the row operand more often per product.  The two accumulators take
// all 512 TMEM columns, so the read-back of an item does not overlap the products of the next.
__global__ void __launch_bounds__(kKThreads, 1) k_ksum(const __grid_constant__ KSumArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    unsigned char* sA = smem;                              // [stage][slice][atom/8][row][8 halves]
    unsigned char* sB = smem + kKStages * kKBytesA;        // [stage][slice][atom/8][column][8 halves]
    KSmem& m = *reinterpret_cast<KSmem*>(smem + kKStages * (kKBytesA + kKBytesB));
    const int tid = threadIdx.x, lane = tid & 31, w = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const KTables& tb = a.tb;
    const int nch = tb.npad / kKA, N = 4 * a.pt;
    if (tid == 0) {
        for (int s = 0; s < kKStages; ++s) {
            mbar_init(&m.full[s], 1 + kKBuild);
            mbar_init(&m.empty[s], 1);
        }
        mbar_init(&m.acc_full, 1);
        mbar_init(&m.acc_free, kKBuild);
        mbar_fence_init();
    }
    if (w == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&m.tmem))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = m.tmem;
    // bounded waits: a role whose wait runs out reports it and leaves, and the others' waits then run out too
    auto wait = [&](uint64_t* bar, int parity) {
        if (mbar_wait_bounded(bar, (uint32_t)parity, a.wlim)) return true;
        report_error(a.err, DEV_TIMEOUT, WHERE_KSPACE);
        return false;
    };
    auto all = [](bool v) { return __all_sync(0xffffffffu, v) != 0; };
    // position in the ring of stages: n counts chunks up to the first reuse of a stage
    struct Ring {
        int s = 0, ph = 0, n = 0;
        __device__ void next() {
            if (++s == kKStages) {
                s = 0;
                ph ^= 1;
            }
            n = min(n + 1, kKStages);
        }
        __device__ bool reused() const { return n == kKStages; }
    };
    if (w == kKBuild) {
        // ---- the row operand: one bulk copy per chunk
        if (lane == 0) {
            Ring r;
            bool ok = true;
            KItem it;
            for (int i = blockIdx.x; ok && item_at(a, i, it) && !it.zero; i += gridDim.x) {
                const uint4* src = tb.xs + (int64_t)it.t * nch * (kKBytesA / 16);
                for (int c = 0; c < nch; ++c, src += kKBytesA / 16, r.next()) {
                    if (r.reused() && !(ok = wait(&m.empty[r.s], r.ph ^ 1))) break;
                    mbar_expect_tx(&m.full[r.s], kKBytesA);
                    bulk_g2s(sA + r.s * kKBytesA, src, kKBytesA, &m.full[r.s]);
                }
            }
            // the copies have landed once their products are done (or, after a failed wait, by these waits' limit)
            for (int q = 0; q < r.n; ++q) {
                if (r.s-- == 0) {
                    r.s = kKStages - 1;
                    r.ph ^= 1;
                }
                mbar_wait_bounded(&m.full[r.s], (uint32_t)r.ph, a.wlim);
            }
        }
    } else if (w == kKBuild + 1) {
        // ---- the products: D1 += v1 w1, D2 += v1 w2 + v2 w1 + v2 w2 + v1 w3 + v3 w1
        if (elect_one()) {
            // FP32 accumulators, FP16 operands, both K-major, N columns, 128 rows
            const uint32_t idesc = 1u << 4 | (uint32_t)(N >> 3) << 17 | (uint32_t)(128 >> 4) << 24;
            // operand descriptors of stage 0; a column group is N 16-byte units
            const uint32_t gb = (uint32_t)N;
            const uint64_t a0 = umma_desc(smem_u32(sA), kKGroupA), b0 = umma_desc(smem_u32(sB), 16 * gb);
            Ring r;
            int accph = 1;  // parity of the last read-back
            bool ok = true, some = false;
            KItem it;
            for (int i = blockIdx.x; ok && item_at(a, i, it) && !it.zero; i += gridDim.x)
                for (int c = 0, left = 0; c < nch; ++c, r.next()) {
                    // The tensor core's queue is short: what this thread does between two chunks' products leaves it
                    // idle, so a chunk is one wait (both operands arrive on one barrier), its products, one commit.
                    const bool first = left == 0;
                    if (first) {
                        left = min(a.block, nch - c);
                        if (some && !(ok = wait(&m.acc_free, accph))) break;
                        some = true;
                        accph ^= 1;
                    }
                    if (!(ok = wait(&m.full[r.s], r.ph))) break;
                    fence_after();
                    const uint64_t da = a0 + (uint32_t)r.s * (kKBytesA / 16), db = b0 + (uint32_t)r.s * (kKBytesB / 16);
#pragma unroll
                    for (int ks = 0; ks < kKA / 16; ++ks) {
                        const uint64_t a1 = da + ks * (2 * kKGroupA / 16), b1 = db + ks * 2 * gb;
                        const uint64_t a2 = a1 + kKSliceA / 16, b2 = b1 + 4 * gb;
                        const bool acc = ks > 0 || !first;
                        umma_f16(tmem, a1, b1, idesc, acc);
                        umma_f16(tmem + kKLo, a1, b2, idesc, acc);
                        umma_f16(tmem + kKLo, a1, b2 + 4 * gb, idesc, true);
                        umma_f16(tmem + kKLo, a2, b1, idesc, true);
                        umma_f16(tmem + kKLo, a2, b2, idesc, true);
                        umma_f16(tmem + kKLo, a2 + kKSliceA / 16, b1, idesc, true);
                    }
                    umma_commit(&m.empty[r.s]);
                    if (--left == 0) umma_commit(&m.acc_full);
                }
            // leave only when every product issued is done: its operands and TMEM are given back after this
            for (int q = 0; q < r.n; ++q) {
                if (r.s-- == 0) {
                    r.s = kKStages - 1;
                    r.ph ^= 1;
                }
                mbar_wait_bounded(&m.empty[r.s], (uint32_t)r.ph, a.wlim);
            }
        }
    } else {
        // ---- builders: thread = (pair, 8 atoms) of a chunk; then the read-back
        const int bp = tid % a.pt, bg = tid / a.pt;  // pair, atom group (groups >= 4: idle)
        const bool act = bg < kKA / 8;
        const int quad = w & 3, part = w >> 2;
        Ring r;
        int accph = 0;
        bool ok = true;
        KItem it;
        for (int i = blockIdx.x; ok && item_at(a, i, it); i += gridDim.x) {
            if (it.zero) {
                zero_fill(a, it, quad, part);
                continue;
            }
            const int pr = pair_at(a, it.p0 + min(bp, it.n - 1));
            const float4* yp = tb.yt + pr % tb.nym + (int64_t)(act ? 4 * bg : 0) * tb.nym;
            const float4* zp = tb.zt + pr / tb.nym + (int64_t)(act ? 4 * bg : 0) * tb.nzm;
            float4 Y[4], Z[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                Y[j] = __ldg(yp + j * tb.nym);
                Z[j] = __ldg(zp + j * tb.nzm);
            }
            bool more = false;  // running sums of earlier blocks
            for (int c = 0, left = min(a.block, nch); c < nch; ++c, r.next()) {
                if (c + 1 < nch) {
                    yp += 16 * (int64_t)tb.nym;
                    zp += 16 * (int64_t)tb.nzm;
                }
                // slices of the thread's 4 columns x 8 atoms; each phase of the next chunk loads as soon as this
                // chunk's is used, so every load has a whole chunk to arrive
                uint32_t o[4][3][4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const f32x2 yc = pk2(Y[j].x, Y[j].y), ys = pk2(Y[j].z, Y[j].w);
                    const f32x2 zc = pk2(Z[j].x, Z[j].y), zs = pk2(Z[j].z, Z[j].w);
                    Y[j] = __ldg(yp + j * tb.nym);
                    Z[j] = __ldg(zp + j * tb.nzm);
                    slice3(mul2(yc, zc), o[0][0][j], o[0][1][j], o[0][2][j]);
                    slice3(mul2(yc, zs), o[1][0][j], o[1][1][j], o[1][2][j]);
                    slice3(mul2(ys, zc), o[2][0][j], o[2][1][j], o[2][2][j]);
                    slice3(mul2(ys, zs), o[3][0][j], o[3][1][j], o[3][2][j]);
                }
                if (r.reused() && !(ok = all(wait(&m.empty[r.s], r.ph ^ 1)))) break;
                if (act) {
                    uint4* dst = reinterpret_cast<uint4*>(sB + r.s * kKBytesB) + bg * N + bp;
#pragma unroll
                    for (int q = 0; q < 4; ++q)
#pragma unroll
                        for (int l = 0; l < 3; ++l)
                            dst[l * 4 * N + q * a.pt] = make_uint4(o[q][l][0], o[q][l][1], o[q][l][2], o[q][l][3]);
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) bar_arrive(&m.full[r.s]);
                if (--left > 0) continue;
                const bool last = c + 1 == nch;
                left = min(a.block, nch - 1 - c);
                // read-back of one block: into the running sums, or (the last) to the outputs
                if (!(ok = all(wait(&m.acc_full, accph)))) break;
                accph ^= 1;
                fence_after();
                read_back(a, it, tmem, quad, part, more, last);
                fence_before();
                __syncwarp();
                if (lane == 0) bar_arrive(&m.acc_free);
                more = true;
            }
        }
    }
    __syncwarp();
    fence_before();
    __syncthreads();
    fence_after();
    if (w == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
}

int round_up(int v, int m) { return (v + m - 1) / m * m; }

// Sizes and places of the tables in one allocation.
size_t table_plan(int64_t n, int nx, int ny, int nz, bool flush, int sms, void* base, KTables* out) {
    KTables tb{};
    tb.npad = round_up((int)std::max<int64_t>(n, 1), kKA);
    tb.nxh = nx / 2 + 1;
    tb.mt = (tb.nxh + kKM - 1) / kKM;
    tb.nym = ny / 2 + 1;
    tb.nzm = nz / 2 + 1;
    tb.np = tb.nym * tb.nzm;
    size_t at = 0;
    auto take = [&](size_t bytes) {
        void* p = base ? static_cast<unsigned char*>(base) + at : nullptr;
        at += (bytes + 255) / 256 * 256;
        return p;
    };
    tb.xs = static_cast<uint4*>(take((size_t)tb.mt * (tb.npad / kKA) * kKBytesA));
    tb.yt = static_cast<float4*>(take(sizeof(float4) * (size_t)(tb.npad / 2) * tb.nym));
    tb.zt = static_cast<float4*>(take(sizeof(float4) * (size_t)(tb.npad / 2) * tb.nzm));
    tb.kx2 = static_cast<double*>(take(sizeof(double) * tb.nxh));
    tb.ky2 = static_cast<double*>(take(sizeof(double) * tb.nym));
    tb.kz2 = static_cast<double*>(take(sizeof(double) * tb.nzm));
    tb.list = static_cast<int*>(take(sizeof(int) * (size_t)tb.np));
    tb.cnt = static_cast<int*>(take(sizeof(int) * (size_t)tb.mt));
    tb.flush = flush ? static_cast<float2*>(take(kKFlush * (size_t)sms)) : nullptr;
    if (out) *out = tb;
    return at;
}

}  // namespace

// Block length: the exact accumulator holds integers below 2^24; with |v1| <= 256 and |w1| <= 256 |Q|/qscale + 1/2
// a block of atoms stays below that while 256 (256 sum |Q|/qscale + atoms/2) does.
void kspace_charge_plan(const double* raw, int64_t n, KspaceSetup& s) {
    double qmax = 0.0;
    s.qabs = 0.0;
    const int64_t nch = (std::max<int64_t>(n, 1) + kKA - 1) / kKA;
    std::vector<double> sum((size_t)nch, 0.0);
    for (int64_t i = 0; i < n; ++i) {
        const double q = std::fabs(raw[6 * i + 3]);
        s.qabs += q;
        qmax = std::max(qmax, q);
        sum[(size_t)(i / kKA)] += q;
    }
    // a power of two at least as large as every FP32 charge (1 for uncharged atoms), and no smaller than 2^-110, so that
    // 256 over it and it over 2^16 stay normal FP32 numbers
    int e = 0;
    std::frexp(qmax > 0.0 ? qmax : 0.5, &e);
    s.qscale = std::ldexp(1.0, std::min(std::max(e, -110), 128));
    int64_t len = std::min<int64_t>(nch, kKBlock);
    for (; len > 1; len = len * 3 / 4) {
        double worst = 0.0;
        for (int64_t c0 = 0; c0 < nch; c0 += len) {
            double t = 0.0;
            for (int64_t c = c0; c < std::min(nch, c0 + len); ++c) t += sum[(size_t)c];
            worst = std::max(worst, t);
        }
        if (kKScale * (kKScale * worst / s.qscale + 0.5 * (double)(len * kKA)) < 16777216.0) break;
    }
    s.block = (int)len;
    s.blocks = (int)((nch + len - 1) / len);
}

size_t kspace_table_bytes(int64_t n, int nx, int ny, int nz, const KspaceSetup& s, int sms) {
    return table_plan(n, nx, ny, nz, s.blocks > 1, sms, nullptr, nullptr);
}

double kspace_bound(double k, const KspaceSetup& s) {
    return 4.0 * std::sqrt(2.0) * M_PI * s.beta * s.k_e * s.qmax * std::exp(-k * k * s.eta * s.eta / 4.0) * s.qabs /
           (k * k);
}

// k where the bound equals tol: Newton on log(bound) - log(tol) (decreasing and convex in k), from a start
// below the root, safeguarded by bisection on a bracket.
double kspace_kcut(const KspaceSetup& s, double tol) {
    if (!(tol > 0.0) || !(s.qabs > 0.0) || !(s.qmax > 0.0)) return 0.0;
    double lo = 1e-6, hi = 1.0;
    while (kspace_bound(hi, s) > tol && hi < 1e6) hi *= 2.0;
    if (kspace_bound(lo, s) <= tol) return lo;
    double k = lo;
    for (int it = 0; it < 200; ++it) {
        const double g = std::log(kspace_bound(k, s)) - std::log(tol);
        if (g > 0.0) lo = k; else hi = k;
        const double dg = -k * s.eta * s.eta / 2.0 - 2.0 / k;
        double kn = k - g / dg;
        if (!(kn > lo && kn < hi)) kn = 0.5 * (lo + hi);
        if (std::fabs(kn - k) <= 1e-15 * k) {
            k = kn;
            break;
        }
        k = kn;
    }
    return k;
}

cudaError_t launch_kspace(const DevTables& t, const GridD& g, const KspaceSetup& s, int sms, void* tables,
                          double* c_k, double* h_k, long long wait_limit, cudaStream_t st) {
    KTabArgs ta;
    table_plan(t.n, g.nx, g.ny, g.nz, s.blocks > 1, sms, tables, &ta.tb);
    const KTables& tb = ta.tb;
    ta.srcf = t.srcf;
    ta.n = (int)t.n;
    ta.nx = g.nx;
    ta.ny = g.ny;
    ta.nz = g.nz;
    ta.h = g.h;
    ta.kc2 = s.kcut > 0.0 ? s.kcut * s.kcut : 0.0;
    ta.zscale = (float)(kKScale / s.qscale);
    const int64_t work = (int64_t)tb.mt * kKM * (tb.npad / 8) + (int64_t)(tb.nym + tb.nzm) * (tb.npad / 2);
    k_ktab<<<1 + (int)std::min<int64_t>((work + 255) / 256, 16 * sms), 256, 0, st>>>(ta);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    KSumArgs a;
    a.tb = tb;
    a.nx = g.nx;
    a.ny = g.ny;
    a.nz = g.nz;
    a.S = s.S;
    a.block = s.block;
    a.kc2 = ta.kc2;
    a.fc0 = (float)(-4.0 * M_PI * s.beta * s.k_e);
    a.fh0 = (float)(-4.0 * M_PI * s.beta * s.k_e / s.eps_r);
    a.oscale = (float)(s.qscale / kKScale / kKScale);
    a.eta2q = (float)(s.eta * s.eta / 4.0);
    a.kap2 = (float)(s.kappa * s.kappa);
    for (int k = 0; k < kMaxSites; ++k) a.qs[k] = (float)s.qs[k];
    a.c = c_k;
    a.hk = h_k;
    a.err = t.err;
    a.wlim = wait_limit;
    // pairs per item: the fewest waves of one item per SM, each wave as long as its item is wide (plus a fixed
    // share); with a cut-off the pairs inside it are estimated by the area of their quarter ellipse
    double np = (double)tb.np, rows = (double)tb.mt;
    if (ta.kc2 > 0.0) {
        const double ky = s.kcut * g.ny * g.h / (2.0 * M_PI), kz = s.kcut * g.nz * g.h / (2.0 * M_PI);
        np = std::min(np, 0.25 * M_PI * (ky + 1.0) * (kz + 1.0) + 1.0);
        rows = std::min(rows, std::ceil((s.kcut * g.nx * g.h / (2.0 * M_PI) + 1.0) / kKM));
    }
    double best = 1e300;
    a.pt = kKP;
    for (int pt = kKP; pt >= 16; pt -= 8) {
        const double cost = std::ceil(rows * std::ceil(np / pt) / sms) * (pt + 12);
        if (cost < best) {
            best = cost;
            a.pt = pt;
        }
    }
    const size_t sm = kKStages * (kKBytesA + kKBytesB) + sizeof(KSmem);
    raise_dyn_smem(k_ksum, sm);
    k_ksum<<<sms, kKThreads, sm, st>>>(a);
    return cudaGetLastError();
}

}  // namespace rism
