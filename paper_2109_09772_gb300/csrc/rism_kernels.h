// rism_kernels.h -- host-side launch interface between the C ABI layer and
// the CUDA kernels (internal).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "rism_internal.cuh"

namespace rism {

// Device tables of one solute/solvent pair (owned by the context).
struct DevTables {
    int64_t n = 0;    // atoms
    int smax = 2;     // padded site count (2, 4 or 8)
    Geo* geo = nullptr;   // [n] physical positions + charge
    SrcF* srcf = nullptr; // [n] grid-unit positions (relative to the grid origin, float-float) + charge
    LJd* ljd = nullptr;   // [n][smax]
    LJf* ljf = nullptr;   // [n][smax]
    DevErr* err = nullptr;
    // FP32 direct sum: the short-range kernels' pieces (short_range_table) and kNTab / r_short in grid units; null: the
    // kernels are called per pair (a caller without device memory of its own for them)
    const float4* sr = nullptr;
    float sr_inv = 0.f;
    const double* sr64 = nullptr;  // the FP64 direct sum's (short_range_table64), null likewise
};

// The short-range kernels F_c(d) = erfc(x) and F_h(d) = e^{-x^2}[erfcx(x-a) + erfcx(x+a)] as cubic Hermite pieces in d
// over [0, r_short], [kNTab][2] (host).
void short_range_table(const Phys& ph, double h, float4* tab);
// The same two kernels for FP64: kTab64 pieces of kTerm64 coefficients each (F_c then F_h) about the middle of their
// segment of [0, r_short], then 2^(j/256) as pairs (host, kLen64 doubles).
constexpr int kTab64 = 256, kTerm64 = 8, kLen64 = 2 * kTab64 * kTerm64 + 512;
void short_range_table64(const Phys& ph, double* tab);
// The pieces serve the direct sum for a = kappa eta/2 up to 1/2 (e^{-2ax} varies little over a piece) and end where the
// kernels do, so that a wide r_short does not stretch them: beyond 6 eta (FP64) F_c is below 2.2e-17 and F_h below
// 4.4e-17, beyond 5 eta (FP32) below 1.6e-12 and 3.2e-12.  Otherwise the library's functions are called.
inline bool short_pieces(const Phys& ph) { return ph.a <= 0.5; }
inline double short_reach(const Phys& ph, bool f64) { return fmin(ph.rs, (f64 ? 6.0 : 5.0) * ph.eta); }

struct Outputs {
    double* u = nullptr;
    double* c = nullptr;
    double* h = nullptr;
};

// a1: mixing, LJ A/B, per-pair cut-offs, grid-unit positions.
// raw = [n][6] (x, y, z, q, sigma, eps) on the device; site tables on the host (in Phys + arrays).
cudaError_t launch_setup(const double* raw, int64_t n, int S, int smax, const double* sig_s, const double* eps_s,
                         int lj_mode, double lj_rcut, double lj_tol, const GridD& g, DevTables& t,
                         cudaStream_t st);

// a4: I_s = sum_i 4 pi (A/(9 rc^9) - B/(3 rc^3)) into dev_out[S].
cudaError_t launch_lj_tail(const DevTables& t, int S, double* dev_out, cudaStream_t st);

// a2/a3/a5/a6 by direct summation over all atoms (FP64 or FP32 pairs).
cudaError_t launch_direct(const GridD& g, const Phys& ph, const DevTables& t, int precision, Outputs o,
                          long long wait_limit, int variant, int debug_flags, cudaStream_t st);

int direct_variant_count();

}  // namespace rism
