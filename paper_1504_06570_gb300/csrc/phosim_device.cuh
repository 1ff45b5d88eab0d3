// Device-side data layout and per-photon physics of the GB300 photon Monte Carlo library.
//
// One thread follows one photon through Sec. 2 of Peterson et al. (2015): sampling (Sec. 2.2), the
// frozen-flow screen layers (Sec. 2.3), the surfaces (Sec. 2.4.1-2.4.2), the silicon sensor and the
// pixel (Sec. 2.4.2, 2.5).  Scene constants travel in the kernel parameter block (constant bank), so every
// per-surface read is a uniform constant-cache hit; screens and tables are read through the L1/L2 path.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "phosim.h"
#include "ds.cuh"
#include "fp64.cuh"

namespace phosim {

constexpr int kMaxMaterials = 8;
constexpr int kMaxCoatings = 8;
constexpr int kZPoly = 28;                 // monomials x^a y^b, a + b <= 6
constexpr int kSedGuide = 256;             // guide-table buckets of the wavelength-bin draw (its top 8 bits)

enum SurfFlags : int {
    SF_CONIC = 1, SF_EVEN = 2, SF_ODD = 4, SF_ZERN = 8, SF_FLAT_ONLY = 16, SF_ROTATED = 32,
    SF_DECENTERED = 64          // a vertex off the axis (the double-single transforms skip zero x, y offsets)
};

struct DSurface {
    int kind, material, coating, coat_slot;   // coat_slot: index of this surface's accept draw, -1 none
    int flags;
    int mat_before;                           // medium in front of the surface (material index, -1 vacuum)
    int ne, no;                               // terms of the even / odd polynomials up to the last nonzero one
    double c, k1c2, kc;                       // 1/R, (1 + kappa) / R^2, (1 + kappa) / R
    double ae[4];                             // alpha_4, alpha_6, alpha_8, alpha_10
    double ao[4];                             // alpha_3, alpha_5, alpha_7, alpha_9
    double aed[4], aod[4];                    // the same times their powers of r: terms of (1/r) dz/dr
    double M[9];                              // telescope -> surface frame rotation (row-major)
    double o[3];                              // displaced vertex in the telescope frame
    double r_in2, r_out2;
    double zinv;                              // 1 / zern_rnorm
    double zp[kZPoly];                        // sum_j c_j Z_j as monomials of (x zinv, y zinv), row b = y power
};

// The shape and placement of a surface as double-single pairs, for the FP32-pipe optics.  The asphere
// polynomials are rescaled to the normalised radius rho = r / rn (rn the clear radius), so that their
// coefficients stay far from the single-precision underflow that alpha_10 ~ 1e-30 mm^-9 would reach:
// even part  z = sum_k ae[k] u^(k+2),  u = rho^2;   (1/r) dz/dr = inv_rn2 u sum_k aed[k] u^k
// odd part   z = rho^3 sum_k ao[k] u^k;             (1/r) dz/dr = inv_rn2 rho sum_k aod[k] u^k
struct DSurfaceS {
    ds c, k1c2, kc;
    ds kmc;                                   // kc - c = kappa c: the quadric's d_z^2 term for a unit direction
    ds ae[4], aed[4], ao[4], aod[4];
    ds M[9], o[3];
    ds r_in2, r_out2;
    ds inv_rn, inv_rn2;
    float ae2[4];                             // (k + 1) aed[k] / rn^4: d^2 S / (d r^2)^2 terms of the even part, single
    float zinv;
    unsigned char ne, no, pad0, pad1;         // terms of the even / odd polynomials up to the last nonzero one
    float zp[kZPoly];
};

struct DMaterial {
    int kind, pad;
    double B[3], C[3];
    ds Bs[3], Cs[3];
};

struct DCoating {
    double lam0, inv_dlam, th0, inv_dth;
    float lam0f, inv_dlamf, th0f, inv_dthf;
    ds lam0_s, inv_dlam_s;                    // the wavelength grid as double-single pairs (its bins)
    int nl, nt, pad0, pad1;
    // transmissions as integer thresholds ceil(T 2^32 - 1/2) on the draw
    const unsigned long long* T_thr;          // nl x nt
    const unsigned long long* Tmax_thr;       // nl: the largest over angles at each wavelength
    // of T + R (ghosts), or null when the coating does not reflect
    const unsigned long long* TR_thr;
};

// internal scene flag: a coating reflects (ghosts)
constexpr uint32_t kGhostFlag = 1u << 24;
constexpr int kMaxGhostBounces = PHOSIM_MAX_GHOST_BOUNCES;

// A screen scale's central-difference gradient (rad / mm), stored per node (i, j) as the 2 x 2 block of
// nodes the bilinear interpolation needs, (i, j), (i+1, j), (i, j+1), (i+1, j+1) (periodic): one lookup is
// one aligned 32-byte (FP32) or 64-byte (FP64) read instead of two rows of scattered 8- or 16-byte taps.
struct DScale {
    int n, inv_shift;
    double inv_pix;
    unsigned long long inv_m;                 // inv_pix as a factor of integers (factor64), with inv_shift
    ds inv_pix_s;
    const double2* g64;                       // 4 double2 per node, n x n nodes: the bilinear form's coefficients of 1, X, Y
                                              // and X Y, where X and Y are 1 + the distance from the node in pixels
    const float4* g32;                        // 2 float4 per node: (g00, g10), (g01, g11)
};

struct DLayer {
    double z, vx, vy;
    ds zs, vxs, vys;
    ds dzs;                                   // height of the plane above (the previous layer or the top) over z
    double dz;                                // the same
    int n_scales, pad;
    DScale s[PHOSIM_MAX_SCALES];
};

struct SourceS;                              // a source's constants as the double-single path reads them

struct DSource {
    int kind, sed, table;
    uint32_t bundle;                          // photons per ray (Sec. 3.2 background optimisation), >= 1
    double xi, eta, zfac, t0, t_exp, a, b, cpa, spa;
    double bsig;                              // sigma of the spread of a ray's photons on the detector, mm
    double ref_x, ref_y;
    float ref_s[4];                           // ref_x, ref_y as double-single pairs (hi, lo, hi, lo)
    uint64_t first, count, rec_off;           // photons [first, first + count); record index of the first
    uint64_t ufirst, ucount;                  // work units of the two-kernel path: rays of a bundle, else photons
    // Dynamic transmission: the wavelength-bin draws w that some coating may let pass have w - w_lo <= w_span
    // (modulo 2^32); every other draw is a wavelength that a coating stops whatever its own draw (pass_draws)
    uint32_t w_lo, w_span;
};

// counters: [0] traced, [1] detected, [1 + r] dropped for reason r
constexpr int kNumCounters = 10;

struct TraceParams {
    // scene
    uint32_t k0, k1;                          // Philox key
    uint32_t flags;
    int n_surf, n_layers, n_coated, n_mat, n_coat;
    int coated_surface[PHOSIM_MAX_COATED];    // surface index of coated-surface draw k
    // Dynamic transmission: outside [pass_lo, pass_hi) nm one of the coated surfaces it tests lets nothing pass; solid:
    // inside none of them does
    int pass_solid, pad_solid;
    double pass_lo, pass_hi;
    double pr_in2, pr_dr2;                    // pupil annulus
    double h_top, z_ent;
    double lam_ref, kick0;                    // kick0 = lambda_ref [mm] / 2 pi
    double inv_lam_ref;
    double pupil_z;                           // nominal vertex height of the first surface
    DSurface pupil_surf;                      // its nominal shape (no figure error, no misalignment)
    DSurface surf[PHOSIM_MAX_SURFACES];
    DMaterial mat[kMaxMaterials];
    DCoating coat[kMaxCoatings];
    DLayer layer[PHOSIM_MAX_LAYERS];
    // the same scene in double-single / single precision for the FP32-pipe path
    DSurfaceS surf_s[PHOSIM_MAX_SURFACES];
    DSurfaceS pupil_s;
    ds pr_in2_s, pr_dr2_s, h_top_s, z_ent_s, pupil_z_s, xlo_s, ylo_s, inv_pixel_s, chip_w_s, chip_h_s;
    float kick0f, inv_lam_ref_f, sed_lam0f, sed_dlamf, t_sif, dead_layerf, ell_lam0f, inv_ell_dlamf, sig_scalef;
    // sensor / detector
    int nx, ny, n_ell, n_sig;
    const double* draw_table;     // log_draw64, sincos_draw64
    double pixel, inv_pixel, xlo, ylo, chip_w, chip_h, t_si, ell_lam0, inv_ell_dlam, sig_scale, dead_layer;
    // fringing (PHOSIM_FRINGE): the silicon's optical thickness at (x, y) of the detector surface frame is
    // fr_t0 + fr_gx x + fr_gy y
    double fr_t0, fr_gx, fr_gy;
    ds fr_t0_s;
    float fr_gxf, fr_gyf;
    const double* ell;
    const float* ell32;
    const double* sig;
    const float* sig32;
    // spectra, shapes
    int n_bins, sersic_K;
    double sed_lam0, sed_dlam;
    ds sed_lam0_s, sed_dlam_s;
    const unsigned long long* thr;            // n_sed x (n_bins - 1) integer thresholds on the bin draw
    const int* sed_guide;                     // n_sed x (kSedGuide + 1): first threshold above j 2^24
    const double* sersic;
    const float* sersic32;
    int hf_K;                                 // quantiles of the high-frequency kick (0 = none)
    const double* hf;
    const float* hf32;
    // work and outputs: tile t of the launch is tile t - tile_prefix[s] of the source s with
    // tile_prefix[s] <= t < tile_prefix[s + 1]; a tile holds tile_photons consecutive photons
    const DSource* sources;
    SourceS* sources_s;                       // the same sources converted once by call_prep_kernel (two-kernel path)
    const unsigned long long* tile_prefix;
    int n_src;
    uint32_t tile_photons;
    uint64_t n_tiles;
    unsigned long long* tile_counter;
    unsigned long long* counters;
    uint32_t* image;
    double* moments;
    phosim_photon_record* records;
    // the two-kernel double-single path's moment accumulators: kMomStripes copies of the per-source sums
    // (PHOSIM_MOMENT_WORDS a source, mom_stripe_stride doubles a copy), a block adding to copy blockIdx %
    // kMomStripes so that a bright source's atomics spread over several cache lines; null: add to moments
    double* mom_stripes;
    unsigned long long mom_stripe_stride;
};
constexpr int kMomStripes = 16;
// warps of the entry and bundle stages' blocks (the shared-memory queues and counters are sized for it)
constexpr int kWarpsPerBlock = 8;

// Up to 32 photons of one source that go on past the dynamic transmission test, for one warp: photons first + k
struct __align__(16) PhotonBatch {
    int src;
    uint32_t n;
    unsigned long long first;
    uint32_t k[32];
};
// the words of a photon's forward state: of each surface, and after the surfaces
enum { kTapeH = 0, kTapeD = 3, kTapeL = 6, kTapeN = 7, kTapeMu = 10, kTapeSurface = 11 };       // words of a surface
enum { kTapeDepth = 0, kTapeX = 1, kTapeY = 2, kTapeOn = 3, kTapeEnd = 4 };                     // words after the surfaces
// The batches of tiles [tile_begin, tile_end): their number, and the next one to be taken
struct BatchList {
    PhotonBatch* batch;
    unsigned long long *n, *next;
    uint64_t tile_begin, tile_end;
    // For the adjoint, the photons' forward state (ForwardRecord in photon.cuh): the first tape_batches batches' in a slot
    // each of tape_stride words, and after those a slot for each block that works on a batch without one
    double* tape;
    unsigned long long tape_batches, tape_stride;
    int tape_first;               // the first surface recorded
};

// What a trace call does before its rays (call_prep_kernel): the source list and the tile prefix, given here when they
// are few (no copy then), the sources' constants and passing wavelength draws, and zeroes for the call's scratch.
constexpr int kInlineSources = 12;
struct CallPrep {
    DSource* sources;
    SourceS* sources_s;                       // null outside the two-kernel path
    unsigned long long* tile_prefix;
    int n_src, n_inline;                      // n_inline: n_src when the lists are below, else 0 (they were copied)
    int n_bins, pad;
    double pass_lo, pass_hi, sed_lam0, sed_dlam;
    const unsigned long long* thr;
    uint32_t* zero[3];                        // words to clear
    unsigned long long zero_words[3];
    DSource inline_sources[kInlineSources];
    unsigned long long inline_prefix[kInlineSources + 1];
};

// ------------------------------------------------------------------------------------------------------
// Programmatic dependent launch: a kernel that lets the next one on the stream start beside it, and the next one's
// wait for it (no effect on a kernel launched without that attribute).
// ------------------------------------------------------------------------------------------------------
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ------------------------------------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds, two 32x32 multiplications per round.
// ------------------------------------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return c;
}

// slot map of one photon's random words: counter = (photon lo, photon hi, source, block)
//   block 0: pupil r, pupil phi, wavelength bin, wavelength blur
//   block 1: time, shape a, shape b, conversion
//   block 2: diffusion a, diffusion b, coated surface 0, coated surface 1
//   block 3: coated surfaces 2..5
//   block 4: high-frequency kick magnitude, direction, back-side reflection
//   blocks 5, 6 (photons of a bundle, counter of the photon; the ray uses blocks 0-4 of the ray's counter):
//            spread a, spread b, conversion, diffusion a; diffusion b, back-side reflection
//   blocks 7, 8, ... (ghosts): the coating decisions after the first reflection, one word each, in order
// (exact, by the bits of 2^20 + w 2^-32)
__device__ __forceinline__ double u64of(uint32_t w) { return __hiloint2double(0x41300000, (int)w) - (1048576.0 - 1.1641532182693481e-10); }
// the uniform (w + 1/2) 2^-32 of a word in single precision: the whole word converts (exactly below 2^24), so
// the small values that the -log u of the conversion depth and of Box-Muller reach keep 24 significant bits
__device__ __forceinline__ float u32of(uint32_t w) {
    return __fadd_rn(__fmul_rn((float)w, 2.3283064365386963e-10f), 1.1641532182693481e-10f);
}

// ------------------------------------------------------------------------------------------------------
// surface shape (Sec. 2.4.1)
// ------------------------------------------------------------------------------------------------------
// Zernike figure as a bivariate polynomial of degree 6 in normalised coordinates (u, v).
__device__ __forceinline__ void zern_eval(const double* __restrict__ zp, double u, double v, double& z, double& zu,
                                          double& zv) {
    // rows b = 0..6 hold the x-polynomial of y^b, degree 6 - b, ascending powers of x
    double q[7], dq[7];
    int off = 0;
#pragma unroll
    for (int b = 0; b <= 6; ++b) {
        const int deg = 6 - b;
        double acc = zp[off + deg], dacc = 0.0;
#pragma unroll
        for (int a = deg - 1; a >= 0; --a) {
            dacc = fma(dacc, u, acc);
            acc = fma(acc, u, zp[off + a]);
        }
        q[b] = acc;
        dq[b] = dacc;
        off += deg + 1;
    }
    double zz = q[6], zzu = dq[6], zzv = 0.0;
#pragma unroll
    for (int b = 5; b >= 0; --b) {
        zzv = fma(zzv, v, zz);
        zz = fma(zz, v, q[b]);
        zzu = fma(zzu, v, dq[b]);
    }
    z = zz; zu = zzu; zv = zzv;
}

// Second derivatives of the Zernike figure in its normalised coordinates, single precision
__device__ __forceinline__ void zern_hess_f(const float* __restrict__ zp, float u, float v, float& zuu, float& zuv, float& zvv) {
    float q[7], dq[7], d2q[7];
    int off = 0;
#pragma unroll
    for (int b = 0; b <= 6; ++b) {
        const int deg = 6 - b;
        float acc = zp[off + deg], dacc = 0.f, hacc = 0.f;     // hacc: half the second derivative
#pragma unroll
        for (int a = deg - 1; a >= 0; --a) {
            hacc = fmaf(hacc, u, dacc);
            dacc = fmaf(dacc, u, acc);
            acc = fmaf(acc, u, zp[off + a]);
        }
        q[b] = acc; dq[b] = dacc; d2q[b] = 2.f * hacc;
        off += deg + 1;
    }
    float z = q[6], zv = 0.f, hv = 0.f, zu = dq[6], wuv = 0.f, wuu = d2q[6];
#pragma unroll
    for (int b = 5; b >= 0; --b) {
        hv = fmaf(hv, v, zv);
        zv = fmaf(zv, v, z);
        z = fmaf(z, v, q[b]);
        wuv = fmaf(wuv, v, zu);
        zu = fmaf(zu, v, dq[b]);
        wuu = fmaf(wuu, v, d2q[b]);
    }
    zuu = wuu; zuv = wuv; zvv = 2.f * hv;
}

// The aspheric and Zernike part of the sag, its slopes, and its second derivatives H = (xx, xy, yy) in single
// precision (from g = (1/r) dS/dr and its derivative in r^2: S_xx = g + 2 x^2 g1 and so on).  E: the single-precision
// constants of the surface.
__device__ __forceinline__ void aspheric(const DSurface& S, const DSurfaceS& E, double x, double y, double r2, double& z,
                                         double& zx, double& zy, float H[3]) {
    double g = 0.0;
    float g1 = 0.f;
    z = 0.0;
    // Horner from the last nonzero coefficient: the zero terms above it would add exact zeros
    if (S.flags & SF_EVEN) {
        int k = S.ne - 1;
        double pe = S.ae[k], pd = S.aed[k];
#pragma unroll 1
        while (--k >= 0) {
            pe = fma(r2, pe, S.ae[k]);
            pd = fma(r2, pd, S.aed[k]);
        }
        z = r2 * r2 * pe;
        g = r2 * pd;
        const float u = f32_trunc(r2) * E.inv_rn2.hi;
        k = E.ne - 1;
        float q = E.ae2[k];
#pragma unroll 1
        while (--k >= 0) q = fmaf(q, u, E.ae2[k]);
        g1 += q;
    }
    if (S.flags & SF_ODD) {
        const double r = sqrt64(r2);
        int k = S.no - 1;
        double po = S.ao[k], pd = S.aod[k];
#pragma unroll 1
        while (--k >= 0) {
            po = fma(r2, po, S.ao[k]);
            pd = fma(r2, pd, S.aod[k]);
        }
        z = fma(r2 * r, po, z);
        g = fma(r, pd, g);
        // with rho = r / rn the odd part of g is rho sum_k aod[k] rho^(2k) / rn^2
        const float rho = f32_trunc(r) * E.inv_rn.hi, u = rho * rho;
        k = E.no - 1;
        float q = ((float)k + 0.5f) * E.aod[k].hi;
#pragma unroll 1
        while (--k >= 0) q = fmaf(q, u, ((float)k + 0.5f) * E.aod[k].hi);
        if (rho > 1e-12f) g1 += q / rho * (E.inv_rn2.hi * E.inv_rn2.hi);
    }
    zx = x * g;
    zy = y * g;
    const float xf = f32_trunc(x), yf = f32_trunc(y), gf = f32_trunc(g);
    H[0] = fmaf(2.f * xf * xf, g1, gf);
    H[1] = 2.f * xf * yf * g1;
    H[2] = fmaf(2.f * yf * yf, g1, gf);
    if (S.flags & SF_ZERN) {
        double zz, zu, zv;
        zern_eval(S.zp, x * S.zinv, y * S.zinv, zz, zu, zv);
        z += zz;
        zx = fma(zu, S.zinv, zx);
        zy = fma(zv, S.zinv, zy);
        float huu, huv, hvv;
        zern_hess_f(E.zp, xf * E.zinv, yf * E.zinv, huu, huv, hvv);
        const float k = E.zinv * E.zinv;
        H[0] = fmaf(huu, k, H[0]); H[1] = fmaf(huv, k, H[1]); H[2] = fmaf(hvv, k, H[2]);
    }
}

// Sag of the conic, even and odd terms at squared radius r2 (the pupil is sampled on the nominal first surface)
__device__ __forceinline__ double sag(const DSurface& S, double r2) {
    double z = 0.0;
    if (S.flags & SF_CONIC) {
        const double arg = fma(-S.k1c2, r2, 1.0);
        if (negative64(arg)) return 0.0;          // outside the conic's domain
        z = S.c * r2 * rcp64(1.0 + sqrt64(arg));
    }
    if (S.flags & SF_EVEN) {
        int k = S.ne - 1;
        double pe = S.ae[k];
#pragma unroll 1
        while (--k >= 0) pe = fma(r2, pe, S.ae[k]);
        z = fma(r2 * r2, pe, z);
    }
    if (S.flags & SF_ODD) {
        int k = S.no - 1;
        double po = S.ao[k];
#pragma unroll 1
        while (--k >= 0) po = fma(r2, po, S.ao[k]);
        z = fma(r2 * sqrt64(r2), po, z);
    }
    return z;
}

__device__ __forceinline__ void zern_eval_f(const float* __restrict__ zp, float u, float v, float& z, float& zu,
                                            float& zv) {
    float q[7], dq[7];
    int off = 0;
#pragma unroll
    for (int b = 0; b <= 6; ++b) {
        const int deg = 6 - b;
        float acc = zp[off + deg], dacc = 0.f;
#pragma unroll
        for (int a = deg - 1; a >= 0; --a) {
            dacc = fmaf(dacc, u, acc);
            acc = fmaf(acc, u, zp[off + a]);
        }
        q[b] = acc;
        dq[b] = dacc;
        off += deg + 1;
    }
    float zz = q[6], zzu = dq[6], zzv = 0.f;
#pragma unroll
    for (int b = 5; b >= 0; --b) {
        zzv = fmaf(zzv, v, zz);
        zz = fmaf(zz, v, q[b]);
        zzu = fmaf(zzu, v, dq[b]);
    }
    z = zz; zu = zzu; zv = zzv;
}

// Sag and slopes in single precision (the hi parts of the surface's constants), for the first Newton steps
__device__ __forceinline__ bool sag_f(const DSurfaceS& E, int flags, float x, float y, float& z, float& zx, float& zy) {
    const float r2 = fmaf(x, x, y * y);
    float g = 0.f;
    z = 0.f;
    if (flags & SF_CONIC) {
        const float arg = fmaf(-E.k1c2.hi, r2, 1.f);
        if (arg < 0.f) return false;
        const float rs = rsqrtf(arg);
        z = quotient_f(E.c.hi * r2, fmaf(arg, rs, 1.f));
        g = E.c.hi * rs;
    }
    if (flags & SF_EVEN) {
        const float u = r2 * E.inv_rn2.hi;
        int k = E.ne - 1;
        float pe = E.ae[k].hi, pd = E.aed[k].hi;
#pragma unroll 1
        while (--k >= 0) {
            pe = fmaf(pe, u, E.ae[k].hi);
            pd = fmaf(pd, u, E.aed[k].hi);
        }
        z = fmaf(u * u, pe, z);
        g = fmaf(u * E.inv_rn2.hi, pd, g);
    }
    if (flags & SF_ODD) {
        const float rho = sqrtf(r2) * E.inv_rn.hi;
        const float u = rho * rho;
        int k = E.no - 1;
        float po = E.ao[k].hi, pd = E.aod[k].hi;
#pragma unroll 1
        while (--k >= 0) {
            po = fmaf(po, u, E.ao[k].hi);
            pd = fmaf(pd, u, E.aod[k].hi);
        }
        z = fmaf(u * rho, po, z);
        g = fmaf(rho * E.inv_rn2.hi, pd, g);
    }
    zx = x * g;
    zy = y * g;
    if (flags & SF_ZERN) {
        float zz, zu, zv;
        zern_eval_f(E.zp, x * E.zinv, y * E.zinv, zz, zu, zv);
        z += zz;
        zx = fmaf(zu, E.zinv, zx);
        zy = fmaf(zv, E.zinv, zy);
    }
    return true;
}

// Exact root of the conic's quadric c (x^2 + y^2) + kc z^2 - 2 z = 0 (kc = (1 + kappa) c) along the ray p + l d on
// the vertex branch (1 - kc z >= 0), of two such the one nearer to the ray's own start at l = -from; infinity when the ray
// misses it, and NaN for a ray without a place or a direction.  Out of line: only rays that graze the conic, where the single-precision root says too little, come here.
static __device__ __noinline__ double conic_root(double c, double kc, double p0, double p1, double p2, double d0, double d1,
                                                 double d2, double from) {
    const double A = c * fma(d0, d0, d1 * d1) + kc * d2 * d2;
    const double b = c * fma(p0, d0, p1 * d1) + fma(kc * p2, d2, -d2);
    const double C = c * fma(p0, p0, p1 * p1) + fma(kc * p2, p2, -2.0 * p2);
    const double disc = fma(b, b, -A * C);
    if (disc < 0.0) return INFINITY;
    const double q = -(b + copysign(sqrt(disc), b));
    if (q == 0.0) return INFINITY;
    const double near = C / q;                                        // the root nearer to p; the other is q / A
    const bool second = fabs((from + near) * A) > fabs(fma(from, A, q));
    const double l = second ? q / A : near;
    if (A != 0.0 && fma(-kc, fma(l, d2, p2), 1.0) < 0.0) return second ? near : q / A;   // the other is the vertex branch
    return l;
}

// The sag and its slopes in FP64, term by term in rolled loops, which take few registers from the caller; false outside the
// conic's domain.
static __device__ __forceinline__ bool far_sag(const DSurface& S, double x, double y, double& z, double& zx, double& zy) {
    const double r2 = fma(x, x, y * y);
    double g = 0.0;                       // (1/r) dz/dr of the terms of the radius
    z = 0.0;
    if (S.flags & SF_CONIC) {
        const double arg = fma(-S.k1c2, r2, 1.0);
        if (arg < 0.0) return false;
        const double root = sqrt(arg);
        z = S.c * r2 / (1.0 + root);
        g = S.c / root;
    }
    double p = 0.0, q = 0.0;
    if (S.flags & SF_EVEN) {
#pragma unroll 1
        for (int k = S.ne - 1; k >= 0; --k) {
            p = fma(r2, p, S.ae[k]);
            q = fma(r2, q, S.aed[k]);
        }
        z = fma(r2 * r2, p, z);
        g = fma(r2, q, g);
    }
    if (S.flags & SF_ODD) {
        const double r = sqrt(r2);
        p = q = 0.0;
#pragma unroll 1
        for (int k = S.no - 1; k >= 0; --k) {
            p = fma(r2, p, S.ao[k]);
            q = fma(r2, q, S.aod[k]);
        }
        z = fma(r2 * r, p, z);
        g = fma(r, q, g);
    }
    zx = x * g;
    zy = y * g;
    if (S.flags & SF_ZERN) {
        const double u = x * S.zinv, v = y * S.zinv;
        double zz = 0.0, zu = 0.0, zv = 0.0;
        const double* row = S.zp + kZPoly - 1;           // the rows of powers of v, each of the powers of u, from the last
#pragma unroll 1
        for (int n = 1; n <= 7; ++n) {
            double a = 0.0, da = 0.0;
#pragma unroll 1
            for (int k = 0; k < n; ++k, --row) {
                da = fma(da, u, a);
                a = fma(a, u, *row);
            }
            zv = fma(zv, v, zz);
            zz = fma(zz, v, a);
            zu = fma(zu, v, da);
        }
        z += zz;
        zx = fma(zu, S.zinv, zx);
        zy = fma(zv, S.zinv, zy);
    }
    return true;
}

// An aspheric or Zernike surface where the single-precision start below does not come near it: Newton's method on the sag
// in FP64 from the conic's root along p + l d (the ray's own start is at l = -from), until the step is below 1e-8 mm.
// Whether it gets there within 20 steps, and whether it leaves the conic's domain on its way, is what says that a ray meets
// such a surface or how it is lost: steep terms have roots of their own beyond the aperture, which a method with larger
// steps finds where this one ends.  Out of line, for the rays that come in far off the aperture: those that a lens or a
// mirror is made for do not get here (2e7 photons all FP64 6.24 ms with it, 6.33 where every ray went on from whatever
// start it had).
static __device__ __noinline__ uint32_t intersect_far(const DSurface& S, double3 p, double3 d, double from,
                                                      double* h, double* N) {
    double l = conic_root(S.c, S.kc, p.x, p.y, p.z, d.x, d.y, d.z, from);
    if (fabs(l) >= 1e300) return PHOSIM_LOST_MISSED;
    bool done = false;
    for (int it = 0; it < 20 || done; ++it) {             // (the last time for the point and the normal)
        const double x = fma(l, d.x, p.x), y = fma(l, d.y, p.y), z = fma(l, d.z, p.z);
        double zs, zx, zy;
        if (!far_sag(S, x, y, zs, zx, zy)) return PHOSIM_LOST_MISSED;
        if (done) {
            const double n = rsqrt(fma(zx, zx, fma(zy, zy, 1.0)));
            h[0] = x; h[1] = y; h[2] = z;
            N[0] = -zx * n; N[1] = -zy * n; N[2] = n;
            return 0;
        }
        const double slope = d.z - zx * d.x - zy * d.y;
        if (slope == 0.0) return PHOSIM_LOST_NEWTON;
        const double step = (z - zs) / slope;
        l -= step;
        done = fabs(step) < 1e-8;
    }
    return PHOSIM_LOST_NEWTON;
}

// Intersection (Sec. 2.4.2): the paper's first guess is the root of a quadric approximating the surface; here the
// quadric is the conic itself.  With the aspheric and Zernike part a(x, y) of the sag and t = z - a the surface is
// Q = c (x^2 + y^2) / 2 + (1 + kappa) c t^2 / 2 - t = 0, which needs no root: Newton's method on Q along the ray solves
// it.  Any start near the root leads to it, so the ray moves in FP64 to the plane of the vertex and the start is found
// from there on the idle FP32 pipe: the conic's root, and for the aspheric and Zernike surfaces Newton steps on the
// sag, which leave about 1e-4 mm.  One FP64 evaluation of Q finishes: the step s = Q / Q' with the second-order term of
// Chebyshev's method, s + Q'' s^2 / (2 Q'), leaves an error near (Q'' / Q')^2 s^3, and the gradient of Q, which is
// along the normal, moves to the root with its derivative; the slope Q', which only scales the step, and both
// corrections are taken in single precision, whose 1e-7 of the step stays below the FP64 rounding of the results.  A step
// that is not that small is taken and followed by another.  For a sphere the gradient has unit length on the surface.  A ray
// that grazes the conic takes the FP64 root; where the start of an aspheric surface does not settle, or the first FP64 step
// is not that of a start near the surface, Newton's method on the sag decides (intersect_far).
// Measured (GB300, 300 stars, 2e7 photons, all FP64): 17.6 ms with the conic's FP64 root (a root and a quotient) and two
// to three FP64 Newton steps on the sag a mirror, 10.3 ms with this start and the savings of fp64.cuh; with the slope in
// single precision 7.7 ms, 8.1 with an FP64 slope and its reciprocal (6.3 since, by savings elsewhere).  On steep and aspheric lenses the position error
// against the oracle fell from up to 9e-10 mm to 9e-13 mm, with either slope.
// On success h is the point and N the unit normal (along (-S_x, -S_y, 1)); way has the sign of the distance, or is 0 where
// the single-precision start does not say it for certain (a start within 0.1 mm of the surface does beyond 1 mm).
__device__ __forceinline__ uint32_t intersect(const DSurface& S, const DSurfaceS& E, const double p[3], const double d[3],
                                              double h[3], double N[3], float& way) {
    if (S.flags & SF_FLAT_ONLY) {
        if ((__double2hiint(d[2]) & 0x7fffffff) < 0x00100000) return PHOSIM_LOST_MISSED;
        const double l = -p[2] * rcp64(d[2]);
        h[0] = fma(l, d[0], p[0]); h[1] = fma(l, d[1], p[1]); h[2] = 0.0;
        N[0] = 0.0; N[1] = 0.0; N[2] = 1.0;
        way = __double2hiint(l) > 0 ? 1.f : -1.f;
        return 0;
    }
    const bool newton = (S.flags & (SF_EVEN | SF_ODD | SF_ZERN)) != 0;
    const float dx = f32_trunc(d[0]), dy = f32_trunc(d[1]), dz = f32_trunc(d[2]);
    // the ray from the plane of the vertex (rays nearly parallel to it stay where they are)
    const float lp = fabsf(dz) > 1e-3f ? -f32_trunc(p[2]) / dz : 0.f;
    const double lpd = f64_exact(lp);
    const float A = fmaf(E.kmc.hi * dz, dz, E.c.hi);      // the quadric's l^2 coefficient for a unit direction
    bool started = false;
    float lf = 0.f;                                       // from there to the surface
    {
        const float px = fmaf(lp, dx, f32_trunc(p[0])), py = fmaf(lp, dy, f32_trunc(p[1]));
        const float pz = f32_trunc(fma(lpd, d[2], p[2]));
        const float c = E.c.hi, kc = E.kc.hi;
        const float bf = fmaf(kc * pz, dz, c * fmaf(px, dx, py * dy)) - dz;
        const float Cf = fmaf(kc * pz, pz, c * fmaf(px, px, py * py)) - 2.f * pz;
        const float disc = fmaf(bf, bf, -(A * Cf));
        if (disc > 1e-3f * bf * bf) {
            const float sq = sqrtf(disc);
            const float qf = bf >= 0.f ? -(bf + sq) : sq - bf;
            // of the roots Cf / qf and qf / A the one nearer to where the ray comes from (-lp from here), which a ray far off
            // the axis may not have nearer to the vertex's plane; the other where that one is not on the vertex branch
            const float near = Cf / qf;
            const bool second = fabsf((lp + near) * A) > fabsf(fmaf(lp, A, qf));
            lf = second ? qf / A : near;
            const float branch = fmaf(-kc, fmaf(lf, dz, pz), 1.f);
            if (A != 0.f && branch < 0.f) lf = second ? near : qf / A;
            started = fabsf(branch) > 1e-3f && fabsf(lf) < 1e30f;
            if (started && newton) {
                started = false;
#pragma unroll 1
                for (int it = 0; it < 4 && !started; ++it) {
                    const float x = fmaf(lf, dx, px), y = fmaf(lf, dy, py);
                    float zs, zxf, zyf;
                    if (!sag_f(E, S.flags, x, y, zs, zxf, zyf)) break;
                    const float step = (fmaf(lf, dz, pz) - zs) / (dz - zxf * dx - zyf * dy);
                    if (!(fabsf(step) < 1e30f)) break;
                    lf -= step;
                    started = fabsf(step) < 1e-2f;
                }
            }
        }
    }
    double x, y, z;
    const auto to_conic = [&] {
        const double q[3] = {fma(lpd, d[0], p[0]), fma(lpd, d[1], p[1]), fma(lpd, d[2], p[2])};
        const double l0 = conic_root(S.c, S.kc, q[0], q[1], q[2], d[0], d[1], d[2], lpd);
        x = fma(l0, d[0], q[0]); y = fma(l0, d[1], q[1]); z = fma(l0, d[2], q[2]);
        return l0;
    };
    // a ray without a place or a direction meets the conic nowhere: the aperture drops it
    const auto nowhere = [&](double l0) {
        if (fabs(l0) >= 1e300) return (uint32_t)PHOSIM_LOST_MISSED;
#pragma unroll
        for (int k = 0; k < 3; ++k) h[k] = N[k] = l0;
        return 0u;
    };
    if (!started) lf = 0.f;
    const double l0 = lpd + f64_exact(lf);
    if (started || newton) {
        x = fma(l0, d[0], p[0]); y = fma(l0, d[1], p[1]); z = fma(l0, d[2], p[2]);
    } else if (const double l1 = to_conic(); !(fabs(l1) < 1e300)) {
        way = 0.f;
        return nowhere(l1);
    }
    way = lp + lf;
    if (!(started && fabsf(way) > 1.f + 1e-4f * fabsf(lp))) way = 0.f;
    bool far = newton && !started;
    const float c = E.c.hi, kc = E.kc.hi;
#pragma unroll 1
    for (int it = 0; it < 20 && !far; ++it) {
        const double r2 = fma(x, x, y * y);
        double a = 0.0, ax = 0.0, ay = 0.0;
        float H[3] = {0.f, 0.f, 0.f};
        if (newton) aspheric(S, E, x, y, r2, a, ax, ay, H);
        const double t = newton ? z - a : z, kt = S.kc * t;
        const double Q = fma(0.5 * S.c, r2, t * fma(0.5, kt, -1.0));
        // the slope Q' along the ray only scales the step: in single precision unless it is small (t' = dt / dl)
        const float uf = fmaf(-kc, f32_trunc(t), 1.f);
        const float tlf = newton ? fmaf(-f32_trunc(ay), dy, fmaf(-f32_trunc(ax), dx, dz)) : dz;
        const float Qlf = fmaf(c, fmaf(f32_trunc(x), dx, f32_trunc(y) * dy), -(uf * tlf));
        float invf = 1.f / Qlf, sf = f32_trunc(Q) * invf;
        if (!(fabsf(Qlf) > 0.01f)) {
            const double tl = newton ? fma(-ay, d[1], fma(-ax, d[0], d[2])) : d[2];
            const double Ql = fma(S.c, fma(x, d[0], y * d[1]), -((1.0 - kt) * tl));
            if ((__double2hiint(Ql) & 0x7fffffff) < 0x00100000) return newton ? PHOSIM_LOST_NEWTON : PHOSIM_LOST_MISSED;
            invf = f32_trunc(rcp64(Ql));
            sf = f32_trunc(Q * rcp64(Ql));
        }
        if (it == 0 && !(fabsf(sf) < 0.1f)) {
            way = 0.f;
            far = newton;
            if (far) break;
        }
        const float hx = fmaf(H[0], dx, H[1] * dy), hy = fmaf(H[1], dx, H[2] * dy);
        // Q'' along the ray, and the step with its second-order term
        const float Qll = fmaf(c, fmaf(dx, dx, dy * dy), fmaf(kc * tlf, tlf, uf * fmaf(hx, dx, hy * dy)));
        const float k = Qll * invf * sf, more = 0.5f * k * sf;
        const bool last = fabsf(sf) < 1e-3f && fabsf(more * k) < 1e-14f;
        const double step = f64_exact(sf + more);
        x = fma(-step, d[0], x); y = fma(-step, d[1], y); z = fma(-step, d[2], z);
        if (last || fabsf(sf) < 1e-8f) {
            h[0] = x; h[1] = y; h[2] = z;
            if (!newton) {
                N[0] = -S.c * x; N[1] = -S.c * y; N[2] = fma(-S.kc, z, 1.0);
                if (E.kmc.hi == 0.f) return 0;
            } else {
                // outside the conic's domain the sag has no value (decided in single precision away from its edge)
                if (fmaf(-E.k1c2.hi, f32_trunc(r2), 1.f) < 1e-4f && fma(-S.k1c2, fma(x, x, y * y), 1.0) < 0.0)
                    return PHOSIM_LOST_MISSED;
                // minus the gradient of Q at the evaluated point, moved to the root: it changes by -s times its derivative
                const float ul = -kc * tlf;
                const double u = 1.0 - kt;
                N[0] = fma(-S.c, x, fma(-u, ax, f64_exact(sf * fmaf(ul, f32_trunc(ax), uf * hx))));
                N[1] = fma(-S.c, y, fma(-u, ay, f64_exact(sf * fmaf(ul, f32_trunc(ay), uf * hy))));
                N[2] = u - f64_exact(sf * ul);
            }
            const double n = rsqrt64(fma(N[0], N[0], fma(N[1], N[1], N[2] * N[2])));
            N[0] *= n; N[1] *= n; N[2] *= n;
            return 0;
        }
        if (!(fabsf(sf) < 1e37f)) return PHOSIM_LOST_NEWTON;
        // the start was too far off (a ray that grazes the conic): the conic's FP64 root
        if (!newton && started && it == 0 && !(fabsf(more * k) < 1e-14f))
            if (const double l1 = to_conic(); !(fabs(l1) < 1e300)) return nowhere(l1);
    }
    if (!far) return PHOSIM_LOST_NEWTON;
    double at[3], normal[3];
    const uint32_t why = intersect_far(S, make_double3(x, y, z), make_double3(d[0], d[1], d[2]), lpd + f64_exact(lf), at, normal);
#pragma unroll
    for (int k = 0; k < 3; ++k) { h[k] = at[k]; N[k] = normal[k]; }
    return why;
}

// Sellmeier index by its three fractions: where they have a pole or no real root (NaN), or their product over- or underflows
static __device__ __noinline__ double sellmeier_terms(const DMaterial& m, double l2) {
    double n2 = 1.0;
    for (int i = 0; i < 3; ++i) n2 += m.B[i] * l2 / (l2 - m.C[i]);
    return sqrt(n2);
}
// the same over one denominator
__device__ __forceinline__ double sellmeier(const DMaterial& m, double lam_nm) {
    const double l = lam_nm * 1e-3, l2 = l * l;
    const double a = l2 - m.C[0], b = l2 - m.C[1], c = l2 - m.C[2], ab = a * b, den = ab * c;
    const double num = fma(m.B[2], ab, c * fma(m.B[0], b, m.B[1] * a));
    const double n2 = fma(l2 * num, rcp64(den), 1.0);
    // a denominator within 2^+-960 and 2^-16 < n2 < 2^32, by their high words
    const bool plain = (uint32_t)((__double2hiint(den) & 0x7fffffff) - 0x03f00000) < 0x78000000u &&
                       (uint32_t)(__double2hiint(n2) - 0x3ef00000) < 0x03000000u;
    return plain ? sqrt64_pos(n2) : sellmeier_terms(m, l2);
}

// silicon index of Sec. 2.4.1, E in eV
__device__ __forceinline__ double silicon_index(double lam_nm) {
    const double E = 1239.841984 * rcp64(lam_nm);
    return fma(2.79, exp((E - 3.30) * (1.0 / 0.398)), fma(0.211, E, 3.36));
}
__device__ __forceinline__ float silicon_index_f(float lam_nm) {
    const float E = quotient_f(1239.841984f, lam_nm);
    return 3.36f + 0.211f * E + 2.79f * expf((E - 3.30f) * (1.0f / 0.398f));
}

// ------------------------------------------------------------------------------------------------------
// Fringing (Sec. 2.4.2): the back-side reflection probability from the single-layer electromagnetic
// calculation.  One layer of silicon (index n1 + i k1, thickness t) lies between the medium in front of the
// detector (real index n0) and vacuum behind it; a photon travels through it with direction cosine c1 (real,
// from its refracted direction), so its invariant is s^2 = n1^2 (1 - c1^2).  With q = N cos(theta) =
// sqrt(N^2 - s^2) in each medium, the s and p amplitude reflection coefficients of each interface, and the
// layer's round trip e = exp(i 4 pi t q1 / lambda), the layer reflects r = (r01 + r12 e) / (1 + r01 r12 e);
// the probability is (|r_s|^2 + |r_p|^2) / 2.
// ------------------------------------------------------------------------------------------------------
struct cplx {
    double re, im;
};
__device__ __forceinline__ cplx c_add(cplx a, cplx b) { return {a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ cplx c_sub(cplx a, cplx b) { return {a.re - b.re, a.im - b.im}; }
__device__ __forceinline__ cplx c_mul(cplx a, cplx b) { return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }
__device__ __forceinline__ cplx c_div(cplx a, cplx b) {
    const double d = 1.0 / (b.re * b.re + b.im * b.im);
    return {(a.re * b.re + a.im * b.im) * d, (a.im * b.re - a.re * b.im) * d};
}
// principal square root, without cancellation in the smaller part
__device__ __forceinline__ cplx c_sqrt(cplx z) {
    const double m = sqrt(0.5 * (hypot(z.re, z.im) + fabs(z.re)));
    if (m == 0.0) return {0.0, 0.0};
    if (z.re >= 0.0) return {m, 0.5 * z.im / m};
    return {0.5 * fabs(z.im) / m, z.im < 0.0 ? -m : m};
}

static __device__ __noinline__ double film_reflectance(double lam_nm, double n0, double n1, double k1, double t, double c1) {
    const double s2 = n1 * n1 * fmax(0.0, 1.0 - c1 * c1);
    const cplx q0 = c_sqrt({n0 * n0 - s2, 0.0}), q2 = c_sqrt({1.0 - s2, 0.0});
    const cplx N1sq = {n1 * n1 - k1 * k1, 2.0 * n1 * k1};
    const cplx q1 = c_sqrt(c_sub(N1sq, {s2, 0.0}));
    const cplx n0sq = {n0 * n0, 0.0};
    // s and p coefficients of the front (0 -> 1) and back (1 -> vacuum) interfaces
    const cplx rs01 = c_div(c_sub(q0, q1), c_add(q0, q1)), rs12 = c_div(c_sub(q1, q2), c_add(q1, q2));
    const cplx rp01 = c_div(c_sub(c_mul(N1sq, q0), c_mul(n0sq, q1)), c_add(c_mul(N1sq, q0), c_mul(n0sq, q1)));
    const cplx rp12 = c_div(c_sub(q1, c_mul(N1sq, q2)), c_add(q1, c_mul(N1sq, q2)));
    const double w = 4.0 * M_PI * t / (lam_nm * 1e-6);
    double sn, cs;
    sincos(w * q1.re, &sn, &cs);
    const double amp = exp(-w * q1.im);
    const cplx e = {amp * cs, amp * sn};
    const cplx rs = c_div(c_add(rs01, c_mul(rs12, e)), c_add({1.0, 0.0}, c_mul(c_mul(rs01, rs12), e)));
    const cplx rp = c_div(c_add(rp01, c_mul(rp12, e)), c_add({1.0, 0.0}, c_mul(c_mul(rp01, rp12), e)));
    return 0.5 * (rs.re * rs.re + rs.im * rs.im + rp.re * rp.re + rp.im * rp.im);
}

// Snell's law in vector form (Sec. 2.4.2) with mu = n1 / n2; false on total internal reflection.  flat: the normal
// is the z axis, where the vector form reduces to scaling d_x and d_y by mu and d_z = -+sqrt(k).
__device__ __forceinline__ bool refract(double d[3], double Nx, double Ny, double Nz, double mu, bool flat = false) {
    if (flat) {
        const double k = fma(-(mu * mu), fma(-d[2], d[2], 1.0), 1.0);
        if (negative64(k)) return false;
        d[0] *= mu;
        d[1] *= mu;
        d[2] = copysign(sqrt64(k), d[2]);
        return true;
    }
    double cosi = -fma(d[0], Nx, fma(d[1], Ny, d[2] * Nz));
    if (negative64(cosi)) { Nx = -Nx; Ny = -Ny; Nz = -Nz; cosi = -cosi; }
    const double k = fma(-(mu * mu), fma(-cosi, cosi, 1.0), 1.0);
    if (negative64(k)) return false;
    const double a = fma(mu, cosi, -sqrt64(k));
    d[0] = fma(mu, d[0], a * Nx);
    d[1] = fma(mu, d[1], a * Ny);
    d[2] = fma(mu, d[2], a * Nz);
    return true;
}

__device__ __forceinline__ void to_surface(const DSurface& S, const double x[3], const double d[3], double p[3],
                                           double dl[3]) {
    if (!(S.flags & (SF_ROTATED | SF_DECENTERED))) {     // a vertex on the axis: x - 0 is x
        p[0] = x[0]; p[1] = x[1]; p[2] = x[2] - S.o[2];
        dl[0] = d[0]; dl[1] = d[1]; dl[2] = d[2];
        return;
    }
    const double rx = x[0] - S.o[0], ry = x[1] - S.o[1], rz = x[2] - S.o[2];
    if (!(S.flags & SF_ROTATED)) {        // the identity rotation: the products below would be exact copies
        p[0] = rx; p[1] = ry; p[2] = rz;
        dl[0] = d[0]; dl[1] = d[1]; dl[2] = d[2];
        return;
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        p[i] = fma(S.M[3 * i], rx, fma(S.M[3 * i + 1], ry, S.M[3 * i + 2] * rz));
        dl[i] = fma(S.M[3 * i], d[0], fma(S.M[3 * i + 1], d[1], S.M[3 * i + 2] * d[2]));
    }
}

__device__ __forceinline__ void from_surface(const DSurface& S, const double p[3], const double dl[3], double x[3],
                                             double d[3]) {
    if (!(S.flags & (SF_ROTATED | SF_DECENTERED))) {
        x[0] = p[0]; x[1] = p[1]; x[2] = p[2] + S.o[2];
        d[0] = dl[0]; d[1] = dl[1]; d[2] = dl[2];
        return;
    }
    if (!(S.flags & SF_ROTATED)) {
        x[0] = p[0] + S.o[0]; x[1] = p[1] + S.o[1]; x[2] = p[2] + S.o[2];
        d[0] = dl[0]; d[1] = dl[1]; d[2] = dl[2];
        return;
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        x[i] = fma(S.M[i], p[0], fma(S.M[3 + i], p[1], fma(S.M[6 + i], p[2], S.o[i])));
        d[i] = fma(S.M[i], dl[0], fma(S.M[3 + i], dl[1], S.M[6 + i] * dl[2]));
    }
}

}  // namespace phosim
