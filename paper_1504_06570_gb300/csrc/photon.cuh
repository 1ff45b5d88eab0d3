// Per-photon forward path shared by the trace kernel and the adjoint kernel (Peterson et al. 2015,
// Sec. 2.2-2.5): one definition, so the adjoint's recomputed forward pass takes exactly the trace's
// decisions.
#pragma once

#include "phosim_device.cuh"

namespace phosim {


struct PhotonOut {
    double x, y, xc, yc, lam;
    uint32_t flags;
    int pix;
};

__device__ __forceinline__ uint32_t lost(uint32_t reason, int surface) {
    return (reason << 8) | ((uint32_t)(surface & 0xff) << 16);
}

__device__ __forceinline__ uint32_t word(const uint4& w, int k) {
    return k == 0 ? w.x : (k == 1 ? w.y : (k == 2 ? w.z : w.w));
}

// Wavelength bin (Sec. 2.2): the first bin whose cumulative photon probability exceeds the draw, decided
// on the integer draw against thresholds precomputed from the FP64 cumulative table.  A guide table (Chen and
// Asau's indexed search) narrows the search to the thresholds between guide[j] and guide[j + 1] for the draw's
// top byte j: every threshold below guide[j] is at most j 2^24 <= w, and the one at guide[j + 1] exceeds
// (j + 1) 2^24 > w, so the answer lies in that range and is the plain search's answer.
__device__ __forceinline__ int sed_bin(const unsigned long long* __restrict__ thr, const int* __restrict__ guide, uint32_t w) {
    const int j = (int)(w >> 24);
    int lo = __ldg(guide + j), hi = __ldg(guide + j + 1);
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if ((unsigned long long)w < __ldg(thr + mid)) hi = mid;
        else lo = mid + 1;
    }
    return lo;
}

__device__ __forceinline__ int wrap_index(long long i, int n) {
    if ((n & (n - 1)) == 0) return (int)(i & (long long)(n - 1));
    long long m = i % n;
    return (int)(m < 0 ? m + n : m);
}

// A node's 2 x 2 block in one or two 32-byte loads.  Lookups share few lines, so they leave the L1 alone, and a fetch
// from memory takes two sectors instead of four: the entry stage's reads of a 1e8-photon field fell from 16.2 to 8.3 GB
// (3.28 to 3.20 ms; two 16-byte loads a block: 3.30 ms).
__device__ __forceinline__ void load_block(const float4* p, float4& A, float4& B) {
    asm("ld.global.nc.L1::no_allocate.L2::64B.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(A.x), "=f"(A.y), "=f"(A.z), "=f"(A.w), "=f"(B.x), "=f"(B.y), "=f"(B.z), "=f"(B.w)
        : "l"(p));
}
__device__ __forceinline__ void load_block(const double2* p, double2& a, double2& b, double2& c, double2& d) {
    asm("ld.global.nc.L1::no_allocate.L2::64B.v4.f64 {%0, %1, %2, %3}, [%4];"
        : "=d"(a.x), "=d"(a.y), "=d"(b.x), "=d"(b.y) : "l"(p));
    asm("ld.global.nc.L1::no_allocate.L2::64B.v4.f64 {%0, %1, %2, %3}, [%4];"
        : "=d"(c.x), "=d"(c.y), "=d"(d.x), "=d"(d.y) : "l"(p + 2));
}

__device__ __forceinline__ int near_index(int i, int n) {
    if ((n & (n - 1)) == 0) return i & (n - 1);
    const int m = i % n;
    return m < 0 ? m + n : m;
}

// A screen coordinate's node and the fraction of a pixel from it, s k - floor(s k).  By integers, on pipes that idle (with
// the product, its floor and the rest on the FP64 pipe 2e7 photons took 7.73 ms all FP64 and 1.5e7 took 4.65 mixed, 7.12
// and 4.33 so); a coordinate beyond 4 km in FP64, from the rounded product, whose last places are all that is left of the
// fraction far out; one that is no number has no fraction (kNoFraction).
static __device__ __noinline__ int far_node(double s, double inv, int n, unsigned long long& frac) {
    const double f = s * inv, fl = floor(f), rest = f - fl;
    frac = isnan(rest) ? kNoFraction : (unsigned long long)fmin(rest * 4503599627370496.0, 4503599627370495.0);
    return wrap_index((long long)fl, n);
}
__device__ __forceinline__ int node_of(const DScale& S, double s, unsigned long long& frac) {
    int i;
    if (!split_product64(s, S.inv_m, S.inv_shift, i, frac)) return far_node(s, S.inv_pix, S.n, frac);
    return near_index(i, S.n);
}

// Gradient of the phase at screen position (sx, sy), bilinear between central-difference nodes (Sec. 2.3.2), added to
// (gx, gy) or, for the first scale, in their place
template <bool MIXED, bool FIRST>
__device__ __forceinline__ void screen_gradient(const DScale& S, double sx, double sy, double& gx, double& gy) {
    const int n = S.n;
    unsigned long long u, v;
    const int i0 = node_of(S, sx, u), j0 = node_of(S, sy, v);
    const size_t node = (size_t)j0 * n + i0;
    if constexpr (MIXED) {
        const float fx = fraction_f32(u), fy = fraction_f32(v);
        float4 A, B;
        load_block(S.g32 + 2 * node, A, B);
        const float w00 = (1.f - fx) * (1.f - fy), w10 = fx * (1.f - fy), w01 = (1.f - fx) * fy, w11 = fx * fy;
        const double ax = f64_any(w00 * A.x + w10 * A.z + w01 * B.x + w11 * B.z);
        const double ay = f64_any(w00 * A.y + w10 * A.w + w01 * B.y + w11 * B.w);
        gx = FIRST ? ax : gx + ax;
        gy = FIRST ? ay : gy + ay;
    } else {
        const double tx = one_and_fraction64(u), ty = one_and_fraction64(v);
        double2 a, b, c, d;
        load_block(S.g64 + 4 * node, a, b, c, d);
        const double ax = fma(ty, fma(tx, d.x, c.x), fma(tx, b.x, a.x)), ay = fma(ty, fma(tx, d.y, c.y), fma(tx, b.y, a.y));
        gx = FIRST ? ax : gx + ax;
        gy = FIRST ? ay : gy + ay;
    }
}

// 1 / |n_z| = (1 - q)^(-1/2) of a unit direction, q = n_x^2 + n_y^2: within half a degree of the axis (q < 1e-4) the
// series to q^3, which leaves 35 q^4 / 128 < 3e-17
__device__ __forceinline__ double inverse_nz(double nx, double ny) {
    const double q = fma(nx, nx, ny * ny);
    if (__double2hiint(q) < 0x3f1a36e2) return fma(q, fma(q, fma(q, 0.3125, 0.375), 0.5), 1.0);
    return rsqrt64(1.0 - q);
}

__device__ __forceinline__ double lerp_table(const double* __restrict__ t, int n, double f) {
    int k = 0;
    double fl = 0.0;
    const bool found = floor_product64(f, 1.0, fl, k);
    double w = f - fl;
    if (!found || k < 0 || k > n - 2) {              // off the table: its first or last value, none where f is no number
        const bool last = found ? k > 0 : f > 0.0;
        k = last ? n - 2 : 0;
        w = isnan(f) ? f : last ? 1.0 : 0.0;
    }
    const double a = __ldg(t + k);
    return fma(w, __ldg(t + k + 1) - a, a);
}
__device__ __forceinline__ float lerp_table_f(const float* __restrict__ t, int n, float f) {
    int k = (int)floorf(f);
    k = k < 0 ? 0 : (k > n - 2 ? n - 2 : k);
    float w = f - (float)k;
    w = w < 0.f ? 0.f : (w > 1.f ? 1.f : w);
    return __ldg(t + k) * (1.f - w) + __ldg(t + k + 1) * w;
}

// Surfaces in order (Sec. 2.4.2).  FULL = apertures, coatings and the sensor; otherwise the bare rays that
// give each source's chief-ray reference.
// Forward state kept for the adjoint sweep (RECORD): at each surface from the tape's first on, in its frame, the hit point,
// the direction before it, the distance travelled to it, the normal and (refracting surfaces, the sensor) the index ratio
// n1 / n2; and the conversion length of the sensor, the final position and whether the photon was detected.  A warp's
// records are words of its 32 lanes side by side (BatchList).
struct ForwardRecord {
    double* w;                    // this lane's first word
    int first, n_surf;
    __device__ __forceinline__ double* surface(int si) const { return w + (size_t)(kTapeSurface * (si - first)) * 32; }
    __device__ __forceinline__ double* end() const { return surface(n_surf); }
};
__device__ __forceinline__ ForwardRecord forward_record(const TraceParams& P, const BatchList& L, unsigned long long slot, int lane) {
    return {L.tape + slot * L.tape_stride + lane, L.tape_first, P.n_surf};
}

// A photon of a bundle (Sec. 3.2 background optimisation): it follows its ray (the photon index divided by
// the bundle size) to the detector surface, lands at a Gaussian offset of the source's spread sigma from the
// ray's hit and takes its own sensor draws, all from blocks 5 and 6 of its own counter.
struct MemberDraw {
    double sx, sy;
    uint32_t conv, diff_a, diff_b, back;
};

template <bool MIXED>
__device__ __forceinline__ MemberDraw member_draw(const TraceParams& P, double bsig, int src, uint64_t i) {
    const uint32_t clo = (uint32_t)i, chi = (uint32_t)(i >> 32);
    const uint4 m5 = philox(make_uint4(clo, chi, (uint32_t)src, 5u), P.k0, P.k1);
    const uint4 m6 = philox(make_uint4(clo, chi, (uint32_t)src, 6u), P.k0, P.k1);
    MemberDraw m;
    if constexpr (MIXED) {
        const float g = sqrtf(-2.f * logf(u32of(m5.x)));
        float sn, cs;
        sincospif(2.f * u32of(m5.y), &sn, &cs);
        m.sx = (double)((float)bsig * g * cs);
        m.sy = (double)((float)bsig * g * sn);
    } else {
        const double g = sqrt64_pos(-2.0 * log_draw64(P.draw_table, m5.x));
        double sn, cs;
        sincos_draw64(P.draw_table, m5.y, sn, cs);
        m.sx = bsig * g * cs;
        m.sy = bsig * g * sn;
    }
    m.conv = m5.z; m.diff_a = m5.w; m.diff_b = m6.x; m.back = m6.y;
    return m;
}

// the ray a photon follows: itself, or for a bundle of n photons per ray, photon index / n
__device__ __forceinline__ uint64_t ray_of(uint32_t bundle, uint64_t i) { return bundle > 1 ? i / bundle : i; }

// Ghosts (Sec. 2.4.2): after a photon's first reflection by a coating, each coating decision draws the next
// word of blocks 7, 8, ... of the ray's counter.
__device__ __forceinline__ uint32_t ghost_word(const TraceParams& P, int src, uint64_t ray, int n) {
    return word(philox(make_uint4((uint32_t)ray, (uint32_t)(ray >> 32), (uint32_t)src, 7u + (uint32_t)n / 4u), P.k0, P.k1),
                n & 3);
}

// Surfaces in order (dir = +1); with reflecting coatings a photon reflected by a refracting surface (a ghost)
// travels back through them (dir = -1) until another reflection turns it round again.  src and ray identify
// the ghost draws.
template <bool MIXED, bool FULL, bool RECORD = false>
__device__ __forceinline__ void optics(const TraceParams& P, double X[3], double D[3], double lam, uint4 w1, uint4 w2,
                                       uint4 w3, uint4 w4, PhotonOut& R, ForwardRecord* fr = nullptr,
                                       const MemberDraw* mb = nullptr, int src = 0, uint64_t ray = 0) {
    constexpr bool GHOSTS = FULL && !RECORD;
    const bool ghosts = GHOSTS && (P.flags & kGhostFlag);
    double n_cur = 1.0;
    int glass_mat = -1;
    double glass_n = 1.0, glass_inv = 1.0;
    int si = 0, dir = 1, bounces = 0, n_ghost = 0;
#pragma unroll 1
    for (;;) {
        if (si < 0 || si >= P.n_surf) break;
        const DSurface& S = P.surf[si];
        double p[3], dl[3];
        to_surface(S, X, D, p, dl);
        double h[3], Nv[3];
        float way;
        const uint32_t why = intersect(S, P.surf_s[si], p, dl, h, Nv, way);
        if (why) { R.flags = lost(why, si); return; }
        // a ghost only meets surfaces ahead of it: a distance near 0 from the points, to their FP64 rounding (for every
        // distance that took 2 % of 2.8e6 photons with ghosts, mixed: 21.0 ms)
        if (GHOSTS && bounces > 0 &&
            !(way != 0.f ? way > 0.f : fma(h[0] - p[0], dl[0], fma(h[1] - p[1], dl[1], (h[2] - p[2]) * dl[2])) > 0.0)) {
            R.flags = lost(PHOSIM_LOST_MISSED, si);
            return;
        }
        if constexpr (RECORD) {
            if (si >= fr->first) {
                double* q = fr->surface(si);
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    q[32 * (kTapeH + k)] = h[k];
                    q[32 * (kTapeD + k)] = dl[k];
                    q[32 * (kTapeN + k)] = Nv[k];
                }
                q[32 * kTapeL] = fma(h[0] - p[0], dl[0], fma(h[1] - p[1], dl[1], (h[2] - p[2]) * dl[2]));
            }
        }
        p[0] = h[0]; p[1] = h[1]; p[2] = h[2];
        const bool flat = (S.flags & SF_FLAT_ONLY) != 0;
        const double Nx = Nv[0], Ny = Nv[1], Nz = Nv[2];
        if (S.kind == PHOSIM_DETECTOR) {
            uint32_t w_conv = w1.w, w_diff_a = w2.x, w_diff_b = w2.y, w_back = w4.z;
            if (mb) {   // a bundle's photon: its offset from the ray's hit and its own sensor draws
                p[0] += mb->sx;
                p[1] += mb->sy;
                w_conv = mb->conv; w_diff_a = mb->diff_a; w_diff_b = mb->diff_b; w_back = mb->back;
            }
            const double hx = p[0] - P.xlo, hy = p[1] - P.ylo;
            if (FULL && !(within64(hx, P.chip_w) && within64(hy, P.chip_h))) {
                R.flags = lost(PHOSIM_LOST_OFF_CHIP, si);
                return;
            }
            double fx = p[0], fy = p[1];
            R.xc = fx; R.yc = fy;
            if (FULL && (P.flags & PHOSIM_SENSOR)) {
                // refraction into the silicon, exponential conversion length (Sec. 2.4.2)
                double L, sigma, gxd, gyd, r_back;
                if constexpr (MIXED) {
                    const float n_si = silicon_index_f((float)lam);
                    if (!refract(dl, Nx, Ny, Nz, n_cur * rcp64((double)n_si), flat)) { R.flags = lost(PHOSIM_LOST_TIR, si); return; }
                    const float ell = lerp_table_f(P.ell32, P.n_ell, (float)((lam - P.ell_lam0) * P.inv_ell_dlam));
                    const float Lf = ell * -logf(u32of(w_conv));
                    L = (double)Lf;
                    const float rf = (n_si - 1.f) / (n_si + 1.f);
                    r_back = (double)(rf * rf);
                } else {
                    const double n_si = silicon_index(lam), mu = n_cur * rcp64(n_si);
                    if constexpr (RECORD) fr->surface(si)[32 * kTapeMu] = mu;
                    if (!refract(dl, Nx, Ny, Nz, mu, flat)) { R.flags = lost(PHOSIM_LOST_TIR, si); return; }
                    const double ell = lerp_table(P.ell, P.n_ell, (lam - P.ell_lam0) * P.inv_ell_dlam);
                    L = ell * -log_draw64(P.draw_table, w_conv);
                    const double rf = (n_si - 1.0) / (n_si + 1.0);
                    r_back = rf * rf;
                }
                double depth = L * fabs(dl[2]);
                if (!(depth <= P.t_si)) {
                    // back-side reflection: the photon turns round at the back and converts on its way back
                    bool back = false;
                    if (P.flags & PHOSIM_BACK_REFLECT) {
                        if (P.flags & PHOSIM_FRINGE) {
                            // fringing: the single-layer calculation in FP64 at the photon's entry point (both
                            // the plain and the mixed path: the phase spans ~10^3 cycles)
                            const double ell = lerp_table(P.ell, P.n_ell, (lam - P.ell_lam0) * P.inv_ell_dlam);
                            r_back = film_reflectance(lam, n_cur, silicon_index(lam), lam * 1e-6 / (4.0 * M_PI * ell),
                                                      P.fr_t0 + P.fr_gx * p[0] + P.fr_gy * p[1], fabs(dl[2]));
                        }
                        if (u64of(w_back) < r_back) {
                            depth = 2.0 * P.t_si - depth;
                            back = depth >= 0.0;
                        }
                    }
                    if (!back) { R.flags = lost(PHOSIM_LOST_NOT_CONVERTED, si); return; }
                }
                // field-free dead layer at the entrance: the charge is not collected
                if (depth < P.dead_layer) { R.flags = lost(PHOSIM_LOST_DEAD_LAYER, si); return; }
                fx = fma(L, dl[0], fx);
                fy = fma(L, dl[1], fy);
                R.xc = fx; R.yc = fy;
                // lateral Gaussian diffusion (Sec. 2.5)
                if constexpr (MIXED) {
                    const float sg = lerp_table_f(P.sig32, P.n_sig, (float)(depth * P.sig_scale));
                    const float g = sqrtf(-2.f * logf(u32of(w_diff_a)));
                    float sn, cs;
                    sincospif(2.f * u32of(w_diff_b), &sn, &cs);
                    sigma = 1.0; gxd = (double)(sg * g * cs); gyd = (double)(sg * g * sn);
                } else {
                    sigma = lerp_table(P.sig, P.n_sig, depth * P.sig_scale);
                    const double g = sqrt64_pos(-2.0 * log_draw64(P.draw_table, w_diff_a));
                    double sn, cs;
                    sincos_draw64(P.draw_table, w_diff_b, sn, cs);
                    gxd = g * cs; gyd = g * sn;
                }
                fx = fma(sigma, gxd, fx);
                fy = fma(sigma, gyd, fy);
                if constexpr (RECORD) fr->end()[32 * kTapeDepth] = L;
            }
            R.x = fx; R.y = fy;
            if (FULL) {
                const double ux = fx - P.xlo, uy = fy - P.ylo;
                int px = -1, py = -1;
                double fl;
                floor_product64(ux, P.inv_pixel, fl, px);
                floor_product64(uy, P.inv_pixel, fl, py);
                if (!(px >= 0 && py >= 0 && px < P.nx && py < P.ny)) {
                    R.flags = lost(PHOSIM_LOST_OFF_CHIP, si);
                    return;
                }
                R.pix = py * P.nx + px;
            }
            R.flags = PHOSIM_F_DETECTED;
            return;
        }
        if (FULL) {
            // clear aperture
            // (decided in single precision unless the radius is within 1e-5, relative, of a bound)
            const float xf = f32_trunc(p[0]), yf = f32_trunc(p[1]), r2f = fmaf(xf, xf, yf * yf);
            const float ro = P.surf_s[si].r_out2.hi, ri = P.surf_s[si].r_in2.hi;
            bool clear = r2f <= ro && r2f >= ri;
            if (!(fabsf(r2f - ro) > 1e-5f * ro && fabsf(r2f - ri) > 1e-5f * ri)) {
                const double r2 = fma(p[0], p[0], p[1] * p[1]);
                clear = r2 <= S.r_out2 && r2 >= S.r_in2;
            }
            if (!clear) { R.flags = lost(PHOSIM_LOST_VIGNETTED, si); return; }
            // coating accept-reject at the incidence angle and wavelength.  A coating of one angle bin, without ghosts, has
            // decided in the dynamic transmission test (early_coating_reject: the same draw, bin and threshold).
            if (S.coat_slot >= 0 && !((P.flags & PHOSIM_EARLY_REJECT) && !ghosts && P.coat[S.coating].nt == 1)) {
                const DCoating& C = P.coat[S.coating];
                int it = 0;
                if (C.nt > 1) {
                    const double cosi = fabs(dl[0] * Nx + dl[1] * Ny + dl[2] * Nz);
                    const double th = acos(fmin(1.0, cosi));
                    it = (int)floor((th - C.th0) * C.inv_dth);
                    it = it < 0 ? 0 : (it > C.nt - 1 ? C.nt - 1 : it);
                }
                int il = __double2int_rd((lam - C.lam0) * C.inv_dlam);
                il = il < 0 ? 0 : (il > C.nl - 1 ? C.nl - 1 : il);
                const size_t ix = (size_t)il * C.nt + it;
                uint32_t w;
                if (GHOSTS && bounces > 0) {
                    w = ghost_word(P, src, ray, n_ghost++);
                } else {
                    const int k = S.coat_slot;
                    w = k < 2 ? word(w2, 2 + k) : word(w3, k - 2);
                }
                if (!((unsigned long long)w < __ldg(C.T_thr + ix))) {    // (w + 1/2) 2^-32 < T
                    // reflected backwards (a ghost) with probability R, absorbed otherwise
                    if (ghosts && S.kind != PHOSIM_MIRROR && C.TR_thr && (unsigned long long)w < __ldg(C.TR_thr + ix)) {
                        const double dn = dl[0] * Nx + dl[1] * Ny + dl[2] * Nz;
                        dl[0] = fma(-2.0 * dn, Nx, dl[0]);
                        dl[1] = fma(-2.0 * dn, Ny, dl[1]);
                        dl[2] = fma(-2.0 * dn, Nz, dl[2]);
                        dir = -dir;
                        if (++bounces > kMaxGhostBounces) { R.flags = lost(PHOSIM_LOST_MISSED, si); return; }
                        from_surface(S, p, dl, X, D);
                        si += dir;
                        continue;
                    }
                    R.flags = lost(PHOSIM_LOST_COATING, si);
                    return;
                }
            }
        }
        if (S.kind == PHOSIM_MIRROR) {
            const double dn = dl[0] * Nx + dl[1] * Ny + dl[2] * Nz;
            dl[0] = fma(-2.0 * dn, Nx, dl[0]);
            dl[1] = fma(-2.0 * dn, Ny, dl[1]);
            dl[2] = fma(-2.0 * dn, Nz, dl[2]);
        } else {
            // the medium beyond the surface in the direction of travel (-1: vacuum)
            const int mi = (GHOSTS && dir < 0) ? S.mat_before : S.material;
            double n_next = 1.0, inv_next = 1.0;
            if (mi >= 0) {
                const DMaterial& m = P.mat[mi];
                if (m.kind == PHOSIM_SELLMEIER) {
                    if (glass_mat != mi) {
                        glass_n = sellmeier(m, lam);
                        glass_inv = rcp64(glass_n);
                        glass_mat = mi;
                    }
                    n_next = glass_n;
                    inv_next = glass_inv;
                } else if (m.kind == PHOSIM_SILICON) {
                    n_next = silicon_index(lam);
                    inv_next = rcp64(n_next);
                }
            }
            const double mu = n_cur * inv_next;
            if constexpr (RECORD) {
                if (si >= fr->first) fr->surface(si)[32 * kTapeMu] = mu;
            }
            if (!refract(dl, Nx, Ny, Nz, mu, flat)) { R.flags = lost(PHOSIM_LOST_TIR, si); return; }
            n_cur = n_next;
        }
        from_surface(S, p, dl, X, D);
        si += dir;
    }
    R.flags = lost(PHOSIM_LOST_MISSED, si < 0 ? 0 : P.n_surf);
}

// Wavelength (Sec. 2.2): cumulative photon-number table, blur within the bin, redshift.  FP64 in both FP64-optics
// paths: the coating decisions bin it, and a single-precision wavelength would move about one photon in 5e6
// across a band edge of a filter (a form that blurred in FP32 took as many FP64-pipe operations, in its
// conversions, as this one).
template <bool MIXED>
__device__ __forceinline__ double sample_wavelength(const TraceParams& P, const DSource& s, const uint4& w0) {
    const int bin = sed_bin(P.thr + (size_t)s.sed * (P.n_bins - 1), P.sed_guide + (size_t)s.sed * (kSedGuide + 1), w0.z);
    return fma(u64of(w0.w), P.sed_dlam, fma(f64_of_count((uint32_t)bin), P.sed_dlam, P.sed_lam0)) * s.zfac;
}

// The wavelength-bin draws of a source that the dynamic transmission test may let pass, as one interval of the
// 32-bit draw: the draws of the bins that reach into [pass_lo, pass_hi).  A bin whose last wavelength (its blur draw is
// at most 1 - 2^-33) lies below pass_lo is left out, and so at the other end; delta is that distance in bins less the
// rounding of the wavelengths the paths compute (a double-single wavelength is off by 2^-46 at most).
template <class Params>
__device__ __forceinline__ void pass_draws(const Params& P, const DSource& s, uint32_t& w_lo, uint32_t& w_span) {
    const double scale = P.sed_dlam * s.zfac;
    const double x = (P.pass_lo / s.zfac - P.sed_lam0) / P.sed_dlam, y = (P.pass_hi / s.zfac - P.sed_lam0) / P.sed_dlam;
    const double last = fabs(P.sed_lam0 + P.n_bins * P.sed_dlam) + fabs(P.sed_lam0);
    const double delta = 1.16e-10 - 1e-12 - 8e-14 * last * s.zfac / scale;
    const int n = P.n_bins;
    const int k0 = (int)fmin(fmax(floor(x + delta), 0.0), (double)n);       // the first bin that may pass
    const int k1 = (int)fmin(fmax(ceil(y - delta), 0.0), (double)n);        // the first one past the last
    const unsigned long long* thr = P.thr + (size_t)s.sed * (n - 1);
    const unsigned long long lo = k0 == 0 ? 0ull : k0 == n ? 1ull << 32 : thr[k0 - 1];
    const unsigned long long hi = k1 == 0 ? 0ull : k1 == n ? 1ull << 32 : thr[k1 - 1];
    // no draw at all: one that the full test will stop
    w_lo = lo < hi ? (uint32_t)lo : 0u;
    w_span = lo < hi ? (uint32_t)(hi - lo - 1) : 0u;
}

// Dynamic transmission (Sec. 3.2): the index of the first coated surface whose accept draw is not below the
// largest transmission any incidence angle allows at this wavelength (the photon is certainly rejected
// there), or -1.
__device__ __forceinline__ int early_coating_reject(const TraceParams& P, double lam, const uint4& w2, const uint4& w3) {
    // with reflecting coatings only the first coated surface's draw is certain to be used (a ghost decides
    // later surfaces with its own words)
    const int nk = (P.flags & kGhostFlag) ? min(1, P.n_coated) : P.n_coated;
#pragma unroll 1
    for (int k = 0; k < nk; ++k) {
        const int si = P.coated_surface[k];
        const DCoating& C = P.coat[P.surf[si].coating];
        int il = __double2int_rd((lam - C.lam0) * C.inv_dlam);
        il = il < 0 ? 0 : (il > C.nl - 1 ? C.nl - 1 : il);
        const uint32_t w = k < 2 ? word(w2, 2 + k) : word(w3, k - 2);
        if (!((unsigned long long)w < __ldg(C.Tmax_thr + il))) return si;
    }
    return -1;
}

// The early-rejection decision of photon i alone (no propagation): -1 if it goes on, else the surface.
template <bool MIXED>
__device__ __forceinline__ int early_reject_surface(const TraceParams& P, const DSource& s, int src, uint64_t i,
                                                    double& lam) {
    i = ray_of(s.bundle, i);
    const uint32_t clo = (uint32_t)i, chi = (uint32_t)(i >> 32);
    const uint4 w0 = philox(make_uint4(clo, chi, (uint32_t)src, 0u), P.k0, P.k1);
    lam = sample_wavelength<MIXED>(P, s, w0);
    const uint4 w2 = philox(make_uint4(clo, chi, (uint32_t)src, 2u), P.k0, P.k1);
    uint4 w3 = make_uint4(0u, 0u, 0u, 0u);
    if (P.n_coated > 2) w3 = philox(make_uint4(clo, chi, (uint32_t)src, 3u), P.k0, P.k1);
    return early_coating_reject(P, lam, w2, w3);
}

// TESTED: the photon has passed the dynamic transmission test (or is not subject to it)
template <bool MIXED, bool RECORD = false, bool TESTED = false>
__device__ __forceinline__ void trace_photon(const TraceParams& P, const DSource& s, int src, uint64_t photon,
                                             PhotonOut& R, ForwardRecord* fr = nullptr) {
    const uint64_t i = ray_of(s.bundle, photon);
    const uint32_t clo = (uint32_t)i, chi = (uint32_t)(i >> 32);
    const uint4 w0 = philox(make_uint4(clo, chi, (uint32_t)src, 0u), P.k0, P.k1);
    const uint4 w1 = philox(make_uint4(clo, chi, (uint32_t)src, 1u), P.k0, P.k1);
    R.flags = 0; R.pix = -1; R.x = R.y = R.xc = R.yc = 0.0;
    // time stamp (Sec. 2.2)
    const double t = fma(s.t_exp, u64of(w1.x), s.t0);
    const double lam = sample_wavelength<MIXED>(P, s, w0);
    R.lam = lam;
    // direction: tangent-plane components, paraxial shape offset, renormalised (Sec. 2.2, 2.2.1)
    double nx = s.xi, ny = s.eta;
    if (s.kind == PHOSIM_SERSIC) {
        if constexpr (MIXED) {
            const float r = lerp_table_f(P.sersic32 + (size_t)s.table * P.sersic_K, P.sersic_K,
                                         u32of(w1.y) * (float)P.sersic_K - 0.5f);
            float sp, cp;
            sincospif(2.f * u32of(w1.z), &sp, &cp);
            const float dx = (float)s.a * r * cp, dy = (float)s.b * r * sp;
            nx += (double)(dx * (float)s.cpa - dy * (float)s.spa);
            ny += (double)(dx * (float)s.spa + dy * (float)s.cpa);
        } else {
            const double r = lerp_table(P.sersic + (size_t)s.table * P.sersic_K, P.sersic_K,
                                        u64of(w1.y) * P.sersic_K - 0.5);
            double sp, cp;
            sincos_draw64(P.draw_table, w1.z, sp, cp);
            const double dx = s.a * r * cp, dy = s.b * r * sp;
            nx += dx * s.cpa - dy * s.spa;
            ny += dx * s.spa + dy * s.cpa;
        }
    } else if (s.kind == PHOSIM_GAUSS) {
        if constexpr (MIXED) {
            const float g = sqrtf(-2.f * logf(u32of(w1.y)));
            float sp, cp;
            sincospif(2.f * u32of(w1.z), &sp, &cp);
            nx += (double)((float)s.a * g * cp);
            ny += (double)((float)s.a * g * sp);
        } else {
            const double g = sqrt64_pos(-2.0 * log_draw64(P.draw_table, w1.y));
            double sp, cp;
            sincos_draw64(P.draw_table, w1.z, sp, cp);
            nx += s.a * g * cp;
            ny += s.a * g * sp;
        }
    }
    // 1 / |n_z| = rsqrt(1 - n_x^2 - n_y^2): layer-to-layer distances are height differences times it
    double rinv = inverse_nz(nx, ny);
    const uint4 w2 = philox(make_uint4(clo, chi, (uint32_t)src, 2u), P.k0, P.k1);
    uint4 w3 = make_uint4(0u, 0u, 0u, 0u);
    if (P.n_coated > 2) w3 = philox(make_uint4(clo, chi, (uint32_t)src, 3u), P.k0, P.k1);
    if (!TESTED && (P.flags & PHOSIM_EARLY_REJECT)) {
        const int si = early_coating_reject(P, lam, w2, w3);
        if (si >= 0) { R.flags = lost(PHOSIM_LOST_COATING, si); return; }
    }
    // pupil point on the annulus, on the nominal first surface, moved back to the top of the atmosphere
    const double r = sqrt64(fma(u64of(w0.x), P.pr_dr2, P.pr_in2));
    double sp, cp;
    sincos_draw64(P.draw_table, w0.y, sp, cp);
    double x = r * cp, y = r * sp;
    double z = P.pupil_z + sag(P.pupil_surf, fma(x, x, y * y));
    {
        const double l = (P.h_top - z) * rinv;
        x = fma(-nx, l, x);
        y = fma(-ny, l, y);
        z = P.h_top;
    }
    uint4 w4 = make_uint4(0u, 0u, 0u, 0u);
    if (P.hf_K > 0 || (P.flags & PHOSIM_BACK_REFLECT)) w4 = philox(make_uint4(clo, chi, (uint32_t)src, 4u), P.k0, P.k1);
    // frozen-flow layers top to bottom: propagate, refractive kick from the screen gradient (Sec. 2.3)
    if (P.flags & PHOSIM_ATMOSPHERE) {
        double kick;
        if constexpr (MIXED) {
            kick = (double)((float)P.kick0 * exp2f(-0.2f * log2f(f32_rn_pos(lam * P.inv_lam_ref))));
        } else {
            // (lambda / lambda_ref)^(-1/5): a single-precision seed y and one third-order step, with e = 1 - a y^5:
            // y (1 - e)^(-1/5) = y (1 + e / 5 + 3 e^2 / 25 + ...)
            const double a = lam * P.inv_lam_ref;
            double y5 = f64_exact(powf(f32_trunc(a), -0.2f));
            const double y2 = y5 * y5, e = fma(-(a * y5), y2 * y2, 1.0);
            y5 = fma(y5 * e, fma(0.12, e, 0.2), y5);
            kick = __double2hiint(a) < 0x47f00000 ? P.kick0 * y5 : 0.0;       // none beyond single precision
        }
#pragma unroll 1
        for (int k = 0; k < P.n_layers; ++k) {
            const DLayer& L = P.layer[k];
            const double ll = L.dz * rinv;            // the drop from the plane above
            x = fma(nx, ll, x);
            y = fma(ny, ll, y);
            z = L.z;
            const double sx = fma(-L.vx, t, x), sy = fma(-L.vy, t, y);
            double gx, gy;
            screen_gradient<MIXED, true>(L.s[0], sx, sy, gx, gy);
#pragma unroll 1
            for (int q = 1; q < L.n_scales; ++q) screen_gradient<MIXED, false>(L.s[q], sx, sy, gx, gy);
            nx = fma(kick, gx, nx);
            ny = fma(kick, gy, ny);
            rinv = inverse_nz(nx, ny);
        }
        // second kick (Sec. 2.3.2): a draw from the long-exposure PSF of the screens above kappa_crit,
        // scaled like the refractive kick by (lambda / lambda_ref)^(-1/5)
        if (P.hf_K > 0) {
            const double scale = kick / P.kick0;
            if constexpr (MIXED) {
                const float ang = lerp_table_f(P.hf32, P.hf_K, u32of(w4.x) * (float)P.hf_K - 0.5f) * (float)scale;
                float sp, cp;
                sincospif(2.f * u32of(w4.y), &sp, &cp);
                nx += (double)(ang * cp);
                ny += (double)(ang * sp);
            } else {
                const double ang = lerp_table(P.hf, P.hf_K, u64of(w4.x) * P.hf_K - 0.5) * scale;
                double sp, cp;
                sincos_draw64(P.draw_table, w4.y, sp, cp);
                nx = fma(ang, cp, nx);
                ny = fma(ang, sp, ny);
            }
            rinv = inverse_nz(nx, ny);
        }
    }
    const double nz = -fma(-nx, nx, fma(-ny, ny, 1.0)) * rinv;
    {
        const double l = (z - P.z_ent) * rinv;
        x = fma(nx, l, x);
        y = fma(ny, l, y);
        z = P.z_ent;
    }
    double X[3] = {x, y, z}, D[3] = {nx, ny, nz};
    MemberDraw mb;
    const bool bundled = s.bundle > 1;
    if (bundled) mb = member_draw<MIXED>(P, s.bsig, src, photon);
    optics<MIXED, true, RECORD>(P, X, D, lam, w1, w2, w3, w4, R, fr, bundled ? &mb : nullptr, src, i);
}


// v[k] of every lane to lane k's sum of v[k] over the warp: at each step a lane keeps half of its values and adds
// its partner's copies of them, so that N values cost N - 1 additions a lane (and log2(32 / N) more, below, where N is
// less than 32: lane k holds the sum of v[k % N] over the lanes of its group of N)
template <int N>
__device__ __forceinline__ double transpose_sum(double v[N], int lane) {
#pragma unroll
    for (int s = N / 2; s >= 1; s >>= 1) {
        const bool up = (lane & s) != 0;
#pragma unroll
        for (int k = 0; k < s; ++k) {
            const double keep = up ? v[k + s] : v[k], send = up ? v[k] : v[k + s];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, send, s);
        }
    }
    return v[0];
}

// Which source owns launch tile t: binary search over the per-source tile prefix (lane 0, then broadcast).
__device__ __forceinline__ int tile_source(const TraceParams& P, uint64_t t, int lane) {
    int src = 0;
    if (lane == 0) {
        int lo = 0, hi = P.n_src - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (P.tile_prefix[mid] <= t) lo = mid;
            else hi = mid - 1;
        }
        src = lo;
    }
    return __shfl_sync(0xffffffffu, src, 0);
}

}  // namespace phosim
