// Adjoint raytrace: pathwise gradients of per-source PSF moments with respect to surface misalignments and
// Zernike figure coefficients (the optics of Peterson et al. 2015, Sec. 2.4.1-2.4.2, differentiated).
//
// The forward path is the trace's (same random numbers, same accept decisions), which keeps at each surface the hit
// point, the direction, the distance, the normal and the index ratio in its frame: the forward pass that gives the
// moments does so for the batches of photons that find room on the tape (512 MB), the others are traced again here.  The
// reverse sweep then walks the surfaces backwards and applies the hand-derived
// vector-Jacobian products of: the frame transform, the implicit intersection (dl = -F_theta / F_l at the
// root), the normal from the sag slopes, and reflection or Snell refraction.
//
// What bounds it is the FP64 pipe, so the sweep recomputes nothing that the forward pass had, and the parameter
// sums cost about one FP64 addition a value: all Zernike coefficients of a surface are linear in the sums of the 28
// monomials of its figure, which a photon adds to whatever the number of coefficients, and the lanes' values
// are summed by a transposed butterfly (31 additions for 32 values, the total of value k in lane k) and added to the
// source's sums.  A surface's misalignments take the force and the torque on it, six sums.  A second kernel turns the
// sums into the parameters' gradients.
// Measured (GB300, 64 stars of 3e4 photons, 97 parameters of which 57 Zernike coefficients), a whole call: 11.9 ms
// with every coefficient's polynomial evaluated per photon, per-lane accumulators in local memory and the
// intersections recomputed in the sweep; 5.6 ms without; 3.8 ms with the photons in batches; 3.2 ms with force and
// torque for the nine elements of each matrix's adjoint, and the figure's second derivatives from their own
// coefficients; 2.5 ms with the forward states kept (a photon's 1.1 KB written and read once, against 40 % of the sweep's
// FP64 operations); 2.3 ms with the forward pass as it is now.
#include "phosim_device.cuh"
#include "phosim_scene.hpp"
#include "photon.cuh"
#include "grad.hpp"

namespace phosim {

// Second derivatives of the sag at the surface-frame point (x, y), without the Zernike figure's
__device__ __forceinline__ void sag_hessian(const DSurface& S, double x, double y, double& zxx, double& zxy, double& zyy) {
    const double r2 = fma(x, x, y * y);
    double g = 0.0, G2 = 0.0;          // (1/r) dz/dr and (1/r) dg/dr
    if (S.flags & SF_CONIC) {
        const double rs = rsqrt64(fma(-S.k1c2, r2, 1.0));
        g = S.c * rs;
        G2 = S.k1c2 * g * (rs * rs);
    }
    if (S.flags & SF_EVEN) {
        int k = S.ne - 1;
        double pd = S.aed[k], p2 = (2 * k + 2) * S.aed[k];
#pragma unroll 1
        while (--k >= 0) {
            pd = fma(r2, pd, S.aed[k]);
            p2 = fma(r2, p2, (2 * k + 2) * S.aed[k]);
        }
        g = fma(r2, pd, g);
        G2 += p2;
    }
    if (S.flags & SF_ODD) {
        const double r = sqrt64(r2);
        int k = S.no - 1;
        double pd = S.aod[k], p2 = (2 * k + 1) * S.aod[k];
#pragma unroll 1
        while (--k >= 0) {
            pd = fma(r2, pd, S.aod[k]);
            p2 = fma(r2, p2, (2 * k + 1) * S.aod[k]);
        }
        g = fma(r, pd, g);
        if (r > 0.0) G2 = fma(p2, rcp64(r), G2);
    }
    zxx = fma(x * x, G2, g);
    zxy = x * y * G2;
    zyy = fma(y * y, G2, g);
}

// Snell refraction's adjoint, with the forward direction d, normal Nin, dn = d . Nin and index ratio mu: given
// ob = d(L)/d(out), db = d(L)/d(d) and Nb = d(L)/d(Nin).
__device__ __forceinline__ void refract_adjoint(const double d[3], const double Nin[3], double dn, double mu,
                                                const double ob[3], double db[3], double Nb[3]) {
    const bool turn = !negative64(dn);        // the normal on the side the ray comes from is s N, s = +-1
    const double s = turn ? -1.0 : 1.0, cosi = turn ? dn : -dn;
    const double k = fma(-(mu * mu), fma(-cosi, cosi, 1.0), 1.0);
    const double ik = rsqrt64(k), sk = k * ik;
    const double a = fma(mu, cosi, -sk);
    // out = mu d + a s N with a = mu cosi - sqrt(k)
    const double ab = s * fma(Nin[0], ob[0], fma(Nin[1], ob[1], Nin[2] * ob[2]));
    const double cb = ab * fma(-(mu * mu) * cosi, ik, mu), scb = s * cb, sa = s * a;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        db[i] = fma(mu, ob[i], -scb * Nin[i]);            // cosi = -s d . N
        Nb[i] = fma(sa, ob[i], -scb * d[i]);
    }
}

// Adjoint of one surface for a warp of photons (on: this lane's photon takes part).  For the detector, fb is the
// adjoint of the final (x, y) in its frame and L the conversion length (the diffusion offset does not depend on the
// optics); otherwise Xb / Db carry the adjoint of the telescope-frame state leaving the surface in and of the state
// entering it out.  sums: the source's sums of this surface, kGradWords.
__device__ __forceinline__ void surface_adjoint(const TraceParams& P, const GradParams& G, int si, const double* q,
                                                bool on, bool detector, const double fb[2], double L, double Xb[3],
                                                double Db[3], double* sums, int lane) {
    const DSurface& S = P.surf[si];
    const bool rotated = (S.flags & SF_ROTATED) != 0;
    double h[3], d[3], N[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        h[k] = on ? q[32 * (kTapeH + k)] : 0.0;
        d[k] = on ? q[32 * (kTapeD + k)] : 0.0;
        N[k] = on ? q[32 * (kTapeN + k)] : 0.0;
    }
    const double q_l = on ? q[32 * kTapeL] : 0.0, mu = on && S.kind != PHOSIM_MIRROR ? q[32 * kTapeMu] : 0.0;
    const double dn = fma(d[0], N[0], fma(d[1], N[1], d[2] * N[2]));
    double hb[3] = {0.0, 0.0, 0.0}, c[3] = {0.0, 0.0, 0.0}, ob[3] = {0.0, 0.0, 0.0}, db[3] = {0.0, 0.0, 0.0}, Nb[3] = {0.0, 0.0, 0.0};
    if (detector) {
        hb[0] = fb[0];
        hb[1] = fb[1];
        if (P.flags & PHOSIM_SENSOR) {
            ob[0] = L * fb[0];
            ob[1] = L * fb[1];
            refract_adjoint(d, N, dn, mu, ob, db, Nb);
        }
    } else {
        // X' = M^T h + o, D' = M^T out: adjoints into h and out
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            hb[i] = rotated ? fma(S.M[3 * i], Xb[0], fma(S.M[3 * i + 1], Xb[1], S.M[3 * i + 2] * Xb[2])) : Xb[i];
            ob[i] = rotated ? fma(S.M[3 * i], Db[0], fma(S.M[3 * i + 1], Db[1], S.M[3 * i + 2] * Db[2])) : Db[i];
        }
        if (S.kind == PHOSIM_MIRROR) {
            const double n2 = -2.0 * fma(N[0], ob[0], fma(N[1], ob[1], N[2] * ob[2])), d2 = -2.0 * dn;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                db[i] = fma(n2, N[i], ob[i]);
                Nb[i] = fma(d2, ob[i], n2 * d[i]);
            }
        } else {
            refract_adjoint(d, N, dn, mu, ob, db, Nb);
        }
    }
    // normal N = (-S_x, -S_y, 1) / |.|: adjoint into the slopes; slopes at the hit: into h by the second derivatives
    const bool curved = !(S.flags & SF_FLAT_ONLY), figure = G.figure[si] != 0, zernike = (S.flags & SF_ZERN) != 0;
    double zxb = 0.0, zyb = 0.0, m[kZPoly];              // m: the monomials u^a v^b, row by row in b
    if (curved || figure) {
        const double t = fma(Nb[0], N[0], fma(Nb[1], N[1], Nb[2] * N[2]));
        zxb = N[2] * fma(t, N[0], -Nb[0]);
        zyb = N[2] * fma(t, N[1], -Nb[1]);
    }
    if (figure || zernike) {
        const double u = h[0] * S.zinv, v = h[1] * S.zinv;
        m[0] = 1.0;
        int off = 0;
#pragma unroll
        for (int b = 0; b <= 6; ++b) {
            if (b > 0) {
                m[off + 7 - (b - 1)] = m[off] * v;       // the row's first: v^b
                off += 7 - (b - 1);
            }
#pragma unroll
            for (int a = 1; a + b <= 6; ++a) m[off + a] = m[off + a - 1] * u;
        }
    }
    if (curved) {
        double sxx, sxy, syy;
        sag_hessian(S, h[0], h[1], sxx, sxy, syy);
        if (zernike) {
            const ZernikeHessian& Z = G.hessian[si];
            int off = 0, k = 0;
#pragma unroll
            for (int b = 0; b <= 4; ++b) {
#pragma unroll
                for (int a = 0; a + b <= 4; ++a, ++k) {
                    sxx = fma(Z.xx[k], m[off + a], sxx);
                    sxy = fma(Z.xy[k], m[off + a], sxy);
                    syy = fma(Z.yy[k], m[off + a], syy);
                }
                off += 7 - b;
            }
        }
        c[0] = fma(sxx, zxb, sxy * zyb);
        c[1] = fma(sxy, zxb, syy * zyb);
        hb[0] += c[0];
        hb[1] += c[1];
    }
    // h = p + l d with the implicit intersection F(l; p, d, c) = p_z + l d_z - S(p_xy + l d_xy; c) = 0:
    // F_l = d . N / N_z, so l's adjoint enters p along the normal with weight W
    const double lb = fma(hb[0], d[0], fma(hb[1], d[1], hb[2] * d[2]));
    const double W = -lb * rcp64(dn);
    double pb[3], Xn[3], Dn[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) pb[i] = fma(W, N[i], hb[i]);
    if (figure) {
        // Zernike coefficients: dF/dc_j = -Z_j(h), d(slopes)/dc_j = grad Z_j(h); here for the monomials of Z
        double g[32];
        const double w = on ? -W * N[2] : 0.0, gu = on ? zxb * S.zinv : 0.0, gv = on ? zyb * S.zinv : 0.0;
        int off = 0, down = 0;
#pragma unroll
        for (int b = 0; b <= 6; ++b) {
#pragma unroll
            for (int a = 0; a + b <= 6; ++a) {
                double s = w * m[off + a];
                if (a >= 1) s = fma(a * gu, m[off + a - 1], s);
                if (b >= 1) s = fma(b * gv, m[down + a], s);
                g[off + a] = on ? s : 0.0;
            }
            down = off; off += 7 - b;
        }
#pragma unroll
        for (int k = kZPoly; k < 32; ++k) g[k] = 0.0;
        const double sum = transpose_sum<32>(g, lane);
        if (lane < kZPoly) atomicAdd(sums + lane, sum);
    }
    const bool shift = G.shift[si] != 0, tilt = G.tilt[si] != 0;
    // p = M (X - o), d = M D
    double dt[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) dt[i] = fma(q_l, pb[i], db[i]);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        Xn[k] = rotated ? fma(S.M[k], pb[0], fma(S.M[3 + k], pb[1], S.M[6 + k] * pb[2])) : pb[k];
        Dn[k] = rotated ? fma(S.M[k], dt[0], fma(S.M[3 + k], dt[1], S.M[6 + k] * dt[2])) : dt[k];
    }
    if (shift || tilt) {
        // The surface as a rigid body, in its frame: the force F on its vertex and the torque T on its axes, from which
        // grad_finish_kernel takes the parameters' gradients.  M enters p + l d = M (X + l D - o), d = M D and past the
        // surface X' = M^T h + o, D' = M^T out; with dM = [w] M its terms are w . (h x (pb - hb0) + d x db - out x ob),
        // where pb - hb0 is c, the part of the hit's adjoint that the surface put in, and d x db - out x ob is Nb x N for
        // a reflection as for a refraction (both commute with a rotation of d, N and out together).
        double g[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) g[k] = 0.0;
#pragma unroll
        for (int i = 0; i < 3; ++i) c[i] = detector ? pb[i] : fma(W, N[i], c[i]);
        if (shift) {
#pragma unroll
            for (int k = 0; k < 3; ++k) g[k] = -c[k];
        }
        if (tilt) {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int i = (k + 1) % 3, j = (k + 2) % 3;
                const double hc = fma(h[i], c[j], -(h[j] * c[i]));
                g[3 + k] = detector ? fma(d[i], db[j], fma(-d[j], db[i], hc)) : fma(Nb[i], N[j], fma(-Nb[j], N[i], hc));
            }
        }
#pragma unroll
        for (int k = 0; k < 6; ++k) g[k] = on ? g[k] : 0.0;
        const double sum = transpose_sum<8>(g, lane);
        if ((lane & 7) < 6) atomicAdd(sums + 32 + lane, sum);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) { Xb[k] = Xn[k]; Db[k] = Dn[k]; }
}

__global__ void __launch_bounds__(32, 12) grad_kernel(const __grid_constant__ TraceParams P,
                                                      const __grid_constant__ GradParams G,
                                                      const __grid_constant__ BatchList L) {
    // a warp a batch of photons of one source that go on past the dynamic transmission test, as in the trace
    const int lane = threadIdx.x;
    const unsigned long long n = *L.n;
    for (;;) {
        unsigned long long b = 0;
        if (lane == 0) b = atomicAdd(L.next, 1ull);
        b = __shfl_sync(0xffffffffu, b, 0);
        if (b >= n) break;
        const PhotonBatch& B = L.batch[b];
        const int src = B.src;
        const bool v = lane < (int)B.n;
        const DSource& s = P.sources[src];
        const double* sd = G.seeds + (size_t)src * 8;
        // what the trace kept, or the photons once more
        const bool taped = b < L.tape_batches;
        ForwardRecord fr = forward_record(P, L, taped ? b : L.tape_batches + blockIdx.x, lane);
        const double* end = fr.end();
        bool on = false;
        if (taped) {
            on = v && end[32 * kTapeOn] != 0.0;
        } else if (v) {
            PhotonOut R;
            R.flags = 0;
            trace_photon<false, true, true>(P, s, src, B.first + B.k[lane], R, &fr);
            on = (R.flags & PHOSIM_F_DETECTED) != 0;
            double* q = fr.end();
            q[32 * kTapeX] = R.x;
            q[32 * kTapeY] = R.y;
        }
        // the whole warp sweeps (the sums need every lane); the other lanes' values are dropped
        if (!__any_sync(0xffffffffu, on)) continue;
        const double dx = on ? end[32 * kTapeX] - sd[5] : 0.0, dy = on ? end[32 * kTapeY] - sd[6] : 0.0;
        const double depth = on && (P.flags & PHOSIM_SENSOR) ? end[32 * kTapeDepth] : 0.0;
        const double fb[2] = {fma(sd[2], dx, fma(sd[3], dy, sd[0])), fma(sd[4], dy, fma(sd[3], dx, sd[1]))};
        double Xb[3] = {0.0, 0.0, 0.0}, Db[3] = {0.0, 0.0, 0.0};
        double* out = G.sums + (size_t)src * P.n_surf * kGradWords;
#pragma unroll 1
        for (int si = P.n_surf - 1; si >= G.first_surface; --si)
            surface_adjoint(P, G, si, fr.surface(si), on, si == P.n_surf - 1, fb, depth, Xb, Db, out + si * kGradWords, lane);
    }
}

// The parameters' gradients from the sums, one thread a source and parameter
__global__ void grad_finish_kernel(const __grid_constant__ GradParams G, int n_src, int n_surf) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (size_t)n_src * G.n_params) return;
    const int p = (int)(i % G.n_params), f = G.param_field[p];
    const double* a = G.sums + ((i / G.n_params) * n_surf + G.param_surface[p]) * kGradWords;
    double s = 0.0;
    if (f >= 100) {
        const double* z = G.zmono + (size_t)(f - 100) * kZPoly;
#pragma unroll
        for (int k = 0; k < kZPoly; ++k) s = fma(z[k], a[k], s);
    } else {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            double sum = 0.0;                            // of the force (f < 3) or the torque
#pragma unroll
            for (int g = 0; g < 4; ++g) sum += a[32 + (f < 3 ? 0 : 3) + i + 8 * g];
            s = fma(G.axis[G.param_surface[p]][f][i], sum, s);
        }
    }
    G.grad[i] = s;
}

cudaError_t launch_grad(const TraceParams& P, const GradParams& G, const BatchList& L, int blocks, cudaStream_t st) {
    grad_kernel<<<blocks, 32, 0, st>>>(P, G, L);
    return cudaGetLastError();
}

cudaError_t launch_grad_finish(const TraceParams& P, const GradParams& G, cudaStream_t st) {
    const size_t n = (size_t)P.n_src * G.n_params;
    grad_finish_kernel<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(G, P.n_src, P.n_surf);
    return cudaGetLastError();
}

cudaError_t grad_occupancy(int* blocks_per_sm) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, grad_kernel, 32, 0);
}

}  // namespace phosim
