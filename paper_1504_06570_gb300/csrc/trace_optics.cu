// The optics and bundle stages of the two-kernel double-single path (Peterson et al. 2015, Sec. 2.4-2.5): the
// surfaces, the sensor, the pixel counts and the per-source moment sums of the states the entry stage
// (trace.cu) leaves on the telescope's entrance plane.  This translation unit compiles the double-single
// quotient, square root and reciprocal root inline: with them inline the optics stage (80 registers) measured
// 3 % faster, and the entry stage, which keeps them out of line, 15 % slower.  The generator is inline here
// too (1 % faster; the entry stage keeps its call).
#ifndef PHOSIM_DS_HEAVY_OPTICS
#define PHOSIM_DS_HEAVY_OPTICS __forceinline__
#endif
#define PHOSIM_DS_HEAVY PHOSIM_DS_HEAVY_OPTICS
#ifndef PHOSIM_DS_PHILOX_OPTICS
#define PHOSIM_DS_PHILOX_OPTICS __forceinline__
#endif
#define PHOSIM_DS_PHILOX PHOSIM_DS_PHILOX_OPTICS

#include "phosim_device.cuh"
#include "phosim_scene.hpp"
#include "photon.cuh"
#include "photon_ds.cuh"

namespace phosim {

// blocks per SM the optics stage is compiled for: 3 of 80 registers (the ghost walks: 3.56 ms for 4e6 photons, 3.70 with 4
// of 64, 3.91 with 2 of 128); for simple surfaces 4 of 64, which hold that walk with few spills (the 1000-star field of
// 1e8 photons: 4.62 ms, 4.92 with 3 and 4.99 with 5)
#ifndef PHOSIM_DS_OPTICS_MIN_BLOCKS
#define PHOSIM_DS_OPTICS_MIN_BLOCKS 3
#endif
#ifndef PHOSIM_DS_SIMPLE_MIN_BLOCKS
#define PHOSIM_DS_SIMPLE_MIN_BLOCKS 4
#endif
// threads per block of the optics stage (0: the schedule's block size).  Fixed at 256: the lockstep wants
// blocks of 8 warps (128- and 64-thread blocks measured 17 % and 28 % slower), whatever the schedule chosen
// for the entry stage.
#ifndef PHOSIM_DS_OPTICS_THREADS
#define PHOSIM_DS_OPTICS_THREADS 256
#endif
constexpr int kOpticsMaxThreads = PHOSIM_DS_OPTICS_THREADS ? PHOSIM_DS_OPTICS_THREADS : 256;

#ifndef PHOSIM_DS_MEMBERS_MIN_BLOCKS
#define PHOSIM_DS_MEMBERS_MIN_BLOCKS 4
#endif

// The sums over the warp of five values a lane: v0 in lanes 0-3, v1 in 4-7, v2 in 8-11, v3 in 16-19 and v4 in 20-23
// (zeros in the others).  At each of the first three steps a lane keeps part of its values and adds its partner's copies
// of them, so that the five sums cost 3 + 2 + 1 + 1 + 1 additions a lane.
__device__ __forceinline__ ds pick_ds(bool p, ds a, ds b) { return {p ? a.hi : b.hi, p ? a.lo : b.lo}; }
__device__ __forceinline__ ds from_lane_ds(ds v, int d) {
    return {__shfl_xor_sync(0xffffffffu, v.hi, d), __shfl_xor_sync(0xffffffffu, v.lo, d)};
}
__device__ __forceinline__ ds transpose_sum_ds(ds v0, ds v1, ds v2, ds v3, ds v4, int lane) {
    const ds zero = ds_f(0.f);
    bool up = (lane & 16) != 0;
    const ds2 a = add2(ds2_of(pick_ds(up, v3, v0), pick_ds(up, v4, v1)),
                       ds2_of(from_lane_ds(pick_ds(up, v0, v3), 16), from_lane_ds(pick_ds(up, v1, v4), 16)));
    const ds a2 = pick_ds(up, zero, v2) + from_lane_ds(pick_ds(up, v2, zero), 16);
    up = (lane & 8) != 0;
    const ds2 b = add2(ds2_of(pick_ds(up, a2, ds2_x(a)), pick_ds(up, zero, ds2_y(a))),
                       ds2_of(from_lane_ds(pick_ds(up, ds2_x(a), a2), 8), from_lane_ds(pick_ds(up, ds2_y(a), zero), 8)));
    up = (lane & 4) != 0;
    ds c = pick_ds(up, ds2_y(b), ds2_x(b)) + from_lane_ds(pick_ds(up, ds2_x(b), ds2_y(b)), 4);
    c = c + from_lane_ds(c, 2);
    return c + from_lane_ds(c, 1);
}

// runs of one source in a warp up to which each is summed before its atomics
constexpr int kMaxWarpSources = 8;

// Account for one photon per lane of the optics or bundle stage: record, image, counters (cnt: the warp's
// counters in shared memory, lane 0) and the moment sums about the source's chief-ray position.  Every lane of the warp calls it.
__device__ __forceinline__ void account_ds(const TraceParams& P, const PhotonOutS& R, bool v, int src, uint64_t i,
                                           int lane, unsigned long long* cnt) {
    const DSource& s = P.sources[src];
    if (v && P.records) {
        phosim_photon_record rec;
        rec.x = ds_value(R.x); rec.y = ds_value(R.y); rec.xc = ds_value(R.xc); rec.yc = ds_value(R.yc);
        rec.lambda = (double)R.lam;
        rec.flags = R.flags; rec.pix = R.pix;
        P.records[s.rec_off + (i - s.first)] = rec;
    }
    const bool det = v && (R.flags & PHOSIM_F_DETECTED);
    const unsigned dmask = __ballot_sync(0xffffffffu, det);
    // a lane's count each: adding the lanes of one pixel up first (a match and a popcount) costs more than it saves, also
    // where a tenth of all photons hit one pixel (1.206 ms with it, 1.201 without; the 1000-star field 5.56 and 5.48)
    if (det) atomicAdd(P.image + R.pix, 1u);
    if (lane == 0) cnt[1] += __popc(dmask);
    const uint32_t reason = v ? ((R.flags >> 8) & 0xffu) : 0u;
#pragma unroll
    for (int q = 1; q <= 8; ++q) {
        const unsigned bq = __ballot_sync(0xffffffffu, reason == (uint32_t)q);
        if (lane == 0) cnt[1 + q] += __popc(bq);
    }
    if (P.moments && dmask) {
        // Per-source partial sums of the warp in double-single (exact products of the single-precision offsets from
        // the chief ray, sums to ~2^-47), added to the source's double-precision moments: one set of atomics per source,
        // not per photon, and the FP64 pipe (a sixty-fourth of the FP32 rate on this GPU) converts one sum a lane.  The
        // states arrive in runs of one source (a warp of the entry stage appends its survivors together), so a warp
        // mostly holds one to three sources, each summed in its turn (8 additions against the 25 of a segmented scan of
        // the five sums: optics of the 1000-star field 5.28 ms, not 5.36).  Where a warp holds more (sources of a few
        // photons), that would cost more than the atomics it saves, and every lane adds its own terms.
        const float fx = (R.x - ds{s.ref_s[0], s.ref_s[1]}).hi, fy = (R.y - ds{s.ref_s[2], s.ref_s[3]}).hi;
        double* const sums = P.mom_stripes ? P.mom_stripes + (size_t)(blockIdx.x % kMomStripes) * P.mom_stripe_stride : P.moments;
        const int prev = __shfl_up_sync(0xffffffffu, src, 1);
        const unsigned heads = __ballot_sync(0xffffffffu, lane == 0 || prev != src);
        if (__popc(heads) > kMaxWarpSources) {
            if (det) {
                double* const M = sums + (size_t)src * PHOSIM_MOMENT_WORDS;
                const double x = (double)fx, y = (double)fy;
                atomicAdd(M, 1.0);
                atomicAdd(M + 1, x);
                atomicAdd(M + 2, y);
                atomicAdd(M + 3, x * x);
                atomicAdd(M + 4, x * y);
                atomicAdd(M + 5, y * y);
            }
            return;
        }
        for (unsigned todo = dmask; todo;) {
            const int of = __shfl_sync(0xffffffffu, src, __ffs(todo) - 1);
            const bool in = det && src == of;
            const unsigned mask = __ballot_sync(0xffffffffu, in);
            todo &= ~mask;
            const float x = in ? fx : 0.f, y = in ? fy : 0.f;
            const ds sum = transpose_sum_ds(ds_f(x), ds_f(y), two_prod(x, x), two_prod(x, y), two_prod(y, y), lane);
            double* const M = sums + (size_t)of * PHOSIM_MOMENT_WORDS;
            if (lane == 31) atomicAdd(M, (double)__popc(mask));
            // lanes 0, 4, 8, 16 and 20 hold the sums of x, y, xx, xy and yy
            if ((0x110111u >> lane) & 1u) atomicAdd(M + 1 + (lane < 16 ? lane >> 2 : (lane >> 2) - 1), ds_value(sum));
        }
    }
}

// Rays that a coating has just turned round (parked) go to the round of their number of reflections.  Every lane
// of the warp calls it.
__device__ __forceinline__ void park_ghosts(const DSStage& S, bool parked, const OpticsWalk& W, ds lam, int src, uint64_t ray,
                                            int bin, int lane) {
    const unsigned mask = __ballot_sync(0xffffffffu, parked);
    if (!parked) return;
    GhostRound& round = S.rounds[W.bounces - 1];
    const unsigned below = (1u << lane) - 1u;
    unsigned long long slot = 0;
    if (lane == __ffs(mask) - 1) slot = atomicAdd(&round.n, (unsigned long long)__popc(mask));
    slot = __shfl_sync(mask, slot, __ffs(mask) - 1) + __popc(mask & below);
    const unsigned same = __match_any_sync(mask, bin);
    if (lane == __ffs(same) - 1) atomicAdd(&round.bins[bin], (unsigned)__popc(same));
    DSGhost g;
#pragma unroll
    for (int k = 0; k < 3; ++k) { g.X[k] = W.X[k]; g.D[k] = W.D[k]; }
    g.n_cur = W.media[kHere];
    g.lam = lam.hi; g.lam_lo = lam.lo;
    g.idx = ray; g.src = src; g.n_ghost = W.n_ghost;
    g.si = (short)W.si; g.dir = (short)W.dir; g.bounces = (short)W.bounces; g.pad = 0;
    S.ghost[(W.bounces - 1) & 1][slot] = g;
    S.ghost_bin[slot] = (uint8_t)bin;
}

// The optics stage.  KIND: the scene has no reflecting coating (kWalkPlain; kWalkSimple where its surfaces are simple too),
// the states of the entry stage with rays that a coating may turn round (kWalkForward), or a round of such rays
// (kWalkGhosts, S.round).
//
// Bound by instruction issue (7 of 10 cycles issue): what its registers hold decides how many warps fill the others.
// So they hold the ray and little else: wavelength, source and index are read again from the entry stage's state where a
// surface or the accounting asks for them, the media's indices wait in shared memory, the double-single root of the rays
// that the single-precision one does not serve is out of line, and a scene of simple surfaces has a kernel without the
// code of the others (together 5.27 -> 4.62 ms for the 1000-star field, and 3.81 -> 3.56 with ghosts).
//
// Without ghosts every ray of a block is at the same surface, so the surface's constants are read at a uniform
// index, and nothing of the ghosts is in the code.  (One kernel for all scenes, its surface index a ray's own,
// took 10.2 ms for the 1000-star field of 1e8 photons and 223 ms for a quarter of the batched workload; 9.9 and
// 217 ms in this form.)  With them, a ray that a coating turns round leaves its
// block: in place it would hold the block's other rays at surfaces that only it meets, while the rays on their
// way back and forth diverge.  The rays of one number of reflections are walked together later, ordered by the
// surface that turned them, so that again a block's rays are at one surface.  After kGhostRounds reflections a ray
// goes on in place (few are left).  (Every ray in place: 16 of 32 lanes active and 9.05 ms for 4e6 photons of which
// three in four are turned by a filter that reflects what it does not pass; 3.8 ms in rounds.)
template <WalkKind KIND>
__global__ void __launch_bounds__(kOpticsMaxThreads, KIND == kWalkSimple ? PHOSIM_DS_SIMPLE_MIN_BLOCKS : PHOSIM_DS_OPTICS_MIN_BLOCKS)
    ds_optics_kernel(const __grid_constant__ TraceParams P, const __grid_constant__ DSStage S) {
    __shared__ unsigned long long cnt_mem[kOpticsMaxThreads / 32][kNumCounters];
    __shared__ unsigned long long next_batch;
    __shared__ ds media[kOpticsMaxThreads][kMedia];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lanes_below = (1u << lane) - 1u;
    unsigned long long* cnt = cnt_mem[warp];
    if (lane < kNumCounters) cnt[lane] = 0;
    __syncwarp();
    // launched beside the entry stage's end (a short call waits for launches, not for work)
    wait_for_previous();
    const unsigned long long n = KIND == kWalkGhosts ? S.rounds[S.round].n : *S.n_state;
    unsigned long long* const batch = KIND == kWalkGhosts ? &S.rounds[S.round].batch : S.batch;
    // a block's states at a time, all its warps meeting the surfaces together (a barrier after each), so
    // that the SM's warps fetch the same stretch of code rather than as many stretches as warps; the
    // blocks claim batches as they finish (a block is as slow as its slowest ray at every surface)
    // (the first batch is the block's own)
    for (unsigned long long b0 = (unsigned long long)blockIdx.x * blockDim.x; b0 < n;) {
        const unsigned long long e = b0 + threadIdx.x;
        const bool v = e < n;
        PhotonOutS R;
        R.flags = 0; R.pix = -1; R.lam = 0.f;
        R.x = R.y = R.xc = R.yc = ds_f(0.f);
        int src = 0;
        uint64_t u = 0;
        DetectorHit H;
        OpticsWalk W;
        W.media = media[threadIdx.x];
        ds lam = ds_f(0.f);
        bool go = false, bundled = false, parked = false;
        if (v) {
            if constexpr (KIND == kWalkGhosts) {
                const DSGhost& g = S.ghost[S.round & 1][S.ghost_order[e]];
                src = g.src;
                bundled = P.sources[src].bundle > 1;
                u = g.idx;
                lam = ds{g.lam, g.lam_lo};
                walk_start(W, g.X, g.D);
                W.media[kHere] = g.n_cur;
                W.si = g.si; W.dir = g.dir; W.bounces = g.bounces; W.n_ghost = g.n_ghost;
            } else {
                const DSState& st = S.state[e];
                const ds X[3] = {st.x, st.y, P.z_ent_s}, D[3] = {st.nx, st.ny, st.nz};
                walk_start(W, X, D);
                bundled = P.sources[st.src].bundle > 1;
            }
            go = true;
        }
        int bin = 0;
        if constexpr (KIND == kWalkGhosts) {
#pragma unroll 1
            while (__syncthreads_or(go)) {
                if (!go) continue;
                const int si = W.si, before = W.bounces;
                go = surface_step_ds<KIND>(P, W, si, RayHeld{lam, src, u}, R, nullptr, bundled ? &H : nullptr);
                if (go && W.bounces > before && W.bounces <= kGhostRounds) {
                    parked = true;
                    go = false;
                    bin = P.surf[si].coat_slot;
                }
            }
        } else {
            const RayInState ray = {S.state + (v ? e : 0)};
#pragma unroll 1
            for (int si = 0; __syncthreads_or(go); ++si) {
                if (!go) continue;
                go = surface_step_ds<KIND>(P, W, si, ray, R, nullptr, bundled ? &H : nullptr);
                if (KIND == kWalkForward && go && W.bounces > 0) {
                    parked = true;
                    go = false;
                    bin = P.surf[si].coat_slot;
                }
            }
            if (v) {
                src = ray.src();
                u = ray.idx();
                lam = ray.lam();
            }
        }
        if constexpr (KIND == kWalkForward || KIND == kWalkGhosts) park_ghosts(S, parked, W, lam, src, u, bin, lane);
        R.lam = lam.hi;
        // a bundle's ray that reached the detector surface hands its hit over to the bundle stage
        const bool handed = v && R.flags == kHandedOff;
        const unsigned hmask = __ballot_sync(0xffffffffu, handed);
        if (hmask) {
            unsigned long long slot = 0;
            if (lane == 0) slot = atomicAdd(S.n_hits, (unsigned long long)__popc(hmask));
            slot = __shfl_sync(0xffffffffu, slot, 0) + __popc(hmask & lanes_below);
            if (handed) {
                DSHit h;
                h.H = H;
                h.lam = lam.hi;
                h.lam_lo = lam.lo;
                h.src = src;
                h.ray = u;
                S.hits[slot] = h;
            }
        }
        // every other unit is one photon, or a bundle's ray lost before the detector (all its photons)
        const uint32_t nb = v ? P.sources[src].bundle : 1u;
        uint64_t lo = u;
        uint32_t nm = 1;
        if (nb > 1) unit_members(P.sources[src], nb, u, lo, nm);
        const bool ended = v && !handed && !parked;
        const uint32_t n_loop = __reduce_max_sync(0xffffffffu, ended ? nm : 0u);
        for (uint32_t m = 0; m < n_loop; ++m) account_ds(P, R, ended && m < nm, src, lo + m, lane, cnt);
        if ((unsigned long long)gridDim.x * blockDim.x >= n) break;
        if (threadIdx.x == 0) next_batch = (gridDim.x + atomicAdd(batch, 1ull)) * blockDim.x;
        __syncthreads();
        b0 = next_batch;
    }
    __syncwarp();
    if (lane < kNumCounters && cnt[lane]) atomicAdd(P.counters + lane, cnt[lane]);
}

// The order of a round's rays: those that the same coated surface turned round next to each other.  A block places 2048
// rays at a time: their places among the block's rays of their surface by shared-memory atomics, then one global atomic a
// surface and block, on which all blocks meet (one a surface and warp: 26 us for the first round of 1e6 photons, 5 us so;
// 4e6 photons 4.11 and 4.03 ms).
constexpr int kOrderThreads = 256, kOrderRays = 8;
__global__ void __launch_bounds__(kOrderThreads) ghost_order_kernel(const __grid_constant__ DSStage S) {
    __shared__ unsigned count[8], base[8];
    GhostRound& round = S.rounds[S.round];
    const unsigned n = (unsigned)round.n, lane = threadIdx.x & 31;
    for (unsigned b = blockIdx.x * (kOrderThreads * kOrderRays); b < n; b += gridDim.x * (kOrderThreads * kOrderRays)) {
        if (threadIdx.x < 8) count[threadIdx.x] = 0;
        __syncthreads();
        int bin[kOrderRays];
        unsigned place[kOrderRays];
#pragma unroll
        for (int k = 0; k < kOrderRays; ++k) {
            const unsigned e = b + k * kOrderThreads + threadIdx.x;
            bin[k] = e < n ? S.ghost_bin[e] : 8;
        }
#pragma unroll
        for (int k = 0; k < kOrderRays; ++k) {
            const unsigned same = __match_any_sync(0xffffffffu, bin[k]);
            const int first = __ffs(same) - 1;
            unsigned at = 0;
            if ((int)lane == first && bin[k] < 8) at = atomicAdd(&count[bin[k]], (unsigned)__popc(same));
            place[k] = __shfl_sync(0xffffffffu, at, first) + __popc(same & ((1u << lane) - 1u));
        }
        __syncthreads();
        if (threadIdx.x < 8) {
            unsigned at = count[threadIdx.x] ? atomicAdd(&round.placed[threadIdx.x], count[threadIdx.x]) : 0u;
            for (int k = 0; k < (int)threadIdx.x; ++k) at += round.bins[k];
            base[threadIdx.x] = at;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kOrderRays; ++k)
            if (bin[k] < 8) S.ghost_order[base[bin[k]] + place[k]] = b + k * kOrderThreads + threadIdx.x;
        __syncthreads();
    }
}

// The photons of the bundles whose ray reached the detector surface: each its own Gaussian offset and its
// own sensor draws from the shared hit (Sec. 3.2), one hit per thread.
__global__ void __launch_bounds__(256, PHOSIM_DS_MEMBERS_MIN_BLOCKS) ds_members_kernel(const __grid_constant__ TraceParams P,
                                                                                       const DSStage S) {
    __shared__ unsigned long long cnt_mem[kWarpsPerBlock][kNumCounters];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long* cnt = cnt_mem[warp];
    if (lane < kNumCounters) cnt[lane] = 0;
    __syncwarp();
    const unsigned long long n = *S.n_hits;
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long b = (unsigned long long)blockIdx.x * blockDim.x + (unsigned long long)warp * 32ull; b < n;
         b += stride) {
        const unsigned long long e = b + lane;
        const bool v = e < n;
        DSHit h;
        h.src = 0; h.ray = 0; h.lam = 0.f; h.lam_lo = 0.f;
        if (v) h = S.hits[e];
        const DSource& s = P.sources[h.src];
        const uint32_t nb = v ? s.bundle : 0u;
        uint64_t lo = 0;
        uint32_t nm = 0;
        if (v) unit_members(s, nb, h.ray, lo, nm);
        const uint32_t n_loop = __reduce_max_sync(0xffffffffu, nm);
        for (uint32_t m = 0; m < n_loop; ++m) {
            const bool vm = m < nm;
            PhotonOutS R;
            R.flags = 0; R.pix = -1; R.lam = h.lam;
            R.x = R.y = R.xc = R.yc = ds_f(0.f);
            if (vm) {
                const MemberDrawS mb = member_draw_s(P, (float)s.bsig, h.src, lo + m);
                detect_ds(P, h.H, ds{h.lam, h.lam_lo}, h.src, h.ray, R, &mb);
            }
            account_ds(P, R, vm, h.src, lo + m, lane, cnt);
        }
    }
    __syncwarp();
    if (lane < kNumCounters && cnt[lane]) atomicAdd(P.counters + lane, cnt[lane]);
}

// The striped moment accumulators of the two-kernel path added into the caller's moment sums (one thread a
// source and word)
__global__ void moment_stripes_kernel(const __grid_constant__ TraceParams P) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.n_src * 6) return;
    const size_t w = (size_t)(i / 6) * PHOSIM_MOMENT_WORDS + (size_t)(i % 6);
    double sum = 0.0;
#pragma unroll
    for (int k = 0; k < kMomStripes; ++k) sum += P.mom_stripes[(size_t)k * P.mom_stripe_stride + w];
    P.moments[w] += sum;
}

const void* ds_optics_kernel_ptr(int kind) {
    return kind == kWalkGhosts ? (const void*)ds_optics_kernel<kWalkGhosts>
                               : kind == kWalkForward ? (const void*)ds_optics_kernel<kWalkForward>
                               : kind == kWalkSimple  ? (const void*)ds_optics_kernel<kWalkSimple>
                                                      : (const void*)ds_optics_kernel<kWalkPlain>;
}
const void* ghost_order_kernel_ptr() { return (const void*)ghost_order_kernel; }

const void* moment_stripes_kernel_ptr() { return (const void*)moment_stripes_kernel; }

cudaError_t launch_moment_stripes(const TraceParams& P, cudaStream_t st) {
    if (P.n_src <= 0 || !P.moments || !P.mom_stripes) return cudaSuccess;
    moment_stripes_kernel<<<(P.n_src * 6 + 255) / 256, 256, 0, st>>>(P);
    return cudaGetLastError();
}

int ds_optics_threads(int threads) { return PHOSIM_DS_OPTICS_THREADS ? PHOSIM_DS_OPTICS_THREADS : threads; }

cudaError_t launch_ds_optics(const TraceParams& P, const DSStage& S, int kind, int blocks, int threads, cudaStream_t st, bool beside) {
    const int block = ds_optics_threads(threads);
    if (beside && kind == kWalkSimple) return launch_beside(ds_optics_kernel<kWalkSimple>, blocks, block, st, P, S);
    if (beside && kind == kWalkPlain) return launch_beside(ds_optics_kernel<kWalkPlain>, blocks, block, st, P, S);
    if (beside && kind == kWalkForward) return launch_beside(ds_optics_kernel<kWalkForward>, blocks, block, st, P, S);
    if (kind == kWalkGhosts) ds_optics_kernel<kWalkGhosts><<<blocks, block, 0, st>>>(P, S);
    else if (kind == kWalkForward) ds_optics_kernel<kWalkForward><<<blocks, block, 0, st>>>(P, S);
    else if (kind == kWalkSimple) ds_optics_kernel<kWalkSimple><<<blocks, block, 0, st>>>(P, S);
    else ds_optics_kernel<kWalkPlain><<<blocks, block, 0, st>>>(P, S);
    return cudaGetLastError();
}

cudaError_t launch_ghost_order(const DSStage& S, int blocks, cudaStream_t st) {
    ghost_order_kernel<<<blocks, kOrderThreads, 0, st>>>(S);
    return cudaGetLastError();
}

cudaError_t launch_ds_members(const TraceParams& P, const DSStage& S, int blocks, int threads, cudaStream_t st) {
    ds_members_kernel<<<blocks, threads, 0, st>>>(P, S);
    return cudaGetLastError();
}

const void* ds_members_kernel_ptr() { return (const void*)ds_members_kernel; }

cudaError_t ds_stage_occupancy(int kind, int threads, int* entry_per_sm, int* optics_per_sm, int* members_per_sm) {
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(entry_per_sm, ds_entry_kernel_ptr(), threads, 0);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(optics_per_sm, ds_optics_kernel_ptr(kind),
                                                          ds_optics_threads(threads), 0);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(members_per_sm, ds_members_kernel, threads, 0);
}

}  // namespace phosim
