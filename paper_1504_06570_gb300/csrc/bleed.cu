// Saturation and bleeding of a finished image (Peterson et al. 2015, Sec. 2.5): charge above the full well
// moves along the row to the closest pixels with room, never across the centre implant, and is lost once
// the half-row is full.  The electron-by-electron alternation (left, right, left, ...) at each distance is
// applied in closed form.
#include <algorithm>
#include <cstdint>

#include <cuda_runtime.h>

#include "phosim.h"

namespace {

constexpr unsigned kAll = 0xffffffffu;

__device__ __forceinline__ uint32_t warp_total(uint32_t v) { return __reduce_add_sync(kAll, v); }
__device__ __forceinline__ unsigned long long warp_total(unsigned long long v) {
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) v += __shfl_xor_sync(kAll, v, s);
    return v;
}
// the sum of the lanes below
template <class Sum>
__device__ __forceinline__ Sum warp_before(Sum v, int lane) {
    Sum sum = v;
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
        const Sum up = __shfl_up_sync(kAll, sum, s);
        if (lane >= s) sum += up;
    }
    return sum - v;
}

// words of shared memory a half-row of at most (nx + 1) / 2 pixels takes at any offset from a 16-byte boundary
__host__ __device__ constexpr size_t shared_row(int nx) { return (((size_t)nx + 1) / 2 + 3 + 3) / 4 * 4; }

// One warp takes one half-row.  What bounds the pass is reading the image (64 MB of a 4096^2 chip: 10 us at
// 6.8 TB/s): the warp reads its half-row with coalesced 16-byte loads, eight in flight a lane, and is done unless a pixel is
// above the full well.  The half-rows with saturated pixels are worked in shared memory, pixel after pixel
// from the left as the definition has it, but 32 distances at a time: lane k looks at the two pixels at
// distance d + k, a sum over the warp says whether the excess fills them all, and only the chunk in which the
// excess ends needs the prefix sum that finds the lane.  The pixels around the last saturated one that are
// known to have no room are skipped, so a run of saturated pixels does not search its own trail again.
// One thread a half-row, walking it in global memory, took 1302 us (kernel time) on a 4096^2 chip with 300
// stars and 3087 us on a crowded 1023 x 517 image; this form takes 28 us (2.4 TB/s; 4-byte loads: 39 us) and
// 23 us, where the chain of its fullest half-row is what is left.
// Sum: 32 bits where the room of 64 pixels fits them (a full well below 2^26), else 64.
// SHARED: the half-row fits the block's shared memory; otherwise it is worked in place.
template <bool SHARED, class Sum>
__global__ void bleed_kernel(uint32_t* __restrict__ img, int nx, int ny, uint32_t w, unsigned long long* removed) {
    extern __shared__ __align__(16) uint32_t rows[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long t = (long long)blockIdx.x * (blockDim.x >> 5) + warp;
    if (t >= 2ll * ny) return;
    const int y = (int)(t >> 1), half = (int)(t & 1);
    const int lo = half ? nx / 2 : 0, n = (half ? nx : nx / 2) - lo;
    uint32_t* const home = img + (size_t)y * nx + lo;
    // 16-byte loads from the boundary at or before the half-row, which keeps its offset in shared memory
    const int shift = (int)(((uintptr_t)home >> 2) & 3);
    uint32_t* const row = SHARED ? rows + (size_t)warp * shared_row(nx) + shift : home;
    int first = n, last = -1;                 // this lane's first and last saturated pixel
    for (int b = -shift; b < n; b += 32 * 4 * 8) {
        uint4 v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int x = b + 4 * (32 * k + lane);
            if (x >= 0 && x + 4 <= n) {
                v[k] = *reinterpret_cast<const uint4*>(home + x);
            } else {                          // the ends: the neighbours' pixels read as empty
                v[k].x = x >= 0 && x < n ? home[x] : 0u;
                v[k].y = x + 1 >= 0 && x + 1 < n ? home[x + 1] : 0u;
                v[k].z = x + 2 >= 0 && x + 2 < n ? home[x + 2] : 0u;
                v[k].w = x + 3 >= 0 && x + 3 < n ? home[x + 3] : 0u;
            }
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int x = b + 4 * (32 * k + lane);
            if (x >= n) continue;
            if (SHARED) *reinterpret_cast<uint4*>(row + x) = v[k];
            if (max(max(v[k].x, v[k].y), max(v[k].z, v[k].w)) > w) {
                first = min(first, v[k].x > w ? x : v[k].y > w ? x + 1 : v[k].z > w ? x + 2 : x + 3);
                last = v[k].w > w ? x + 3 : v[k].z > w ? x + 2 : v[k].y > w ? x + 1 : x;
            }
        }
    }
    first = __reduce_min_sync(kAll, first);
    last = __reduce_max_sync(kAll, last);
    if (last < 0) return;
    __syncwarp();
    // the pixels strictly between nl and nr are known to have no room
    int nl = 0, nr = 0;
    int touched_lo = first, touched_hi = last;
    unsigned long long lost = 0;
    for (int b = first & ~31; b <= last; b += 32) {
        const uint32_t here = b + lane < n ? row[b + lane] : 0u;
        // saturated pixels take no charge, before their turn or after it, so they are all set at once
        if (here > w) row[b + lane] = w;
        __syncwarp();
        unsigned above = __ballot_sync(kAll, here > w);
        while (above) {
            const int k = __ffs(above) - 1, x = b + k;
            above &= above - 1;
            unsigned long long e = __shfl_sync(kAll, here, k) - w;
            if (!(x > nl && x <= nr)) nl = nr = x;
            nl = min(nl, x - 1);
            nr = max(nr, x + 1);
            while (e > 0) {
                if (nl < 0 && nr >= n) { lost += e; break; }
                // the nearest distance at which there may be room
                const int d0 = nl < 0 ? nr - x : (nr >= n ? x - nl : min(x - nl, nr - x));
                const int xl = x - d0 - lane, xr = x + d0 + lane;
                const uint32_t vl = xl >= 0 ? row[xl] : w, vr = xr < n ? row[xr] : w;
                const uint32_t cl = vl < w ? w - vl : 0u, cr = vr < w ? w - vr : 0u;
                const Sum room = (Sum)cl + cr, total = warp_total(room);
                uint32_t gl = cl, gr = cr;
                int full = 32;                // lanes whose two pixels are filled (or have no room)
                if (total > e) {              // the excess ends in this chunk: prefix sum of the room over the distances
                    const Sum before = warp_before(room, lane), left = before < e ? (Sum)e - before : 0;
                    const Sum m = cl < cr ? cl : cr;
                    if (left <= 2 * m) {                  // alternating pairs, the odd one to the left
                        gl = (uint32_t)((left + 1) / 2);
                        gr = (uint32_t)(left / 2);
                    } else if (left < room) {             // one side fills; the other takes what it can
                        gl = (uint32_t)(m + (cl > m ? left - 2 * m : 0));
                        gr = (uint32_t)(m + (cr > m ? left - 2 * m : 0));
                    }
                    full = __ffs(__ballot_sync(kAll, left < room)) - 1;
                    e = 0;
                } else {
                    e -= total;
                }
                if (gl) row[xl] = vl + gl;
                if (gr) row[xr] = vr + gr;
                __syncwarp();
                nl = min(nl, x - d0 - full);
                nr = max(nr, x + d0 + full);
            }
            touched_lo = min(touched_lo, nl);
            touched_hi = max(touched_hi, nr);
        }
    }
    if (SHARED) {
        __syncwarp();
        for (int x = max(touched_lo, 0) + lane; x <= min(touched_hi, n - 1); x += 32) home[x] = row[x];
    }
    if (removed && lost && lane == 0) atomicAdd(removed, lost);
}

}  // namespace

extern "C" phosim_status phosim_bleed(uint32_t* image, int nx, int ny, uint32_t full_well, unsigned long long* removed,
                                      void* stream) {
    if (!image || nx < 2 || ny < 1) return PHOSIM_ERR_INVALID_ARGUMENT;
    // Blocks of up to four half-rows (four of 2048 pixels take 32 KB: seven blocks a SM), as many as fit the 48 KB
    // of shared memory that need no opt-in; a half-row of more than 12285 pixels is worked in place.
    constexpr size_t kMaxShared = 48u << 10;
    const size_t row_bytes = shared_row(nx) * sizeof(uint32_t);
    const bool shared = row_bytes <= kMaxShared;
    const int warps = shared ? (int)std::max<size_t>(1, std::min<size_t>(4, kMaxShared / row_bytes)) : 4;
    const unsigned blocks = (unsigned)((2ll * ny + warps - 1) / warps);
    const cudaStream_t st = (cudaStream_t)stream;
    const size_t bytes = shared ? (size_t)warps * row_bytes : 0;
    if (full_well < (1u << 26)) {
        const auto kernel = shared ? bleed_kernel<true, uint32_t> : bleed_kernel<false, uint32_t>;
        kernel<<<blocks, 32 * warps, bytes, st>>>(image, nx, ny, full_well, removed);
    } else {
        const auto kernel = shared ? bleed_kernel<true, unsigned long long> : bleed_kernel<false, unsigned long long>;
        kernel<<<blocks, 32 * warps, bytes, st>>>(image, nx, ny, full_well, removed);
    }
    if (cudaGetLastError() != cudaSuccess) return PHOSIM_ERR_CUDA;
    return PHOSIM_OK;
}
