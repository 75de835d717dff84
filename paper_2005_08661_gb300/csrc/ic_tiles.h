// ic_tiles.h -- tiles of the IC(0) sweeps (k_ic.cu), and what fm_set_data records of a support mask for them
// and for the drop-tolerance IC's row wavefront (k_ict.cu): which steps of a tile or row group reach a mask
// voxel, and the tiles that hold any in claim order.
//
// Both follow from the mask alone, so their blocks run in the launches that count the mask voxels and scan the counts
// (k_setup.cu): fm_set_data of 64 x 64 x 16 voxels, back to back, 36.3 us without them, 39.5 so, 52.1 as
// launches of their own behind the setup kernel; the row groups of 256 x 256 x 128 376, 386 and 459 us (with
// a thread to a row).
#pragma once
#include "fm_internal.h"

namespace fm {

__device__ __forceinline__ bool in_mask(const uint8_t* mask, long long j) { return mask ? mask[j] != 0 : true; }

#ifndef FM_IC_CSF
#define FM_IC_CSF 4
#endif
#ifndef FM_IC_CSB
#define FM_IC_CSB 4
#endif
#ifndef FM_IC_FWF
#define FM_IC_FWF 2
#endif
#ifndef FM_IC_FWB
#define FM_IC_FWB 3
#endif
constexpr int kTX = kTileX, kTY = kTileY, kTZ = 8;  // 64 x 16 x 8 voxels
constexpr int kRows = kTY * kTZ;                     // rows along x: one per compute thread
constexpr int kWarps = kRows / 32;                   // compute warps, two z planes each
constexpr int kVox = kTX * kRows;
static_assert(kTX == 64 && kTY == 16 && kWarps == 4, "lane = (y, plane of the warp's pair)");
// Steps per chunk (the unit of the face hand-off, of the barrier between the warps and of
// their lag), and the warps that fetch incoming faces, taking the chunks in turn, so that the
// polls for consecutive chunks are in flight together (a poll round trip is about 0.7 us, a chunk
// 0.2 to 0.4).  Forward / back substitution on 256 x 256 x 128 (us), measured before the dot products
// moved behind the back substitution (which made it 109): chunks of 4 with 2 fetch warps 122 / 97, with 3
// 125 / 98, with 4 127 / 103; chunks of 3 with 3 130 / 95, of 2 with 4 146 / 101, of 6 with 2 126 / 104.
constexpr int kCSF = FM_IC_CSF, kCSB = FM_IC_CSB;
constexpr int kFetchF = FM_IC_FWF, kFetchB = FM_IC_FWB;
// compute warps, one warp that publishes the outgoing faces, fetch warps
constexpr int kThreadsF = kRows + 32 + 32 * kFetchF, kThreadsB = kRows + 32 + 32 * kFetchB;
constexpr int kSweep = kRows + 32;  // threads that meet at the end of a chunk: compute and publishing warps

// First step of plane lz with chunks of C steps: the two planes of a warp follow each other by
// one step, and each warp starts C + 1 steps after the warp below.
template <int C> __host__ __device__ constexpr int tz(int lz) { return (C + 1) * (lz >> 1) + (lz & 1); }

// Steps of one tile that reach a mask voxel, packed as TileLists.range holds them.  256 threads, half a
// row each.
__device__ __forceinline__ void tile_steps(const Geo& geo, const uint8_t* mask, int ntx, int nty, int tile,
                                           unsigned* range) {
    static_assert(kTX == 64, "half a row in a word's bits");
    __shared__ int s_lim[4];
    const int X = tile % ntx, Y = (tile / ntx) % nty, Z = tile / (ntx * nty);
    const int row = threadIdx.x >> 1, ly = row % kTY, lz = row / kTY;
    const int y = Y * kTY + ly, z = Z * kTZ + lz, half = (threadIdx.x & 1) * (kTX / 2), x0 = X * kTX + half;
    if (threadIdx.x < 4) s_lim[threadIdx.x] = (threadIdx.x & 1) ? 0 : 255;
    __syncthreads();
    if (y < geo.ny && z < geo.nz) {
        const long long j0 = ((long long)z * geo.ny + y) * geo.nx + x0;
        const int n = min(kTX / 2, geo.nx - x0);
        unsigned bits = 0;
#pragma unroll
        for (int i = 0; i < kTX / 2; ++i) bits |= i < n && in_mask(mask, j0 + i) ? 1u << i : 0u;
        if (bits) {
            const int lo = half + __ffs(bits) - 1, hi = half + 31 - __clz(bits);
            const int f = ly + tz<kCSF>(lz), b = (kTY - 1 - ly) + tz<kCSB>(kTZ - 1 - lz);
            atomicMin(&s_lim[0], lo + f);
            atomicMax(&s_lim[1], hi + f);
            atomicMin(&s_lim[2], kTX - 1 - hi + b);
            atomicMax(&s_lim[3], kTX - 1 - lo + b);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0)
        range[tile] = (unsigned)s_lim[0] | (unsigned)s_lim[1] << 8 | (unsigned)s_lim[2] << 16 | (unsigned)s_lim[3] << 24;
}

// First and last step of a row group (32 rows of a plane) that reach a mask voxel, forward (x + 2 lane) and
// mirrored (nx - 1 - x + 2 (31 - lane)).  256 threads, four rows to a warp.
__device__ __forceinline__ void row_steps(const Geo& geo, const uint8_t* mask, int u, int4* rows) {
    __shared__ int s_lo[2], s_hi[2];
    const int nyb = (geo.ny + 31) / 32, z = u / nyb, y0 = (u % nyb) * 32, lane = threadIdx.x & 31;
    if (threadIdx.x < 2) {
        s_lo[threadIdx.x] = 1 << 30;
        s_hi[threadIdx.x] = -(1 << 30);
    }
    __syncthreads();
    const int l0 = (threadIdx.x >> 5) * 4, nrow = min(4, geo.ny - y0 - l0);  // this warp's rows
    int lo[4], hi[4];                                                         // of this lane's columns
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        lo[k] = 1 << 30;
        hi[k] = -1;
    }
    const long long j0 = ((long long)z * geo.ny + y0 + l0) * geo.nx;
#pragma unroll 4
    for (int x = lane; x < geo.nx; x += 32)
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (k < nrow && in_mask(mask, j0 + (long long)k * geo.nx + x)) {
                lo[k] = min(lo[k], x);
                hi[k] = x;
            }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        lo[k] = __reduce_min_sync(0xffffffffu, lo[k]);
        hi[k] = __reduce_max_sync(0xffffffffu, hi[k]);
        if (lane == 0 && hi[k] >= 0) {
            const int l = l0 + k;
            atomicMin(&s_lo[0], lo[k] + 2 * l);
            atomicMax(&s_hi[0], hi[k] + 2 * l);
            atomicMin(&s_lo[1], geo.nx - 1 - hi[k] + 2 * (31 - l));
            atomicMax(&s_hi[1], geo.nx - 1 - lo[k] + 2 * (31 - l));
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) rows[u] = make_int4(s_lo[0], s_hi[0], s_lo[1], s_hi[1]);
}

// The lists of the tiles that hold a mask voxel, in claim order: list 0 those of the forward order
// (out[0..ntiles)), list 1 those of the back substitution's (out[ntiles..)), and list 2, in the same order,
// the tiles that stand for a dot-product unit: a unit is a pair of tiles Y = 2k, 2k + 1 and belongs to the
// lower one (the later of the two to be swept back) if that is not empty.  1024 threads.
__device__ __forceinline__ void list_tiles(const TileLists& a, int list) {
    __shared__ int s_warp[32], s_base;
    constexpr int U = 4;  // tiles of a thread, their loads in flight together
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int* in = a.order + (list == 0 ? 0 : a.ntiles);
    int* out = a.out + (size_t)list * a.ntiles;
    auto empty = [&](int t) { return (a.range[t] & 255u) == 255u; };
    if (threadIdx.x == 0) s_base = 0;
    __syncthreads();
    for (int b = 0; b < a.ntiles; b += 1024 * U) {
        int t[U], n = 0;
        bool keep[U];
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int i = b + U * threadIdx.x + k;
            t[k] = i < a.ntiles ? in[i] : -1;
        }
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const bool upper = list == 2 && t[k] >= 0 && ((t[k] / a.ntx) % a.nty & 1);
            keep[k] = t[k] >= 0 && !empty(t[k]) && (!upper || empty(t[k] - a.ntx));
            n += keep[k];
        }
        int incl = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) s_warp[wid] = incl;
        __syncthreads();
        int at = s_base + incl - n, tot = 0;
        for (int w = 0; w < 32; ++w) {
            if (w < wid) at += s_warp[w];
            tot += s_warp[w];
        }
#pragma unroll
        for (int k = 0; k < U; ++k)
            if (keep[k]) out[at++] = t[k];
        __syncthreads();
        if (threadIdx.x == 0) s_base += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0 && list != 1) a.istate[list == 0 ? I_NTILE : I_NUNIT] = s_base;
}

}  // namespace fm
