// lr_bins.cuh -- binning of the LR set in three launches and no clears.
//   arrive  one thread per particle (fused with whatever computes its
//           position): its cell's count, its place in the cell's bucket of
//           kBucket indices in order of arrival, and the count of the cell's
//           tile of kBinTile cells (summed per block in shared memory first);
//   scan    one block per tile: the counts of the tiles before it, then the
//           tile's own exclusive scan, into the cell starts;
//   place   one thread per particle: its rank among the indices of its cell
//           is its place in the stable order, and it copies itself there.
// Every launch leaves what the next binning counts in at zero: place clears
// the counts, scan moves the flag that later kernels read out of the word that
// arrive adds to.  A particle beyond kBucket of its cell (a 3 r_LR cube holds
// 8 LR particles of a 2 r_LR lattice) goes to one list of all cells; the scan
// block of its tile puts it from there where its cell's particles find it next
// to the others of the cell, so that a rank costs the cell's own count.  In
// cells of more than kCrowd a warp counts its particles' cell together, which
// divides that by 32 again.
// A binning is a chain of dependent launches, so their number and each one's
// latency bound it: clear, keys, two scan launches, scatter and a per-cell
// order that copied cell by cell in one thread before.  With the candidate
// search they took 30 us of an LR step on the digging bed (50,527 LR, 33,213
// cells) and take 15; gs_bin_low by itself 31 us, now 17 (launches included).
#pragma once

#include <cuda_runtime.h>

#include "grid.cuh"
#include "gs_internal.cuh"

constexpr int kBucket = 16;
// Counted by a thread up to here, by a warp beyond: of 50,527 LR in cells of
// 1,024 84 and 139 us, of 4,096 176 and 221, of 16,384 586 and 346; of 202,112
// 313 and 277, 885 and 806, 2,114 and 1,385.
constexpr uint32_t kCrowd = 2048;
constexpr int kBinTile = 4096;       // cells per tile of the scan
constexpr int kMaxBinTiles = 1024;   // beyond that (4 M cells) the general counting sort

// Clears the block's tile counts (s_tile: b.n_tiles words); a barrier follows
// in bins_arrive's callers.
__device__ __forceinline__ void bins_begin(const LrBins& b, uint32_t* s_tile)
{
    for (int t = threadIdx.x; t < b.n_tiles; t += blockDim.x) s_tile[t] = 0u;
    __syncthreads();
}

__device__ __forceinline__ void bins_arrive(const LrBins& b, uint32_t* s_tile, uint32_t cell, uint32_t i)
{
    const uint32_t rank = atomicAdd(b.count + cell, 1u);
    if (rank < (uint32_t)kBucket) b.bucket[(size_t)cell * kBucket + rank] = i;
    else b.spill[atomicAdd(b.words + kBinSpill, 1u)] = make_uint4(i, cell, rank, 0u);
    atomicAdd(s_tile + cell / kBinTile, 1u);
}

// The same by the lanes `mask` of a warp without the block's help (the last
// pass of a step): lanes of the same tile add to it once.
__device__ __forceinline__ void bins_arrive_warp(const LrBins& b, unsigned mask, uint32_t cell, uint32_t i)
{
    const uint32_t rank = atomicAdd(b.count + cell, 1u);
    if (rank < (uint32_t)kBucket) b.bucket[(size_t)cell * kBucket + rank] = i;
    else b.spill[atomicAdd(b.words + kBinSpill, 1u)] = make_uint4(i, cell, rank, 0u);
    const unsigned peers = __match_any_sync(mask, cell / kBinTile);
    if ((int)(threadIdx.x & 31u) == __ffs(peers) - 1) atomicAdd(b.tile + cell / kBinTile, (uint32_t)__popc(peers));
}

// Adds the block's tile counts to the tiles' (after every thread's arrival).
__device__ __forceinline__ void bins_end(const LrBins& b, uint32_t* s_tile)
{
    __syncthreads();
    for (int t = threadIdx.x; t < b.n_tiles; t += blockDim.x)
        if (s_tile[t]) atomicAdd(b.tile + t, s_tile[t]);
}
