// Tile sort of one species' particle store (single-run launches).
//
// Two orders, both grouping particles by tile (tiles and cells in a tile numbered x-fastest);
// rank = the particle's rank among the particles of its cell in the previous order:
//  * cell-major (FP32 form): by (tile, cell, rank).  A warp's 32 consecutive particles sit in
//    one cell or two neighbouring ones: shared-memory gathers broadcast, and the warp's
//    Esirkepov currents are summed in registers before they reach shared memory.
//  * slot-major (FP64 form): by (tile, rank, cell).  A tile runs through groups holding one
//    particle of every cell with more than `rank` particles, so a warp's lanes sit in 32
//    different cells and their per-lane shared-memory atomics do not collide.
// Both orders are stable and a pure function of the cells of the previous order: the same on
// every run, whatever the order in which the atomics of the counting stage were served.
//
//   1. count    : tile-major cell key per particle, its count and a provisional place
//   2. tile_sum : particles per tile;  scan: exclusive scan over tiles -> tile_start
//   3. layout   : one CTA per tile; first position of every cell (cell-major) and, for the
//                 slot-major order, the position of every (cell, rank)
//   4. place    : every particle index at its provisional cell-major position
//   5. scatter  : per cell-major position, the rank of its particle in its cell (indices below
//                 it in the cell's segment); the particle is copied to the position of that
//                 rank in the other buffer
//
// A run whose scratch sets all fit (RunDev::sc_more) sorts its species side by side, blockIdx.y
// naming the species, and a grid of few keys takes stages 2 and 3 in one launch: a sort of a small
// run is launches of about 4 us each, whatever they do.  Two species of 64x32 cells: 14 launches
// -> 5 per sort; 50 steps with 8 or 9 sorts 2146 -> 1780 us (FP32 form), 2285 -> 1973 (FP64 form).
#include "pic_launch.h"
#include "pic_sort_dev.cuh"

namespace pic {

namespace {

constexpr int kBlock = 256;
// keys per thread of a tile's block up to which the block sums the counts before it itself
constexpr int64_t kFewKeys = 64;

__global__ void __launch_bounds__(kBlock) k_zero_cnt(const __grid_constant__ RunDev rd, int64_t nkeys)
{
    const SortScratch sc = sort_scratch(rd, blockIdx.y);
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < nkeys) sc.cnt[i] = 0;
}

__global__ void __launch_bounds__(kBlock) k_count(const __grid_constant__ RunDev rd, int s0)
{
    const SortScratch sc = sort_scratch(rd, blockIdx.y);
    const int s = s0 + blockIdx.y;
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p < rd.sp[s].n) sort_count_one(rd, sc, s, p);
}

__global__ void k_tile_sum(const __grid_constant__ RunDev rd)
{
    sort_tile_sum_block(rd, sort_scratch(rd, blockIdx.y), blockIdx.x);
}

__global__ void k_scan(const __grid_constant__ RunDev rd, int s0)
{
    sort_scan_block(sort_scratch(rd, blockIdx.x).tile_count, rd.sp[s0 + blockIdx.x].tile_start,
                    rd.ntiles);
}

__global__ void k_layout(const __grid_constant__ RunDev rd, int s0)
{
    sort_layout_block(rd, sort_scratch(rd, blockIdx.y), rd.sp[s0 + blockIdx.y].tile_start[blockIdx.x],
                      blockIdx.x);
}

__global__ void k_start_layout(const __grid_constant__ RunDev rd, int s0)
{
    sort_start_layout_block(rd, sort_scratch(rd, blockIdx.y), rd.sp[s0 + blockIdx.y].tile_start,
                            blockIdx.x);
}

__global__ void __launch_bounds__(kBlock) k_place(const __grid_constant__ RunDev rd, int s0)
{
    const SortScratch sc = sort_scratch(rd, blockIdx.y);
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p < rd.sp[s0 + blockIdx.y].n) sort_place_one(sc, p);
}

__global__ void __launch_bounds__(kBlock) k_scatter(const __grid_constant__ RunDev rd, int s0)
{
    const SortScratch sc = sort_scratch(rd, blockIdx.y);
    const int s = s0 + blockIdx.y;
    const int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r < rd.sp[s].n) sort_scatter_one(rd, sc, s, r);
}

}  // namespace

cudaError_t launch_sort(const RunDev &rd, int s0, int ns, cudaStream_t st, int64_t *launches)
{
    const int TC = rd.tile[0] * rd.tile[1] * rd.tile[2];
    const int64_t nkeys = rd.ntiles * TC;
    auto blocks = [](int64_t n) { return (unsigned)((n + kBlock - 1) / kBlock); };
    int64_t n = 0;
    for (int s = s0; s < s0 + ns; ++s) n = rd.sp[s].n > n ? rd.sp[s].n : n;
    const dim3 tiles((unsigned)rd.ntiles, ns), parts(blocks(n), ns);
    const int tb = ((TC + 31) / 32) * 32;
    k_zero_cnt<<<dim3(blocks(nkeys), ns), kBlock, 0, st>>>(rd, nkeys);
    if (n > 0) k_count<<<parts, kBlock, 0, st>>>(rd, s0);
    if (nkeys <= kFewKeys * tb && nkeys <= 65536) {
        k_start_layout<<<tiles, tb, 0, st>>>(rd, s0);
        *launches += 2;
    } else {
        k_tile_sum<<<tiles, tb, 0, st>>>(rd);
        k_scan<<<ns, 1024, 0, st>>>(rd, s0);
        k_layout<<<tiles, tb, 0, st>>>(rd, s0);
        *launches += 4;
    }
    if (n > 0) {
        k_place<<<parts, kBlock, 0, st>>>(rd, s0);
        k_scatter<<<parts, kBlock, 0, st>>>(rd, s0);
        *launches += 3;
    }
    return cudaGetLastError();
}

}  // namespace pic
