// Batched execution: many lattices of different sizes advanced together.
//
// Each member lattice is described on the device by a LatDesc (its buffers,
// geometry, parameters and row-segment length).  One step of the batch is one
// launch:
//   k_batch_interior: a persistent kernel whose blocks take items from a shared
//                     counter until the list is exhausted: first the members'
//                     near-wall tiles (wall_tile), then their interior
//                     tiles (member, strip, segment), running the same tile
//                     code as the single-lattice kernels;
//   k_batch_tile:     for batches whose members together are small enough for
//                     k_step_tile: two tiles of 32 x 8 nodes per item.
// The item counts live in device memory, so one captured CUDA graph of a pair
// of steps of k_batch_interior stays valid when the membership changes.
#pragma once
#include "tlbm_kernels.cuh"
#include "tlbm_tile.cuh"

namespace tlb {

template <typename R>
struct LatDesc {
    const void* buf[2];  // distribution buffers; steps of parity p read buf[p], write buf[p ^ 1]
    void* cu;
    const uint8_t* cls;
    Geo g;
    Prm<R> P;
    int rows;  // row-segment length of this member's tiles
};

struct TileItem {
    int lat, bx, by;
};

struct WallItem {
    int lat;
    uint32_t packed;  // (row << 16) | column of a near-wall tile of 32 x (threads / 32) nodes
};

constexpr int kBatchTY = 8;  // rows of a tile of k_batch_tile

struct BatchCounters {
    int n_tiles, n_wall;
    int next, done;  // items taken and blocks finished of the running launch (zero between launches)
};

// The near-wall tiles go through the interior kernel's own queue, before the
// interior tiles: as a launch of their own beside it they either waited for
// the persistent blocks, which fill every register file, or kept some of them
// from starting (32 lattices of 64..512 nodes a side, FP32, GB300: 109
// -> 99 us per step).
template <typename S, typename R, int BLOCK, bool PREFETCH, int MINB, bool MRT>
__global__ void __launch_bounds__(BLOCK, MINB)
k_batch_interior(const LatDesc<R>* __restrict__ descs, const TileItem* __restrict__ items,
                 const WallItem* __restrict__ walls, BatchCounters* ctr, int parity)
{
    constexpr int WTY = BLOCK / 32;
    constexpr bool kStash = kStashPops && std::is_same<R, float>::value && !kDenseMrt<S, MRT>;
    __shared__ MarchShared<R, BLOCK, kStash> sh;
    __shared__ Prm<R> Ps;
    __shared__ int item_s;
    static_assert(sizeof(Prm<R>) % sizeof(R) == 0, "params are whole words");
    constexpr int kWords = (int)(sizeof(Prm<R>) / sizeof(R));
    const int nw = ctr->n_wall, n = nw + ctr->n_tiles;
    // the state, and the counters, are those of the previous launch
    after_previous_launch();
    for (;;) {
        if (threadIdx.x == 0) item_s = atomicAdd(&ctr->next, 1);
        __syncthreads();
        const int it = item_s;
        if (it >= n) break;
        const bool wall = it < nw;
        const TileItem ti = wall ? TileItem{walls[it].lat, (int)(walls[it].packed & 0xffffu), (int)(walls[it].packed >> 16)}
                                 : items[it - nw];
        const LatDesc<R>* d = descs + ti.lat;
        for (int i = threadIdx.x; i < kWords; i += BLOCK)
            reinterpret_cast<R*>(&Ps)[i] = reinterpret_cast<const R*>(&d->P)[i];
        __syncthreads();
        const Geo g = d->g;
        const S* fA = global_ptr((const S*)d->buf[parity]);
        S* fB = global_ptr((S*)d->buf[parity ^ 1]);
        CuT<S>* cu = global_ptr((CuT<S>*)d->cu);
        // members with equal densities and viscosities take the uniform-property
        // update, as they do when stepped alone (the branch is uniform per tile)
        auto* st = reinterpret_cast<PopStash<R, BLOCK>*>(&sh.m.stash);  // used only when kStash
        if (wall)
            wall_tile<S, R, WTY, MRT>(fA, fB, cu, d->cls, g, Ps, ti.bx, ti.by, sh.tile);
        else if (Ps.uni != R(0))
            interior_tile<S, R, BLOCK, PREFETCH, MRT, true, kStash>(fA, fB, cu, d->cls, g, Ps, ti.bx, ti.by, d->rows,
                                                                    sh.m.rings, st);
        else
            interior_tile<S, R, BLOCK, PREFETCH, MRT, false, kStash>(fA, fB, cu, d->cls, g, Ps, ti.bx, ti.by, d->rows,
                                                                     sh.m.rings, st);
        __syncthreads();  // shared data, parameters and item_s are reused by the next item
    }
    // the last block leaves the counters as the next launch expects them
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&ctr->done, 1) == (int)gridDim.x - 1) {
            ctr->next = 0;
            ctr->done = 0;
        }
    }
}

// Blocks 2i, 2i + 1: the left and right tile of 32 x kBatchTY nodes of item i
// (columns 64 bx .., rows kBatchTY by ..).
template <typename S, typename R, int MINB, bool MRT>
__global__ void __launch_bounds__(32 * kBatchTY, MINB)
k_batch_tile(const LatDesc<R>* __restrict__ descs, const TileItem* __restrict__ items, int parity)
{
    __shared__ TileShared<R, kBatchTY> sh;
    __shared__ Prm<R> Ps;
    constexpr int kWords = (int)(sizeof(Prm<R>) / sizeof(R));
    const TileItem ti = items[blockIdx.x >> 1];
    const LatDesc<R>* d = descs + ti.lat;
    const int x0 = ti.bx * 64 + (blockIdx.x & 1) * 32;
    if (x0 >= d->g.nx) return;
    for (int i = threadIdx.x; i < kWords; i += 32 * kBatchTY)
        reinterpret_cast<R*>(&Ps)[i] = reinterpret_cast<const R*>(&d->P)[i];
    __syncthreads();
    const Geo g = d->g;
    const S* fA = (const S*)d->buf[parity];
    S* fB = (S*)d->buf[parity ^ 1];
    const int y0 = ti.by * kBatchTY - tile_shift(g.edge[3] == EDGE_LID, g.ny, kBatchTY);
    if (Ps.uni != R(0))
        tile_step<S, R, kBatchTY, MRT, true, false>(fA, fB, (CuT<S>*)d->cu, d->cls, g, Ps, x0, y0, sh);
    else
        tile_step<S, R, kBatchTY, MRT, false, false>(fA, fB, (CuT<S>*)d->cu, d->cls, g, Ps, x0, y0, sh);
}

}  // namespace tlb
