// Geometry and index helpers of the kernels that take a tile of the grid per
// block through shared memory: the FP32 step (step_tile.cu) and its adjoint
// (adjoint_tile.cu).  Threads work on pairs of neighbouring columns.
#pragma once

#include "chain.cuh"
#include "lattice.cuh"

namespace fdlbm {
namespace {

constexpr int kTX = 32, kTY = 16, kTP = kTX / 2;  // tile; pairs per row
constexpr int kNT = kTP * kTY;                    // threads, one per pair of the tile
constexpr int kAP = kTP + 4, kAR = kTY + 8;       // region of stage A: pairs per row, rows
constexpr int kBP = kTP + 2, kBR = kTY + 4;       // region of stage B
constexpr int kARing = kAP * kAR - kNT, kBRing = kBP * kBR - kNT;  // pairs around the tile
static_assert(kARing <= kNT && kBRing <= kNT, "one pass over the ring");

// Tiles of `size` nodes along an axis of n; a wall node goes with its interior
// neighbour's tile.
__host__ __device__ __forceinline__ int tiles_along(int n, bool wall, int size)
{
    return (n - (wall ? 1 : 0) + size - 1) / size;
}

// Rows of tiles of one launch (the limit of gridDim.y).  A taller grid takes more
// launches of an instance of its own, each with its first row as an argument: in
// the common instance that argument cost the adjoint 0.7 % (2048^2 rollout), and
// one launch over a linear block index, with a division per block, made the forced
// step spill (1000^2 34.1 us against 32.1).
constexpr int kMaxTileRows = 65535;

// Index k of an axis of n nodes: wrapped on a periodic axis, the nearest node
// on a walled one.
__device__ __forceinline__ int axis_index(int k, int n, bool wall)
{
    if (wall) return min(max(k, 0), n - 1);
    if (k < 0) k += n;
    if (k >= n) k -= n;
    return (unsigned)k < (unsigned)n ? k : wrap_index(k, n);
}

// Pair c, row r of site q of the ring around the tile, in the region of
// (kTP + H) pairs x (kTY + 2 H) rows: rows below and above, then the sides.
template <int H>
__device__ __forceinline__ void ring_site(int q, int &c, int &r)
{
    constexpr int W = kTP + H;  // H/2 pairs on each side
    if (q < 2 * H * W) {
        r = q / W;
        c = q - r * W;
        if (r >= H) r += kTY;
    } else {
        q -= 2 * H * W;
        r = q / H;
        c = q - r * H;
        r += H;
        if (c >= H / 2) c += kTP;
    }
}

}  // namespace
}  // namespace fdlbm
