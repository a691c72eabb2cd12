// Declarations of the sweep on staged tiles (sweep_tile.cu; planned by sweep_plan.h).
#pragma once
#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

namespace imf {

constexpr int kSwX = 8;                  // consecutive output rows per thread along the run axis
constexpr int kSwNU = 4, kSwNP = 2;      // warps of a block along the run axis and the plane axis
constexpr int kSwRows = kSwX * kSwNU;
constexpr int kSwThreads = 32 * kSwNU * kSwNP;
constexpr int kSwMaxL = 16;              // longest run (longer ones are split)
constexpr size_t kSwMaxSmem = 100 * 1024;

// A tool's tiles: nq output words of a row per tile, nl words of a source row per lane group (nq plus what the
// shifts reach), ppw planes per warp, UP the (odd) pitch of a column of rows in shared memory.
struct SwGeometry {
    int nq = 0, nl = 0, ppw = 0, UP = 0, somax = 0, planes = 0, words = 0;
    size_t smem = 0;
    // on average per orientation: a thread's shared loads, words a block stages, runs of the cutter along x
    double cost = 0, stage = 0, runs = 0;
};
struct SwOrient {
    int axis;                            // 0: runs along y, planes along z; 1: the other way; -1: no cutter voxels
    int eu, ew;                          // extents - 1 along the run axis and the plane axis
    int ou, ow;                          // window index of the first source row / plane of output 0
    int word0, words;                    // descriptors
};
struct SwArgs {
    const uint32_t *bits;                // free bits [slot][wz][wy][wpr]
    long b_so;
    int wpr, wy, wz;
    const SwOrient *head;
    const int *words;
    int nx, ny, nz, awords, orient_base, nb;
    uint32_t *A;                         // [nz][ny][awords]
    uint32_t *A_per;                     // per-orientation sets, or NULL
    long a_per_so;
    const int *perm;
    SwGeometry geo;
};
void launch_sweep_tile(const SwArgs &a, cudaStream_t s);

} // namespace imf
