// Declarations of the streamed minimum over sharp points (erode_stream.cu; planned by
// erode_stream.h).
#pragma once
#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

namespace imf {

// A block owns kEsTX x kEsRows x kEsW outputs (x, run axis u, plane axis w) in units of 8 x kEsX x 4:
// a warp reduces a unit's runs with lane = x + 8 * plane and kEsX consecutive outputs along u a thread.
constexpr int kEsX = 8, kEsNU = 3, kEsNW = 2, kEsTX = 32;
constexpr int kEsRows = kEsX * kEsNU, kEsW = 4 * kEsNW;
constexpr int kEsMaxL = 16;                // longest run (longer ones are split)
constexpr int kEsUnits = (kEsTX / 8) * kEsNU * kEsNW;
constexpr int kEsWarps = 24;               // warps that reduce
constexpr int kEsProducers = 32 * 4;       // threads that copy
constexpr int kEsThreads = 32 * kEsWarps + kEsProducers;
constexpr int kEsMaxStages = 10, kEsSlots = 4;   // slots: see the producer
constexpr int kEsShare = 256;              // most orientations of one block
constexpr size_t kEsAccBytes = (size_t)kEsUnits * kEsX * 32 * 4;
constexpr size_t kEsBudget = 225 * 1024 - kEsAccBytes;   // ring and descriptor slots
static_assert(kEsUnits <= 32, "the live units of a tile are one word");

// row pitches (floats) the kernel is built for, multiples of 4 (16-byte copies)
__host__ __device__ constexpr int es_pitch(int need)
{
    return need <= 44 ? 44 : need <= 64 ? (need + 3) & ~3 : need <= 76 ? 76 : 0;
}

// runs of length L that one step of a list takes where it can: short runs do not fill a step alone
__host__ __device__ constexpr int es_unroll(int L) { return L == 1 ? 4 : L <= 9 ? 2 : 1; }

struct EsGeometry {
    int P = 0, R = 0, Q = 0, stages = 0;   // row pitch, rows per plane, plane pitch, stages of four planes
    int words = 0;                         // descriptor words of a slot (the most any orientation has)
    double cost = 0;                       // shared loads of a thread per orientation, on average
};

struct EsOrient {
    int axis;                        // 0: runs along y, planes along z; 1: runs along z, planes along y; -1: no points
    int lists;                       // lists, four source planes each
    int rows, quads;                 // rows and 16-byte columns a plane copies
    int ox, ou, ow;                  // tile origin = block output origin + (ox, ou, ow) in window index
    int word0, words;                // descriptor words, multiples of 4
};

// Output tiles of a grid: along x, and along the run and plane axis of either kind of orientation.
struct EsTiles {
    int x, u[2], w[2];
    __host__ __device__ int kind(int a) const { return x * u[a] * w[a]; }
};
inline EsTiles es_tile_counts(int nx, int ny, int nz)
{
    auto up = [](int n, int d) { return (n + d - 1) / d; };
    EsTiles t{};
    t.x = up(nx, kEsTX);
    t.u[0] = up(ny, kEsRows); t.w[0] = up(nz, kEsW);
    t.u[1] = up(nz, kEsRows); t.w[1] = up(ny, kEsW);
    return t;
}

// What a producer's orientation begins with, the same for every producer.
enum class EsOpen { copy, done, leave };

// Control flow of one producer thread over its `orientations` and the ring's `stages`. Io: steps(k), the stages of
// orientation k; wait(st, phase), bounded, false when stage st was not given back in time; open(k, st, late), the
// barrier that every producer of the block passes once an orientation, which is where they learn together that one
// of them is late (leave) or that no output has work left (done); copy(k, s, st). A late thread copies nothing
// more but goes on to that barrier: it counts all of them, and one that had left would hold the others there
// without limit.
template <class Io> __host__ __device__ __forceinline__ EsOpen es_produce(Io &io, int orientations, int stages)
{
    int st = 0;
    uint32_t ph = 0;
    bool wrapped = false, late = false;
    for (int k = 0; k < orientations; ++k) {
        const int steps = io.steps(k);
        for (int s = 0; s < steps; ++s) {
            if (wrapped && !late && !io.wait(st, ph ^ 1)) late = true;
            if (s == 0) {
                const EsOpen o = io.open(k, st, late);
                if (o != EsOpen::copy) return o;
            }
            if (late) continue;
            io.copy(k, s, st);
            if (++st == stages) { st = 0; ph ^= 1; wrapped = true; }
        }
    }
    return late ? EsOpen::leave : EsOpen::copy;
}

struct EsArgs {
    const float *g;
    long g_so;
    int gpx, wx, wy, wz;
    const EsOrient *head;
    const int *words;
    int nx, ny, nz, orient_base, nb;
    int kind[2];                     // orientations of the launch with either run axis
    int ngroups;                     // blocks per tile and run axis; each takes its share of the orientations
    float *f;
    int *status;
    EsGeometry geo;
};
// false (nothing launched) where no instance applies
bool launch_erode_stream(const EsArgs &a, cudaStream_t s);

} // namespace imf
