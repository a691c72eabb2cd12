// Cooperative kernels of the 2D optimisation loop (topopt2d.cu): the multigrid-preconditioned
// conjugate gradient and the optimality-criteria update, each one launch.
#pragma once
#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

namespace imf_to {

constexpr int kMgThreads = 256;
constexpr int kMgMaxLevels = 32;
constexpr int kMgSmall = 1024;           // levels up to this many nodes run inside one block
constexpr int kMgCoarse = 32;            // nodes of the level solved by its inverse

// One grid of the hierarchy: nx x ny elements, nn nodes. S: assembled stencil, 36 planes of nn
// floats, plane ((dj + 1) * 3 + di + 1) * 4 + 2 a + b couples component a of a node with component b of
// its neighbour (di, dj); rows and columns of clamped dofs are 0. dinv: damped inverse diagonal.
struct MgLevel {
    int nx, ny, nn;
    int tw, th;                          // node tile of the up phase
    int cw, ch;                          // coarse-node tile of the restriction to the next level
    float *S, *dinv, *r, *z;             // r unused on the finest level (FP64 there)
    uint8_t *fixed;
};
struct MgArgs {
    MgLevel lv[kMgMaxLevels];
    int levels, first_small;             // first level that runs inside block 0
    const float *inv;                    // inverse of the coarsest operator, 2 nn x 2 nn
    const double *k0, *E, *force;
    const uint8_t *fixed;
    double *S64;                         // the finest stencil in FP64, the operator of the iteration
    double *x, *r0, *r1, *p0, *p1, *q;
    float omega;                         // Jacobi damping
    double *sc;                          // scalars, see kSc* (zeroed before the launch)
    unsigned *bar;                       // [0] barrier counter, [1] error (zeroed before the launch)
    double tol2;
    int max_iter, patience;              // most iterations, and most of them without the residual halving
};
enum { kScPq = 0, kScRr = 3, kScRz = 6, kScFf = 9, kScC = 10, kScIt = 11, kScDone = 12, kScLast = 13, kScN = 16 };
// Whether a solve's scalars can be used: it converged and no block gave up at a barrier. A block that did has left
// without its share of the compliance, while the others may still have passed that barrier and finished.
inline bool mg_converged(const double *sc, const unsigned *bar) { return sc[kScDone] == 1.0 && bar[1] == 0; }

// A hierarchy is five times what a handle holds without it. Above 256 MB (500,000 nodes) it is taken only where
// it is at most a sixteenth of the device memory still free after the handle's own arrays, so that handles made later
// find what they found before: on an empty device up to 33 million nodes (5800 x 5800).
constexpr size_t kMgFreeBytes = (size_t)256 << 20;
inline bool mg_affordable(size_t bytes, size_t room) { return bytes <= kMgFreeBytes || bytes <= room / 16; }

// device bytes of the hierarchy's arrays; fills every level's sizes (0: too many levels)
size_t mg_plan(int nx, int ny, double nu, MgArgs &a);
// places the arrays of a planned hierarchy in `mem` (mg_plan bytes)
void mg_place(MgArgs &a, void *mem);
// assembles the stencils, the coarse operators and the inverse for the current moduli
void mg_setup(const MgArgs &a, cudaStream_t s);
// solves; results in a.x and a.sc
cudaError_t mg_solve(const MgArgs &a, cudaStream_t s);

struct OcArgs {
    long n;
    const float *xi, *S;
    const uint8_t *passive;
    double volfrac, move, eta, beta;
    double *xs;                          // xi S^eta (n doubles of scratch)
    float *out;
    double *sc;                          // [0..5] volume and slope sums, three pairs in turn, [6] count,
                                         // [7] change, [8] final volume (zeroed before the launch)
    unsigned *bar;
};
cudaError_t oc_solve(const OcArgs &a, cudaStream_t s);

} // namespace imf_to
