// TMA-fed persistent axis pass of the two-pass register FFT (fft2.cuh): the y and z passes of
// the collision convolution's transforms (Alg. 1 Convolve; App. B's FFT convolution term),
// with the pointwise product of the design and tool spectra fused into the z pass.
//
// The arithmetic is the one of axis2_kernel (fft2_kernels.cu); what changes is how the pencils
// reach the registers. A block stays resident and walks a strided list of work items (kx
// chunk, orientation, batch row). For each item the tensor memory accelerator copies the W
// pencils of the chunk (and the W pencils of the pointwise factor) into shared memory as [row
// j][pencil w]; zero padding of short inputs comes from the copy's out-of-bounds fill. Results go
// straight from registers to global memory.
//
// Two stages alternate: the copy of the block's next item is in flight while this one is transformed. What
// bounds a pass is how many items an SM has in hand (barriers and waits of one block leave the SM to the others)
// and how many bytes it has in flight. Each split (A, B) is its own kernel with 16 A threads, so that its registers
// are its own (one kernel with every split inside took the largest one's, 112 to 124). Where both factors are at most
// 16 (lengths up to 256, but not 147, 162, 189, 200, 216 or 252, which split into larger ones) the tile between the two
// DFT passes lies in the item's own stage, which pass 1 has read into registers by then: two to four blocks an SM,
// where a tile buffer left room for one with the factor. With a larger factor one block with a tile of its own stays: two with the tile in the stage took 11.2 ms for the 256^3 y pass against 6.0 (a single stage a
// block likewise, 11.5 and 10.8 for the z pass against 7.2). Measured, ms a step, against one kernel per shape:
// z pass with the factor 128^3 x 64 0.787 -> 0.694, 144^3 x 96 1.70 -> 1.52, 75 x 61 x 50 x 24 0.090 -> 0.063, 48^3 x 24 0.068 ->
// 0.047; 256^3 x 128 z 7.40 -> 7.25, y 6.18 -> 5.98. The inverse passes without the factor are held to 80 registers
// and some spill there (16 x 15: 80 bytes); over lengths 64 to 420 none is slower for it than one kernel per shape was
// (8 orientations, us: 240 35.0 -> 29.6, 224 33.2 -> 28.7, 210 33.5 -> 27.8).
//
// Every wait on a copy is bounded (%globaltimer); on a timeout the block records
// IMF_ERR_TIMEOUT in the status word, waits (bounded again) for the copies it still has in
// flight and returns, so no copy lands in shared memory that a later block owns.
#pragma once
#include <cuda.h>

#include "fft2.cuh"
#include "imf.h"
#include "imf_internal.cuh"
#include "tc_primitives.cuh"

namespace imf {
namespace tma_fft {

constexpr int kStages = 2;

int sm_count();   // multiprocessors of the current device (fft_tma.cu)
// Tiled tensor map of 8-byte elements (complex64): dims innermost first, strides of dims 1.. in
// bytes, box in elements; false when a tensor map cannot describe it (fft_tma.cu).
bool encode_tiled(CUtensorMap *m, const void *ptr, int rank, const uint64_t *dims, const uint64_t *strides_bytes,
                  const uint32_t *box);
// the same for 4-byte elements (the direct path's packed BF16 hi / lo words)
bool encode_tiled_u32(CUtensorMap *m, const void *ptr, int rank, const uint64_t *dims, const uint64_t *strides_bytes,
                      const uint32_t *box);
// shortest pencil of the 16-slot shape the persistent kernel is built for (shorter ones, on
// tiny grids, keep the one-shot kernel; fewer instances keep the build short)
constexpr int kMinLength = 64;

// Pencils per item: 8 for warp-specialised blocks, 16 otherwise, except that passes with a factor above 16 take
// what the option asks for (16 of them are 128-byte rows a copy, 8 leave room for longer pencils).
__host__ __device__ constexpr int pencils(bool big, bool ws, bool wide) { return ws || (big && !wide) ? 8 : 16; }
// which of these fft_tma_inst.cu compiles a launch for
__host__ __device__ constexpr bool compiled(bool big, bool ws, int W) { return ws ? W == 8 : W == 16 || (big && W == 8); }

struct Params {
    AxisArgs a;
    int axis_is_plane;   // 1: the FFT axis is the plane dimension of the tensor (z pass), 0: rows
    int nchunks, norient, nbatch;
    long items;
    int box_j, nbox, lrows;
};

// threads of an instance: W pencils by A slots (pass 2; pass 1 needs B <= A of them), in warps
__host__ __device__ constexpr int threads(int W, int A) { return (W * A + 31) / 32 * 32; }
// blocks per SM an instance is compiled for: as many as shared memory (two stages) and registers hold; one with
// a factor above 16
__host__ __device__ constexpr int min_blocks(int W, int A, int B, bool mul)
{
    if (A > fft2::kMaxFactor) return 1;
    const int smem = kStages * A * B * W * 8 * (mul ? 2 : 1) + A * B * 8 + 512, by_smem = 220 * 1024 / smem;
    // the warps of n blocks spread over four partitions of 512 registers a lane each, 80 a thread (the compiler
    // keeps to that; see above for what it costs)
    int n = by_smem < 6 ? by_smem : 6;
    while (n > 1 && (n * threads(W, A) / 32 + 3) / 4 * 80 > 512) --n;
    return n < 1 ? 1 : n;
}

__device__ __forceinline__ void decode_item(const Params &P, long it, int &chunk, int &o, int &b)
{
    chunk = (int)(it % P.nchunks);
    const long r = it / P.nchunks;
    o = (int)(r % P.norient);
    b = (int)(r / P.norient);
}

// One thread issues the tensor copies of item `it` into a stage (W pencils of the input, and of
// the factor when MUL), completing on the stage's mbarrier.
template <int MUL, int W>
__device__ __forceinline__ void issue_item(const Params &P, const void *in_map, const void *mul_map, long it,
                                           float2 *din, float2 *dmul, uint64_t *bar)
{
    int chunk, o, b;
    decode_item(P, it, chunk, o, b);
    tc::mbar_expect_tx(bar, (uint32_t)(P.nbox * P.box_j * W * sizeof(float2)) * (MUL ? 2u : 1u));
    const int c0 = chunk * W;
    for (int k = 0; k < P.nbox; ++k) {
        const int j0 = k * P.box_j;
        if (P.axis_is_plane) tc::tma_load_4d(din + (size_t)j0 * W, in_map, c0, b, j0, o, bar);
        else tc::tma_load_4d(din + (size_t)j0 * W, in_map, c0, j0, b, o, bar);
        if (MUL) {
            if (P.axis_is_plane) tc::tma_load_3d(dmul + (size_t)j0 * W, mul_map, c0, b, j0, bar);
            else tc::tma_load_3d(dmul + (size_t)j0 * W, mul_map, c0, j0, b, bar);
        }
    }
}

// where the tile between the passes lies: in the item's own stage (factors up to 16), or in a buffer of its own
__host__ __device__ constexpr bool tile_in_stage(int A) { return A <= fft2::kMaxFactor; }

// One split L = NA NB: the persistent loop over this block's items.
template <int S, int MUL, int W, int NA, int NB>
__global__ void __launch_bounds__(threads(W, NA), min_blocks(W, NA, NB, MUL != 0))
    axis2_tma_kernel(const __grid_constant__ CUtensorMap in_map, const __grid_constant__ CUtensorMap mul_map, Params P)
{
    constexpr int T = threads(W, NA), LOGW = W == 8 ? 3 : 4, L = NA * NB;
    extern __shared__ unsigned char smraw[];
    const AxisArgs &a = P.a;
    // 128-byte aligned stages (tensor-copy destinations), twiddles, barriers
    unsigned char *base = smraw + ((128 - (tc::smem_addr(smraw) & 127)) & 127);
    const size_t half = (size_t)P.lrows * W, stage = half * (MUL ? 2 : 1);
    constexpr bool INSTAGE = tile_in_stage(NA);
    float2 *st = reinterpret_cast<float2 *>(base), *own = st + kStages * stage, *tw = own + (INSTAGE ? 0 : L * W);
    uint64_t *bar = reinterpret_cast<uint64_t *>(tw + L);
    for (int i = threadIdx.x; i < L; i += T) tw[i] = a.tw[i];
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) tc::mbar_init(&bar[s], 1);
        tc::fence_mbar_init();
    }
    __syncthreads();
    const int w = threadIdx.x & (W - 1), p = threadIdx.x >> LOGW;
    const long G = gridDim.x, first = blockIdx.x;
    const long mine = (P.items - first + G - 1) / G;           // items of this block: first + k G
    if (threadIdx.x == 0)
        for (int s = 0; s < kStages && s < mine; ++s)
            issue_item<MUL, W>(P, &in_map, &mul_map, first + s * G, st + s * stage, st + s * stage + half, &bar[s]);
    for (long k = 0; k < mine; ++k) {
        const int s = (int)(k % kStages);
        const bool timeout = !tc::mbar_wait(&bar[s], (uint32_t)((k / kStages) & 1));
        const long it = first + k * G;
        float2 *in = st + s * stage, *tile = INSTAGE ? in : own;
        auto refill = [&]() {
            if (threadIdx.x == 0 && k + kStages < mine) {
                // generic-proxy accesses of the stage above, async-proxy writes into it next
                tc::fence_async_smem();
                issue_item<MUL, W>(P, &in_map, &mul_map, first + (k + kStages) * G, in, in + half, &bar[s]);
            }
        };
        // pass 1: slot p = n1 < NB reads x[n1 + NB n2] (times the factor) from the stage and transforms it
        // in registers (after a timeout the values are not used)
        float2 v[NA];
        const bool act = p < NB;
        if (act) {
#pragma unroll
            for (int n2 = 0; n2 < NA; ++n2) {
                const int j = p + NB * n2;
                v[n2] = in[j * W + w];
                if (MUL) v[n2] = c_mul(v[n2], in[half + j * W + w]);
            }
            fft2::dft_reg<S, NA>(v);
            fft2::twiddle<S, NA>(v, p, tw);
        }
        // the stage is read and the previous item's tile too; every thread knows whether a copy timed out
        if (__syncthreads_or(timeout)) {
            if (threadIdx.x == 0) {
                if (a.status) atomicCAS(a.status, 0, (int)IMF_ERR_TIMEOUT);
                // wait (bounded) for this block's copies still in flight before leaving
                const long issued = k + kStages < mine ? k + kStages : mine;
                for (long q = k; q < issued; ++q) tc::mbar_wait(&bar[q % kStages], (uint32_t)((q / kStages) & 1));
            }
            return;
        }
        if (!INSTAGE) refill();
        if (act) {
#pragma unroll
            for (int k2 = 0; k2 < NA; ++k2) tile[(p * NA + k2) * W + w] = v[k2];
        }
        __syncthreads();
        // pass 2: slot p = k2 < NA, NB-point DFT over n1; X[k2 + NA k1] -> out[j - j0] in the window
        int chunk, o, b;
        decode_item(P, it, chunk, o, b);
        const int c = chunk * W + w;
        const bool act2 = p < NA && c < a.nx;
        float2 u[NB];
        if (act2) {
#pragma unroll
            for (int n1 = 0; n1 < NB; ++n1) u[n1] = tile[(n1 * NA + p) * W + w];
        }
        if (INSTAGE) {
            __syncthreads();
            refill();
        }
        if (act2) {
            fft2::dft_reg<S, NB>(u);
            float2 *out = a.out + (long)o * a.out_so + (long)b * a.out_sb + c;
#pragma unroll
            for (int k1 = 0; k1 < NB; ++k1) {
                const int j = p + NA * k1 - a.j0;
                if (j >= 0 && j < a.lout) {
                    float2 y = c_scale(u[k1], a.scale);
                    if (a.conj_out) y.y = -y.y;
                    out[(long)j * a.out_sl] = y;
                }
            }
        }
    }
}

// ---------------------------------------------------------------------------------------------
// Warp-specialised variant: warp 0 is the producer (one lane issues the tensor copies), the
// other warps are consumers, 8 NA threads of them (pencil w = thread & 7, slot p = thread >> 3),
// so no warp idles through both DFT passes. Each stage has a "full" mbarrier (the copy's bytes)
// and an "empty" one (one arrival per consumer warp once it has read the stage), so the producer
// refills a stage as soon as it is free instead of at a block-wide barrier. Consumers meet once
// per item, at a named reduction barrier after writing the tile, which also makes them agree on a
// timed-out copy; the tile is double-buffered where shared memory allows (else a second named
// barrier guards it). Block barriers are never used after the set-up.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ bool bar_red_or(int id, int nthreads, bool v)
{
    uint32_t r;
    asm volatile("{\n.reg .pred pi, po;\nsetp.ne.u32 pi, %1, 0;\nbar.red.or.pred po, %2, %3, pi;\nselp.u32 %0, 1, 0, po;\n}\n"
                 : "=r"(r)
                 : "r"((uint32_t)v), "r"(id), "r"(nthreads)
                 : "memory");
    return r != 0;
}
__device__ __forceinline__ void bar_named(int id, int nthreads)
{
    asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(nthreads) : "memory");
}

struct WsLayout {
    int ntiles;           // 1 or 2 tile buffers
};

template <int S, int MUL, int W, int NA, int NB>
__device__ __forceinline__ void ws_items(const Params &P, const void *in_map, const void *mul_map, float2 *st,
                                         size_t half, size_t stage, float2 *tile, int ntiles, const float2 *tw,
                                         uint64_t *full, uint64_t *empty)
{
    constexpr int LOGW = W == 8 ? 3 : 4;
    const AxisArgs &a = P.a;
    const long G = gridDim.x, first = blockIdx.x;
    const long mine = (P.items - first + G - 1) / G;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ncons = (int)blockDim.x - 32;
    const size_t tsz = (size_t)NA * NB * W;
    if (warp == 0) {
        // producer: one lane issues every copy of this block, refilling a stage once its empty
        // barrier shows that every consumer warp has read it
        if (lane != 0) return;
        for (long k = 0; k < mine; ++k) {
            const int s = (int)(k % kStages);
            if (k >= kStages && !tc::mbar_wait(&empty[s], (uint32_t)((k / kStages - 1) & 1))) {
                if (a.status) atomicCAS(a.status, 0, (int)IMF_ERR_TIMEOUT);
                // the consumers time out on the stage this copy would have filled
                for (long q = k - kStages + 1; q < k; ++q)
                    if (q >= 0) tc::mbar_wait(&full[q % kStages], (uint32_t)((q / kStages) & 1));
                return;
            }
            tc::fence_async_smem();
            issue_item<MUL, W>(P, in_map, mul_map, first + k * G, st + s * stage, st + s * stage + half, &full[s]);
        }
        return;
    }
    const int ct = threadIdx.x - 32, w = ct & (W - 1), p = ct >> LOGW;
    for (long k = 0; k < mine; ++k) {
        const int s = (int)(k % kStages);
        const bool timeout = !tc::mbar_wait(&full[s], (uint32_t)((k / kStages) & 1));
        const float2 *sin_ = st + s * stage, *smul = sin_ + half;
        float2 v[NA];
        const bool act = p < NB;
        if (act) {
#pragma unroll
            for (int n2 = 0; n2 < NA; ++n2) {
                const int j = p + NB * n2;
                v[n2] = sin_[j * W + w];
                if (MUL) v[n2] = c_mul(v[n2], smul[j * W + w]);
            }
        }
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&empty[s]);
        float2 *tl = tile + (ntiles == 2 ? (size_t)(k & 1) * tsz : 0);
        if (act) {
            fft2::dft_reg<S, NA>(v);
            fft2::twiddle<S, NA>(v, p, tw);
#pragma unroll
            for (int k2 = 0; k2 < NA; ++k2) tl[(p * NA + k2) * W + w] = v[k2];
        }
        if (bar_red_or(1, ncons, timeout)) {
            if (a.status) atomicCAS(a.status, 0, (int)IMF_ERR_TIMEOUT);
            return;
        }
        int chunk, o, b;
        decode_item(P, first + k * G, chunk, o, b);
        const int c = chunk * W + w;
        if (p < NA && c < a.nx) {
            float2 u[NB];
#pragma unroll
            for (int n1 = 0; n1 < NB; ++n1) u[n1] = tl[(n1 * NA + p) * W + w];
            fft2::dft_reg<S, NB>(u);
            float2 *out = a.out + (long)o * a.out_so + (long)b * a.out_sb + c;
#pragma unroll
            for (int k1 = 0; k1 < NB; ++k1) {
                const int j = p + NA * k1 - a.j0;
                if (j >= 0 && j < a.lout) {
                    float2 y = c_scale(u[k1], a.scale);
                    if (a.conj_out) y.y = -y.y;
                    out[(long)j * a.out_sl] = y;
                }
            }
        }
        // one tile: its readers finish before the next item's pass 1 rewrites it
        if (ntiles == 1) bar_named(2, ncons);
    }
}

template <int S, bool BIG, int MUL, int W>
__global__ void __launch_bounds__(256) axis2_ws_kernel(const __grid_constant__ CUtensorMap in_map,
                                                       const __grid_constant__ CUtensorMap mul_map, Params P, int ntiles)
{
    extern __shared__ unsigned char smraw[];
    const int A = P.a.A2, B = P.a.B2, L = A * B;
    unsigned char *base = smraw + ((128 - (tc::smem_addr(smraw) & 127)) & 127);
    const size_t half = (size_t)P.lrows * W;
    const size_t stage = half * (MUL ? 2 : 1);
    float2 *st = reinterpret_cast<float2 *>(base);
    float2 *tile = st + kStages * stage;
    float2 *tw = tile + (size_t)ntiles * L * W;
    uint64_t *full = reinterpret_cast<uint64_t *>(tw + L), *empty = full + kStages;
    const int ncw = ((int)blockDim.x - 32) / 32;
    for (int i = threadIdx.x; i < L; i += blockDim.x) tw[i] = P.a.tw[i];
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            tc::mbar_init(&full[s], 1);
            tc::mbar_init(&empty[s], ncw);
        }
        tc::fence_mbar_init();
    }
    __syncthreads();
    constexpr int maxA = BIG ? fft2::kMaxFactorBig : fft2::kMaxFactor;
    auto outer = [&](auto AA) {
        constexpr int NA = decltype(AA)::value;
        auto inner = [&](auto BB) {
            constexpr int NB = decltype(BB)::value;
            if constexpr (fft2::is_split_choice(NA, NB, maxA) &&
                          (BIG ? NA > fft2::kMaxFactor : NA * NB >= kMinLength))
                ws_items<S, MUL, W, NA, NB>(P, &in_map, &mul_map, st, half, stage, tile, ntiles, tw, full, empty);
        };
        if constexpr (BIG) fft2::with_size_big(B, inner);
        else fft2::with_size(B, inner);
    };
    if constexpr (BIG) fft2::with_size_big(A, outer);
    else fft2::with_size(A, outer);
}

// threads of the warp-specialised block: the producer warp and 8 NA consumer threads in warps
inline int ws_threads(int A) { return 32 + ((8 * A + 31) / 32) * 32; }

inline size_t ws_smem_bytes(const Params &P, int W, bool mul, int ntiles)
{
    const int L = P.a.A2 * P.a.B2;
    return 128 + (size_t)kStages * P.lrows * W * 8 * (mul ? 2 : 1) + (size_t)ntiles * L * W * 8 + (size_t)L * 8 +
           2 * kStages * 8;
}

template <int S, bool BIG, int MUL, int W>
bool launch_ws(const CUtensorMap &in_map, const CUtensorMap &mul_map, Params &P, cudaStream_t s)
{
    static_assert(W == 8, "the warp-specialised pass maps 8 pencils per thread row");
    const int T = ws_threads(P.a.A2);
    if (T > 256) return false;
    auto kernel = axis2_ws_kernel<S, BIG, MUL, W>;
    // two tiles when two blocks of that size still fit an SM, else one
    int ntiles = 2;
    size_t smem = ws_smem_bytes(P, W, MUL != 0, 2);
    if (2 * (smem + 1024) > 228 * 1024) {
        ntiles = 1;
        smem = ws_smem_bytes(P, W, MUL != 0, 1);
    }
    if (smem > 227 * 1024) return false;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    int per = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, T, smem) != cudaSuccess || per < 1) {
        cudaGetLastError();
        return false;
    }
    const long blocks = P.items < (long)per * sm_count() ? P.items : (long)per * sm_count();
    kernel<<<(unsigned)blocks, T, smem, s>>>(in_map, mul_map, P, ntiles);
    return true;
}

// The six instances (16-slot shape s*, 32-slot shape b*; variant 0 = forward, 1 = inverse,
// 2 = inverse with the pointwise factor), each compiled from fft_tma_inst.cu in its own
// translation unit; false when nothing was launched.
#define IMF_TMA_DECL(name) bool name(const CUtensorMap &in_map, const CUtensorMap &mul_map, Params &P, bool ws, int W, cudaStream_t s);
IMF_TMA_DECL(launch_tma_s0)
IMF_TMA_DECL(launch_tma_s1)
IMF_TMA_DECL(launch_tma_s2)
IMF_TMA_DECL(launch_tma_b0)
IMF_TMA_DECL(launch_tma_b1)
IMF_TMA_DECL(launch_tma_b2)
#undef IMF_TMA_DECL


// Shared memory of one block: 128 bytes of alignment slack, the stages, the tile where it has a buffer of its
// own, the twiddles and the barriers.
inline size_t smem_bytes(const Params &P, int W, bool mul)
{
    const int L = P.a.A2 * P.a.B2;
    return 128 + (size_t)kStages * P.lrows * W * 8 * (mul ? 2 : 1) + (tile_in_stage(P.a.A2) ? 0 : (size_t)L * W * 8) +
           (size_t)L * 8 + kStages * 8;
}

template <int S, int MUL, int W, int NA, int NB>
bool launch_split(const CUtensorMap &in_map, const CUtensorMap &mul_map, const Params &P, cudaStream_t s)
{
    constexpr int T = threads(W, NA);
    const size_t smem = smem_bytes(P, W, MUL != 0);
    if (smem > 227 * 1024) return false;
    auto kernel = axis2_tma_kernel<S, MUL, W, NA, NB>;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    int per = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, T, smem) != cudaSuccess || per < 1) {
        cudaGetLastError();
        return false;
    }
    const long blocks = P.items < (long)per * sm_count() ? P.items : (long)per * sm_count();
    kernel<<<(unsigned)blocks, T, smem, s>>>(in_map, mul_map, P);
    return true;
}

// the instance of the split of P.a (16-slot shape: both factors at most 16, length from kMinLength)
template <int S, bool BIG, int MUL, int W>
bool launch_shape(const CUtensorMap &in_map, const CUtensorMap &mul_map, Params &P, cudaStream_t s)
{
    constexpr int maxA = BIG ? fft2::kMaxFactorBig : fft2::kMaxFactor;
    bool done = false;
    auto outer = [&](auto AA) {
        constexpr int NA = decltype(AA)::value;
        auto inner = [&](auto BB) {
            constexpr int NB = decltype(BB)::value;
            if constexpr (fft2::is_split_choice(NA, NB, maxA) &&
                          (BIG ? NA > fft2::kMaxFactor : NA * NB >= kMinLength))
                done = launch_split<S, MUL, W, NA, NB>(in_map, mul_map, P, s);
        };
        if constexpr (BIG) fft2::with_size_big(P.a.B2, inner);
        else fft2::with_size(P.a.B2, inner);
    };
    if constexpr (BIG) fft2::with_size_big(P.a.A2, outer);
    else fft2::with_size(P.a.A2, outer);
    return done;
}

} // namespace tma_fft
} // namespace imf
