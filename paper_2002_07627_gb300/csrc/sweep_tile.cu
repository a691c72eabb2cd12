// Sweep (Eq. eq_conv_A) on staged tiles: A_R(x) = OR_{k in RK} free(x - k), 32 translations per word along x.
//
// The cutter is cut into slices of equal x offset: within one the source words line up with each other, so a
// slice is an OR of whole words over runs along y or z, and only its result is shifted (one shuffle for the
// neighbouring word and a funnel shift per output word). A block stages the words its outputs read (rows along the
// run axis contiguous, an odd pitch between columns: the lanes of a warp, nl words by ppw planes, read 32 banks) and
// each thread keeps kSwX consecutive output rows, so a run of length L costs kSwX + L - 1 shared loads for kSwX
// output words: about 174 a word for a radius-3 cutter against 516 words read through L1 by the kernel on dilation
// levels, which was bound by the sectors its windows touched. Bound by the shared-memory pipe and the descriptors'
// overhead. Measured, ms a step (levels and sweep before, this kernel): 256^3 x 128 5.87 -> 3.63; 128^3 x 64 with
// per-orientation sets 0.67 -> 0.32, union alone 0.39 -> 0.28.
#include "sweep_tile.cuh"

namespace imf {

namespace {

// acc[j] |= OR of s[j .. j + L - 1]
template <int L> __device__ __forceinline__ void run_or(const uint32_t *__restrict__ s, uint32_t *acc)
{
    uint32_t w[kSwX + L - 1];
#pragma unroll
    for (int i = 0; i < kSwX + L - 1; ++i) w[i] = s[i];
    if constexpr (L <= 3) {
#pragma unroll
        for (int j = 0; j < kSwX; ++j) {
#pragma unroll
            for (int t = 0; t < L; ++t) acc[j] |= w[j + t];
        }
    } else {
        // windows of three, then of nine; the last one of a run may overlap its neighbour
        uint32_t v[kSwX + L - 3];
#pragma unroll
        for (int i = 0; i < kSwX + L - 3; ++i) v[i] = w[i] | w[i + 1] | w[i + 2];
        if constexpr (L >= 9) {
            uint32_t n[kSwX + L - 9];
#pragma unroll
            for (int i = 0; i < kSwX + L - 9; ++i) n[i] = v[i] | v[i + 3] | v[i + 6];
#pragma unroll
            for (int j = 0; j < kSwX; ++j) acc[j] |= n[j] | n[j + L - 9];
        } else {
#pragma unroll
            for (int j = 0; j < kSwX; ++j) {
                acc[j] |= v[j] | v[j + L - 3];
                if constexpr (L > 6) acc[j] |= v[j + 3];
            }
        }
    }
}

__device__ __forceinline__ void run_any(int L, const uint32_t *s, uint32_t *acc)
{
    switch (L) {
    case 1: run_or<1>(s, acc); break;
    case 2: run_or<2>(s, acc); break;
    case 3: run_or<3>(s, acc); break;
    case 4: run_or<4>(s, acc); break;
    case 5: run_or<5>(s, acc); break;
    case 6: run_or<6>(s, acc); break;
    case 7: run_or<7>(s, acc); break;
    case 8: run_or<8>(s, acc); break;
    case 9: run_or<9>(s, acc); break;
    case 10: run_or<10>(s, acc); break;
    case 11: run_or<11>(s, acc); break;
    case 12: run_or<12>(s, acc); break;
    case 13: run_or<13>(s, acc); break;
    case 14: run_or<14>(s, acc); break;
    case 15: run_or<15>(s, acc); break;
    default: run_or<16>(s, acc); break;
    }
}

__global__ void __launch_bounds__(kSwThreads) sweep_tile_kernel(const __grid_constant__ SwArgs a)
{
    extern __shared__ uint32_t sm[];
    const SwGeometry &g = a.geo;
    const int ob = blockIdx.y, og = a.orient_base + ob;
    const SwOrient h = a.head[og];
    if (h.axis < 0) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nu = h.axis ? a.nz : a.ny, nw = h.axis ? a.ny : a.nz;          // outputs along the run and plane axes
    const int tp = g.ppw * kSwNP;                                            // output planes of a tile
    const int tq = (a.awords + g.nq - 1) / g.nq, tu = (nu + kSwRows - 1) / kSwRows;
    const int t = blockIdx.x;
    if (t >= tq * tu * ((nw + tp - 1) / tp)) return;
    const int Q0 = (t % tq) * g.nq, U0 = (t / tq % tu) * kSwRows, W0 = (t / (tq * tu)) * tp;
    // this thread's outputs: word q of rows u .. u + kSwX - 1 in plane w
    const int lw = lane % g.nl, lp = lane / g.nl;
    const int pu = (warp % kSwNU) * kSwX, pw = (warp / kSwNU) * g.ppw + lp;
    const int q = Q0 + lw, u = U0 + pu, w = W0 + pw;
    const bool lane_on = lp < g.ppw;
    const bool out_on = lane_on && lw < g.nq && q < a.awords && w < nw;
    const long su = h.axis ? (long)a.ny * a.awords : a.awords, sw = h.axis ? a.awords : (long)a.ny * a.awords;
    uint32_t *dst = a.A + w * sw + u * su + q;
    const int rem = a.nx - 32 * q;
    const uint32_t full = rem < 32 ? (1u << (rem & 31)) - 1u : 0xffffffffu;
    const bool per = a.A_per != nullptr;
    // A only grows: outputs that are already full need no more work (unless this orientation's own set is wanted)
    uint32_t old[kSwX];
    bool live = false;
#pragma unroll
    for (int j = 0; j < kSwX; ++j) {
        old[j] = out_on && u + j < nu ? __ldcg(dst + j * su) : 0xffffffffu;
        live = live || (old[j] & full) != full || (per && out_on && u + j < nu);
    }
    const bool warp_live = __any_sync(0xffffffffu, out_on && live);
    if (!__syncthreads_or(warp_live)) return;
    // stage the words: column (plane, word) of rows, the rows contiguous; zero outside the window
    const int rows = kSwRows + h.eu, planes = tp + h.ew;
    {
        const long ru = h.axis ? (long)a.wy * a.wpr : a.wpr, rw = h.axis ? a.wpr : (long)a.wy * a.wpr;
        const int lu = h.axis ? a.wz : a.wy, lwn = h.axis ? a.wy : a.wz;
        const uint32_t *src = a.bits + ob * a.b_so + Q0;
        // (plane p, row r, word c) of this thread's next word, advanced by kSwThreads words a step
        const int dr = kSwThreads / g.nl, dc = kSwThreads - dr * g.nl;
        int p = 0, r = threadIdx.x / g.nl, c = threadIdx.x - r * g.nl;
        while (true) {
            while (r >= rows) { r -= rows; ++p; }
            if (p >= planes) break;
            const int gu = U0 + h.ou + r, gw = W0 + h.ow + p;
            uint32_t v = 0;
            if (gu < lu && gw < lwn && Q0 + c < a.wpr) v = __ldg(src + gw * rw + gu * ru + c);
            sm[(p * g.nl + c) * g.UP + r] = v;
            r += dr;
            c += dc;
            if (c >= g.nl) { c -= g.nl; ++r; }
        }
    }
    int *d = reinterpret_cast<int *>(sm + (size_t)g.planes * g.nl * g.UP);
    for (int i = threadIdx.x; i < h.words; i += kSwThreads) d[i] = __ldg(a.words + h.word0 + i);
    __syncthreads();
    if (!warp_live) return;
    const uint32_t *own = sm + ((lane_on ? pw : 0) * g.nl + (lane_on ? lw : 0)) * g.UP + pu;
    uint32_t res[kSwX];
#pragma unroll
    for (int j = 0; j < kSwX; ++j) res[j] = 0;
    int so = g.somax;
    for (int i = 0; i < h.words;) {
        const int s = d[i++], n = s >> 16;
        // results so far stand one word further left for every whole word the shift falls
        for (; so > (s & 255); --so) {
#pragma unroll
            for (int j = 0; j < kSwX; ++j) res[j] = __shfl_down_sync(0xffffffffu, res[j], 1);
        }
        uint32_t acc[kSwX];
#pragma unroll
        for (int j = 0; j < kSwX; ++j) acc[j] = 0;
        for (const int e = i + n; i < e; ++i) run_any(d[i] >> 24, own + (d[i] & 0xffffff), acc);
        const int sh = (s >> 8) & 31;
#pragma unroll
        for (int j = 0; j < kSwX; ++j)
            res[j] |= __funnelshift_r(acc[j], __shfl_down_sync(0xffffffffu, acc[j], 1), sh);
    }
    for (; so > 0; --so) {
#pragma unroll
        for (int j = 0; j < kSwX; ++j) res[j] = __shfl_down_sync(0xffffffffu, res[j], 1);
    }
    if (!out_on) return;
#pragma unroll
    for (int j = 0; j < kSwX; ++j) {
        if (u + j >= nu) continue;
        const uint32_t v = res[j] & full;
        const uint32_t add = v & ~old[j];
        if (add) atomicOr(dst + j * su, add);
        if (per) a.A_per[(long)a.perm[og] * a.a_per_so + w * sw + (u + j) * su + q] = v;
    }
}

} // namespace

void launch_sweep_tile(const SwArgs &a, cudaStream_t s)
{
    const SwGeometry &g = a.geo;
    const int tp = g.ppw * kSwNP, tq = (a.awords + g.nq - 1) / g.nq;
    auto up = [](int n, int d) { return (n + d - 1) / d; };
    const int t0 = tq * up(a.ny, kSwRows) * up(a.nz, tp), t1 = tq * up(a.nz, kSwRows) * up(a.ny, tp);
    cudaFuncSetAttribute(sweep_tile_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)g.smem);
    sweep_tile_kernel<<<dim3((unsigned)(t0 > t1 ? t0 : t1), a.nb), kSwThreads, g.smem, s>>>(a);
}

} // namespace imf
