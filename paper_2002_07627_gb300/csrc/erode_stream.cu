// Minimum over sharp points (Eq. eq_imf_2; Alg. 1 "Translate" + "min" over Support(K)), streamed:
//
//   gamma_R(x) = min_{k in sharp_R} g_R(x - k),   f(x) <- min(f(x), gamma_R(x))
//
// the same minima as erode.cu and so the same bits. What bounds it is the shared-memory load pipe (one
// load per output and run and L - 1 more per run and thread) and, beside it, the three-input minima; the
// tiled kernel keeps both at about 60 % because a block waits for each tile before it reduces and warps
// whose outputs are all final idle through the rest. So:
//   - the sharp points of an orientation are runs along y or z, whichever direction needs fewer loads
//     (116 runs against 129 along x for a radius-3 cutter): the lanes of a warp then span x, so the g
//     planes keep their layout and arrive as 16-byte asynchronous copies (four-byte ones before);
//   - four producer warps copy the planes into a ring of stages of four planes, ahead of the reducing
//     warps and across orientations (mbarriers, no block barrier between orientations);
//   - a warp does not own outputs: the running minimum lives in shared memory, and the live units
//     (8 x 8 x 4 outputs, some above 0) of each list of runs go round the 24 warps, so that all of them
//     reduce whatever part of a tile is final (about half of the units of a beam design).
// A unit: lane = x + 8 * plane, eight consecutive outputs along the run axis per thread; plane pitch
// = 8 mod 32 floats, so that 8 columns x 4 planes read 32 banks. List m of an orientation holds the runs
// that read planes 4 m .. 4 m + 3 from the output's own first one: lane plane p reads 4 m + p .. 4 m + p + 3,
// the two stages held while the list runs. The descriptors of an orientation travel with its first stage.
// Tile 32 x 24 x 8 outputs: 17.1 ms a launch at 256^3 x 64 against 17.6 for 32 x 32 x 8, 17.9 for 32 x 16 x 12
// and 18.6 for 32 x 16 x 8. Copies by tensor maps need 128-byte rows of planes and so lanes along x alone
// (32 x 8 x 1 boxes, of which 67 % hold a live output against 53 % of 8 x 8 x 4): 27.9.
// Against the tiled kernel (ms per step): 256^3 x 128 43.5 -> 34.1, 128^3 x 64 2.98 -> 2.47, 144^3 x 96 with a
// radius-6 cutter 17.2 -> 13.5.
//
// Every wait on a stage is bounded; on a timeout the block records IMF_ERR_TIMEOUT and leaves, its producers
// together (es_produce) and after the copies they issued have landed. The two named barriers need no limit:
// all that they count reach them, since every wait before them ends.
#include "erode_stream.cuh"
#include "imf.h"
#include "imf_internal.cuh"
#include "tc_primitives.cuh"

namespace imf {

namespace {

__device__ __forceinline__ float fmin3(float a, float b, float c)
{
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

template <int L> __host__ __device__ constexpr int nblk() { return L <= 3 ? L : (L + 2) / 3; }
template <int L> __host__ __device__ constexpr int blk(int m) { return L <= 3 ? m : (m + 1 < nblk<L>() ? 3 * m : L - 3); }
template <int X, int L> __host__ __device__ constexpr int nv() { return L <= 3 ? X + L - 1 : X + L - 3; }

template <int X, int L, int P> __device__ __forceinline__ void run_blocks(const float *__restrict__ s, float *V)
{
    float w[X + L - 1];
#pragma unroll
    for (int i = 0; i < X + L - 1; ++i) w[i] = s[i * P];
    if constexpr (L <= 3) {
#pragma unroll
        for (int i = 0; i < X + L - 1; ++i) V[i] = w[i];
    } else {
#pragma unroll
        for (int i = 0; i < X + L - 3; ++i) V[i] = fmin3(w[i], w[i + 1], w[i + 2]);
    }
}

template <int X, int L, int P> __device__ __forceinline__ void run_min(const float *__restrict__ s, float *acc)
{
    float V[nv<X, L>()];
    run_blocks<X, L, P>(s, V);
    if constexpr (L >= 12) {
        // windows of nine from three blocks each; two of them cover the run
        float N[X + L - 9];
#pragma unroll
        for (int i = 0; i < X + L - 9; ++i) N[i] = fmin3(V[i], V[i + 3], V[i + 6]);
#pragma unroll
        for (int j = 0; j < X; ++j) acc[j] = fmin3(acc[j], N[j], N[j + L - 9]);
    } else {
        constexpr int K = nblk<L>();
#pragma unroll
        for (int j = 0; j < X; ++j) {
            float m = acc[j];
#pragma unroll
            for (int b = 0; b < K; b += 2) {
                if (b + 1 < K) m = fmin3(m, V[j + blk<L>(b)], V[j + blk<L>(b + 1)]);
                else m = fminf(m, V[j + blk<L>(b)]);
            }
            acc[j] = m;
        }
    }
}

template <int X, int L, int P>
__device__ __forceinline__ void run_pair(const float *__restrict__ s0, const float *__restrict__ s1, float *acc)
{
    float V0[nv<X, L>()], V1[nv<X, L>()];
    run_blocks<X, L, P>(s0, V0);
    run_blocks<X, L, P>(s1, V1);
    constexpr int K = nblk<L>();
#pragma unroll
    for (int j = 0; j < X; ++j) {
        float m = acc[j];
#pragma unroll
        for (int b = 0; b < 2 * K; b += 2) {
            const float u = b < K ? V0[j + blk<L>(b)] : V1[j + blk<L>(b - K)];
            const float v = b + 1 < K ? V0[j + blk<L>(b + 1)] : V1[j + blk<L>(b + 1 - K)];
            m = fmin3(m, u, v);
        }
        acc[j] = m;
    }
}

// A source window starts at `tb` + offset, or one ring length before when that runs past the ring.
struct Ring {
    const unsigned char *base;
    uint32_t tb, len;
    __device__ __forceinline__ const float *at(int off) const
    {
        uint32_t p = tb + (uint32_t)off;
        p = min(p, p - len);                 // p - len is huge for p < len
        return reinterpret_cast<const float *>(base + p);
    }
};

// the `n` runs of one length in a list: offsets from `d` on, which moves past them
template <int X, int L, int P> __device__ __forceinline__ void run_group(int n, const int *&d, const Ring &ring, float *acc)
{
    if constexpr (L == 1) {
        for (; n > 3; n -= 4, d += 4) {
            const int4 o = *reinterpret_cast<const int4 *>(d);
            run_pair<X, 1, P>(ring.at(o.x), ring.at(o.y), acc);
            run_pair<X, 1, P>(ring.at(o.z), ring.at(o.w), acc);
        }
        for (; n > 0; --n) run_min<X, 1, P>(ring.at(*d++), acc);
    } else if constexpr (es_unroll(L) == 2) {
        if (!n) return;
        d = reinterpret_cast<const int *>((reinterpret_cast<uintptr_t>(d) + 7) & ~uintptr_t(7));
        for (; n > 1; n -= 2, d += 2) {
            const int2 o = *reinterpret_cast<const int2 *>(d);
            if constexpr (nblk<L>() & 1) {
                run_pair<X, L, P>(ring.at(o.x), ring.at(o.y), acc);
            } else {
                run_min<X, L, P>(ring.at(o.x), acc);
                run_min<X, L, P>(ring.at(o.y), acc);
            }
        }
        if (n) run_min<X, L, P>(ring.at(*d++), acc);
    } else {
        for (; n > 0; --n) run_min<X, L, P>(ring.at(*d++), acc);
    }
}

// one list (a 16-byte table of runs per length, then the offsets) for the thread's outputs
template <int X, int P> __device__ __forceinline__ void run_list(const int *d, const Ring &ring, float *acc)
{
    const uint4 n = *reinterpret_cast<const uint4 *>(d);
    d += 4;
    auto runs = [](uint32_t w, int i) { return (int)((w >> (8 * i)) & 255u); };
    if (n.x) {
        run_group<X, 1, P>(runs(n.x, 0), d, ring, acc);
        run_group<X, 2, P>(runs(n.x, 1), d, ring, acc);
        run_group<X, 3, P>(runs(n.x, 2), d, ring, acc);
        run_group<X, 4, P>(runs(n.x, 3), d, ring, acc);
    }
    if (n.y) {
        run_group<X, 5, P>(runs(n.y, 0), d, ring, acc);
        run_group<X, 6, P>(runs(n.y, 1), d, ring, acc);
        run_group<X, 7, P>(runs(n.y, 2), d, ring, acc);
        run_group<X, 8, P>(runs(n.y, 3), d, ring, acc);
    }
    if (n.z) {
        run_group<X, 9, P>(runs(n.z, 0), d, ring, acc);
        run_group<X, 10, P>(runs(n.z, 1), d, ring, acc);
        run_group<X, 11, P>(runs(n.z, 2), d, ring, acc);
        run_group<X, 12, P>(runs(n.z, 3), d, ring, acc);
    }
    if (n.w) {
        run_group<X, 13, P>(runs(n.w, 0), d, ring, acc);
        run_group<X, 14, P>(runs(n.w, 1), d, ring, acc);
        run_group<X, 15, P>(runs(n.w, 2), d, ring, acc);
        run_group<X, 16, P>(runs(n.w, 3), d, ring, acc);
    }
}

// the copies of this thread issued so far arrive on `bar` when they land
__device__ __forceinline__ void copies_arrive(uint64_t *bar)
{
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];\n" ::"r"(tc::smem_addr(bar)) : "memory");
}

// whether `p` holds in any of the producers; a barrier of all of them
__device__ __forceinline__ bool any_producer(bool p)
{
    uint32_t r;
    asm volatile("{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbarrier.cta.red.or.pred q, 1, %2, p;\nselp.u32 %0, 1, 0, q;\n}\n"
                 : "=r"(r)
                 : "r"((uint32_t)p), "n"(kEsProducers)
                 : "memory");
    return r != 0;
}

// A producer thread: copies the planes of every orientation of its block's kind into the ring (es_produce).
template <int P> struct EsProducer {
    const EsArgs &a;
    const unsigned short *s_ob;
    int *s_words;
    unsigned char *s_live, (*s_list)[32], (*s_off)[kEsNW + 1];
    uint64_t *full, *empty;
    int *s_stop;
    uint32_t ring0, stage_bytes;
    int X0, U0, W0, nu, nw;                // tile origin, window extents along the run and the plane axis
    long su, sw;                           // strides of g along these
    // the orientation it is at: columns, rows and first place of what it copies, its first plane, its descriptors
    int cols, rows, gw0, words, word0;
    const float *src0;

    __device__ __forceinline__ int steps(int k)
    {
        const int ob = s_ob[k];
        const EsOrient h = a.head[a.orient_base + ob];
        const int gu0 = U0 + h.ou, row0 = (threadIdx.x & 31) >> 4;
        cols = min(h.quads, (a.gpx - (X0 + h.ox)) >> 2);       // columns the window's rows have from here
        rows = min(h.rows, nu - gu0);
        gw0 = W0 + h.ow;
        words = h.words;
        word0 = h.word0;
        src0 = a.g + ob * a.g_so + X0 + h.ox + (gu0 + row0) * su;
        return kEsNW + h.lists;
    }
    __device__ __forceinline__ bool wait(int st, uint32_t phase)
    {
        if (tc::mbar_wait(&empty[st], phase)) return true;
        if (a.status) atomicCAS(a.status, 0, (int)IMF_ERR_TIMEOUT);
        return false;
    }
    __device__ __forceinline__ EsOpen open(int k, int st, bool late)
    {
        const int tid = threadIdx.x - 32 * kEsWarps, lane = tid & 31, slot = k % kEsSlots;
        // the orientation's descriptors; the slot's last readers, four orientations back, gave
        // back their stages at least ten stages ago (an orientation has three or more)
        if (!late)
            for (int i = tid; i < words / 4; i += kEsProducers)
                reinterpret_cast<int4 *>(s_words + slot * a.geo.words)[i] = __ldg(reinterpret_cast<const int4 *>(a.words + word0) + i);
        // the units that still have work, as one warp sees them; none: the block is done
        if (tid < 32) {
            const uint32_t mask = __ballot_sync(0xffffffffu, ((volatile unsigned char *)s_live)[lane] != 0);
            if (!late) {
                if (mask >> lane & 1) s_list[slot][__popc(mask & ((1u << lane) - 1))] = (unsigned char)lane;
                constexpr int per_group = kEsUnits / kEsNW;
                if (lane <= kEsNW)                             // where each plane group's units start
                    s_off[slot][lane] = (unsigned char)__popcll(mask & ((1ull << (lane * per_group)) - 1));
                if (lane == 0 && !mask) *(volatile int *)s_stop = k;
            }
        }
        if (any_producer(late)) return EsOpen::leave;
        if (*(volatile int *)s_stop != k) return EsOpen::copy;
        tc::mbar_arrive(&full[st]);
        if (tid == 0) tc::mbar_arrive(&full[st]);
        return EsOpen::done;
    }
    __device__ __forceinline__ void copy(int k, int s, int st)
    {
        // a producer warp copies whole planes: 16 lanes a row, two rows a step
        const int tid = threadIdx.x - 32 * kEsWarps, lane = tid & 31, ch = lane & 15, row0 = lane >> 4;
        for (int pl = tid >> 5; pl < 4 && gw0 + 4 * s + pl < nw; pl += kEsProducers / 32)
            for (int c = ch; c < cols; c += 16) {
                const float *src = src0 + (gw0 + 4 * s + pl) * sw + 4 * c;
                uint32_t dst = ring0 + st * stage_bytes + 4u * (uint32_t)(pl * a.geo.Q + row0 * P + 4 * c);
#pragma unroll 4
                for (int row = row0; row < rows; row += 2) {
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
                    src += 2 * su;
                    dst += 8 * P;
                }
            }
        copies_arrive(&full[st]);
        if (tid == 0) tc::mbar_arrive(&full[st]);              // publishes the list
    }
};

template <int P> __global__ void __launch_bounds__(kEsThreads, 1) erode_stream_kernel(EsArgs a, EsTiles t)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ int s_stop;
    __shared__ unsigned short s_ob[kEsShare];
    __shared__ unsigned char s_live[32], s_list[kEsSlots][32], s_off[kEsSlots][kEsNW + 1];
    __shared__ uint64_t full[kEsMaxStages], empty[kEsMaxStages];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int Q = a.geo.Q, NS = a.geo.stages;
    const uint32_t ring0 = tc::smem_addr(smraw), stage_bytes = 16u * (uint32_t)Q;
    float *s_acc = reinterpret_cast<float *>(smraw + NS * stage_bytes);
    int *s_words = reinterpret_cast<int *>(s_acc + kEsUnits * kEsX * 32);
    const int per = t.kind(0) + t.kind(1);
    const int grp = blockIdx.x / per;
    int r = blockIdx.x - grp * per;
    const int axis = r >= t.kind(0);
    if (axis) r -= t.kind(0);
    const int X0 = (r % t.x) * kEsTX, U0 = ((r / t.x) % t.u[axis]) * kEsRows, W0 = (r / (t.x * t.u[axis])) * kEsW;
    const int k0 = (int)((long)grp * a.kind[axis] / a.ngroups), k1 = (int)((long)(grp + 1) * a.kind[axis] / a.ngroups);
    if (k0 == k1) return;
    if (threadIdx.x == 0) {
        for (int s = 0; s < NS; ++s) {
            tc::mbar_init(&full[s], kEsProducers + 1);
            tc::mbar_init(&empty[s], kEsWarps);
        }
        tc::fence_mbar_init();
        s_stop = 1 << 30;
    }
    // the running minimum of the block's outputs, from f; outputs outside the grid are final (0)
    const int onu = axis ? a.nz : a.ny, onw = axis ? a.ny : a.nz;
    const long osu = axis ? (long)a.nx * a.ny : a.nx, osw = axis ? a.nx : (long)a.nx * a.ny;
    auto place = [&](int i, bool &ok) -> float * {
        const int l = i & 31, j = (i >> 5) & (kEsX - 1), unit = i / (32 * kEsX);
        const int x = X0 + 8 * (unit & 3) + (l & 7), u = U0 + kEsX * ((unit >> 2) % kEsNU) + j,
                  w = W0 + 4 * ((unit >> 2) / kEsNU) + (l >> 3);
        ok = x < a.nx && u < onu && w < onw;
        return a.f + w * osw + u * osu + x;
    };
    if (warp == 0) {
        s_live[lane] = 0;
        // this block's orientations: number k0 .. k1 - 1 of its kind in the launch
        for (int b = 0, k = 0; b < a.nb && k < k1; b += 32) {
            const bool is = b + lane < a.nb && __ldg(&a.head[a.orient_base + b + lane].axis) == axis;
            const uint32_t m = __ballot_sync(0xffffffffu, is);
            const int mine = k + __popc(m & ((1u << lane) - 1));
            if (is && mine >= k0 && mine < k1) s_ob[mine - k0] = (unsigned short)(b + lane);
            k += __popc(m);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kEsUnits * kEsX * 32; i += kEsThreads) {
        bool ok;
        const float *p = place(i, ok);
        const float v = ok ? __ldcg(p) : 0.f;
        s_acc[i] = v;
        if (v > 0.f) s_live[i / (32 * kEsX)] = 1;
    }
    __syncthreads();
    if (warp >= kEsWarps) {
        const long row = a.gpx, plane = (long)a.gpx * a.wy;
        EsProducer<P> io{a, s_ob, s_words, s_live, s_list, s_off, full, empty, &s_stop, ring0, stage_bytes, X0, U0, W0,
                         axis ? a.wz : a.wy, axis ? a.wy : a.wz, axis ? plane : row, axis ? row : plane};
        es_produce(io, k1 - k0, NS);
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        return;
    }
    // consumers: the tasks (unit, list) of a stage go round the warps
    Ring ring;
    ring.base = smraw;
    ring.len = NS * stage_bytes;
    const uint32_t own = 4u * (uint32_t)((lane >> 3) * Q + (lane & 7));
    int st = 0;
    uint32_t ph = 0;
    int turn = warp;                                           // tasks until this warp's next one
    bool ok = true;
    for (int k = 0; k < k1 - k0 && ok; ++k) {
        const int lists = __ldg(&a.head[a.orient_base + s_ob[k]].lists);
        const int slot = k % kEsSlots;
        const int *words = s_words + slot * a.geo.words;
        for (int s = 0; s < kEsNW + lists; ++s) {
            if (!tc::mbar_wait(&full[st], ph)) {
                if (lane == 0 && a.status) atomicCAS(a.status, 0, (int)IMF_ERR_TIMEOUT);
                ok = false;
                break;
            }
            if (s == 0 && *(volatile int *)&s_stop <= k) { ok = false; break; }
            const int prev = st ? st - 1 : NS - 1;
            // plane group k is at list s - 1 - k
            const int j0 = s_off[slot][max(0, s - lists)], j1 = s_off[slot][min(kEsNW, s)];
            for (; turn < j1 - j0; turn += kEsWarps) {
                const int unit = s_list[slot][j0 + turn];
                const int m = s - 1 - unit / (kEsUnits / kEsNW);
                ring.tb = own + prev * stage_bytes + 4u * (uint32_t)(((unit >> 2) % kEsNU) * kEsX * P + 8 * (unit & 3));
                float *sa = s_acc + unit * (32 * kEsX) + lane;
                float acc[kEsX];
#pragma unroll
                for (int j = 0; j < kEsX; ++j) acc[j] = sa[32 * j];
                run_list<kEsX, P>(words + words[m], ring, acc);
                bool live = false;
#pragma unroll
                for (int j = 0; j < kEsX; ++j) {
                    // another warp may hold an earlier list of the unit: merge (g >= 0, -0 becomes +0,
                    // so the bit patterns order as the values do)
                    const float v = __fadd_rn(acc[j], 0.f);
                    if (v < sa[32 * j]) atomicMin(reinterpret_cast<unsigned int *>(sa + 32 * j), __float_as_uint(v));
                    live = live || v > 0.f;
                }
                if (!__any_sync(0xffffffffu, live) && lane == 0) s_live[unit] = 0;
            }
            turn -= j1 - j0;
            __syncwarp();
            if (lane == 0) {
                if (s > 0) tc::mbar_arrive(&empty[prev]);
                if (s == kEsNW + lists - 1) tc::mbar_arrive(&empty[st]);
            }
            if (++st == NS) { st = 0; ph ^= 1; }
        }
    }
    asm volatile("bar.sync 2, %0;\n" ::"n"(32 * kEsWarps) : "memory");
    for (int i = threadIdx.x; i < kEsUnits * kEsX * 32; i += 32 * kEsWarps) {
        bool in;
        float *p = place(i, in);
        if (in && s_acc[i] < __ldcg(p)) atomicMin(reinterpret_cast<unsigned int *>(p), __float_as_uint(s_acc[i]));
    }
}

template <int P> bool launch_p(const EsArgs &a, const EsTiles &t, long blocks, cudaStream_t s)
{
    const size_t smem = (size_t)a.geo.stages * 16 * a.geo.Q + kEsAccBytes + (size_t)kEsSlots * a.geo.words * 4;
    if (cudaFuncSetAttribute(erode_stream_kernel<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    erode_stream_kernel<P><<<(unsigned)blocks, kEsThreads, smem, s>>>(a, t);
    return true;
}

} // namespace

bool launch_erode_stream(const EsArgs &a, cudaStream_t s)
{
    const EsTiles t = es_tile_counts(a.nx, a.ny, a.nz);
    const long blocks = (long)a.ngroups * (t.kind(0) + t.kind(1));
    if (blocks < 1 || blocks > 0x7fffffffL || (a.kind[0] + a.ngroups - 1) / a.ngroups > kEsShare ||
        (a.kind[1] + a.ngroups - 1) / a.ngroups > kEsShare || a.nb > 0xffff)
        return false;
    switch (a.geo.P) {
    case 44: return launch_p<44>(a, t, blocks, s);
    case 48: return launch_p<48>(a, t, blocks, s);
    case 52: return launch_p<52>(a, t, blocks, s);
    case 56: return launch_p<56>(a, t, blocks, s);
    case 60: return launch_p<60>(a, t, blocks, s);
    case 64: return launch_p<64>(a, t, blocks, s);
    case 76: return launch_p<76>(a, t, blocks, s);
    default: return false;
    }
}

} // namespace imf
