// Conjugate gradient with a multigrid preconditioner (geometric V-cycle, Galerkin coarse operators; as
// Amir, Aage and Lazarov, "On multigrid-CG for efficient topology optimization", 2014, use it) for the FEA
// of Alg. 2, and the optimality-criteria update with its multiplier, each as one cooperative kernel.
//
// What bound the plain Jacobi-preconditioned iteration (kept in topopt2d.cu for what this one does not
// solve): thousands of iterations, each three launches and a few microseconds of FP64 (this part runs
// two FP64 multiply-adds per SM and clock), with a host round trip every sixteen. On the 256 x 128 cantilever
// midway in its loop that was 5500 iterations of 24.8 us, 136.8 ms; here 92 of about 55 us, 5.3 ms with the
// set-up, bound by the grid barriers (eight an iteration) and the latency of the short phases between them.
// The update's bisection took 36 host round trips, 1.0 ms; in one launch 0.17 ms, and with Newton steps instead
// 0.10 ms with the copies, bound by the FP64 exponentials of the projected density and the grid barriers.
//
// The iteration itself (operator, vectors, scalar products, stopping rule) is FP64 as before; only the
// preconditioner, which steers the search directions and not what they converge to, works in FP32: at
// 1/64 of the FP32 rate an FP64 V-cycle would cost more than the rest of the iteration. The FP64 operator
// is assembled once per analysis (36 multiply-adds a node against 72 element by element). Per iteration
// and level above kMgSmall nodes there is one phase down (smoothed residual, restricted) and one up (correction
// and smoothing), each on tiles with a halo staged in shared memory, separated by grid barriers; the update
// of x and r rides on the finest phase down; the levels below run inside block 0 on shared memory, with a
// second smoothing sweep (free of grid barriers: 92 iterations instead of 117 on that cantilever).
//
// Every grid barrier is bounded; when one gives up the error word is set and every block leaves.
#include <algorithm>
#include <cmath>

#include "grid_barrier.cuh"
#include "topopt2d_mg.cuh"

namespace imf_to {

namespace {

using imf::GridBarrier;

constexpr int T = kMgThreads;
constexpr int kHalo = 464;               // nodes of a staged tile with its halo
constexpr int kSweeps = 2;               // smoothing sweeps either way on the levels inside block 0
constexpr int kSmallSum = 2304;          // nodes of all levels inside block 0

__device__ __forceinline__ double block_sum(double v, double *red)
{
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x < T / 32) {
        t = red[threadIdx.x];
        for (int off = T / 64; off > 0; off >>= 1) t += __shfl_xor_sync((1u << (T / 32)) - 1, t, off);
    }
    __syncthreads();
    return t;   // valid in thread 0
}

// a value thread 0 computes for the block: FP64 divisions and roots in every thread would each cost the
// block as much as an operator application
template <typename F> __device__ __forceinline__ double scalar(F &&f, double *slot)
{
    if (threadIdx.x == 0) *slot = f();
    __syncthreads();
    const double v = *slot;
    __syncthreads();
    return v;
}

// ------------------------------------------------------------------------------------- set-up
// stencil of the finest level from the element matrix and the moduli
__global__ void mg_stencil_kernel(MgLevel l, const double *k0, const double *E, const uint8_t *fixed, double *S64, float omega)
{
    const int nx1 = l.nx + 1;
    for (int n = blockIdx.x * blockDim.x + threadIdx.x; n < l.nn; n += gridDim.x * blockDim.x) {
        const int i = n % nx1, j = n / nx1;
        double s[36];
#pragma unroll
        for (int k = 0; k < 36; ++k) s[k] = 0.0;
        // the node is corner 2 of element (i-1, j-1), 3 of (i, j-1), 1 of (i-1, j), 0 of (i, j)
        const int cx[4] = {0, 1, 1, 0}, cy[4] = {0, 0, 1, 1}, own[4] = {2, 3, 1, 0};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int ex = i - cx[own[e]], ey = j - cy[own[e]];
            if (ex < 0 || ey < 0 || ex >= l.nx || ey >= l.ny) continue;
            const double Ee = E[(long)ey * l.nx + ex];
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int di = cx[b] - cx[own[e]], dj = cy[b] - cy[own[e]], k = ((dj + 1) * 3 + di + 1) * 4;
#pragma unroll
                for (int c = 0; c < 4; ++c) s[k + c] += Ee * k0[(2 * own[e] + (c >> 1)) * 8 + 2 * b + (c & 1)];
            }
        }
        const bool f0 = fixed[2 * n], f1 = fixed[2 * n + 1];
        l.fixed[2 * n] = f0;
        l.fixed[2 * n + 1] = f1;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const int ni = i + k % 3 - 1, nj = j + k / 3 - 1;
            const bool in = ni >= 0 && nj >= 0 && ni <= l.nx && nj <= l.ny;
            const int m = nj * nx1 + ni;
            const bool g0 = !in || fixed[2 * m], g1 = !in || fixed[2 * m + 1];
            const bool out[4] = {f0 || g0, f0 || g1, f1 || g0, f1 || g1};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const double v = out[c] ? 0.0 : s[4 * k + c];
                S64[(long)(4 * k + c) * l.nn + n] = v;
                l.S[(long)(4 * k + c) * l.nn + n] = (float)v;
            }
        }
        l.dinv[2 * n] = f0 || !(s[16] > 0.0) ? 0.f : (float)(omega / s[16]);
        l.dinv[2 * n + 1] = f1 || !(s[19] > 0.0) ? 0.f : (float)(omega / s[19]);
    }
}

// whether a coarse dof is clamped: the fine dof it coincides with is
__device__ __forceinline__ bool coarse_fixed(const MgLevel &f, int I, int J, int d)
{
    return 2 * I <= f.nx && 2 * J <= f.ny && f.fixed[2 * ((long)(2 * J) * (f.nx + 1) + 2 * I) + d];
}

// Galerkin operator P^T A P with bilinear interpolation: one thread per coarse node
__global__ void mg_rap_kernel(MgLevel f, MgLevel c, float omega)
{
    const int nx1 = c.nx + 1;
    for (int n = blockIdx.x * blockDim.x + threadIdx.x; n < c.nn; n += gridDim.x * blockDim.x) {
        const int I = n % nx1, J = n / nx1;
        float s[36];
#pragma unroll
        for (int k = 0; k < 36; ++k) s[k] = 0.f;
#pragma unroll
        for (int b = -1; b <= 1; ++b)
#pragma unroll
            for (int a = -1; a <= 1; ++a) {
                const int fi = 2 * I + a, fj = 2 * J + b;
                if (fi < 0 || fj < 0 || fi > f.nx || fj > f.ny) continue;
                const float wi = (a ? 0.5f : 1.f) * (b ? 0.5f : 1.f);
                const long m = (long)fj * (f.nx + 1) + fi;
#pragma unroll
                for (int k = 0; k < 9; ++k) {
                    // offset of the fine neighbour from the coarse node, and the coarse nodes it interpolates from
                    const int tx = a + k % 3 - 1, ty = b + k / 3 - 1;
                    float v[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) v[q] = wi * f.S[(long)(4 * k + q) * f.nn + m];
#pragma unroll
                    for (int dJ = -1; dJ <= 1; ++dJ)
#pragma unroll
                        for (int dI = -1; dI <= 1; ++dI) {
                            const int ox = tx - 2 * dI, oy = ty - 2 * dJ;
                            if (ox < -1 || ox > 1 || oy < -1 || oy > 1) continue;
                            const float w = (ox ? 0.5f : 1.f) * (oy ? 0.5f : 1.f);
#pragma unroll
                            for (int q = 0; q < 4; ++q) s[((dJ + 1) * 3 + dI + 1) * 4 + q] += w * v[q];
                        }
                }
            }
        const bool f0 = coarse_fixed(f, I, J, 0), f1 = coarse_fixed(f, I, J, 1);
        c.fixed[2 * n] = f0;
        c.fixed[2 * n + 1] = f1;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const int ni = I + k % 3 - 1, nj = J + k / 3 - 1;
            const bool in = ni >= 0 && nj >= 0 && ni <= c.nx && nj <= c.ny;
            const bool g0 = !in || coarse_fixed(f, ni, nj, 0), g1 = !in || coarse_fixed(f, ni, nj, 1);
            c.S[(long)(4 * k + 0) * c.nn + n] = f0 || g0 ? 0.f : s[4 * k];
            c.S[(long)(4 * k + 1) * c.nn + n] = f0 || g1 ? 0.f : s[4 * k + 1];
            c.S[(long)(4 * k + 2) * c.nn + n] = f1 || g0 ? 0.f : s[4 * k + 2];
            c.S[(long)(4 * k + 3) * c.nn + n] = f1 || g1 ? 0.f : s[4 * k + 3];
        }
        c.dinv[2 * n] = f0 || !(s[16] > 0.f) ? 0.f : omega / s[16];
        c.dinv[2 * n + 1] = f1 || !(s[19] > 0.f) ? 0.f : omega / s[19];
    }
}

// inverse of the coarsest operator by Gauss-Jordan (it is symmetric positive definite on the free dofs;
// dofs without stiffness get a unit diagonal and a zero row and column in the inverse); one block
__global__ void __launch_bounds__(256) mg_inverse_kernel(MgLevel l, float *inv)
{
    constexpr int N = 2 * kMgCoarse;
    __shared__ float A[N][N + 1], B[N][N + 1];
    const int n = 2 * l.nn, nx1 = l.nx + 1;
    for (int t = threadIdx.x; t < n * n; t += 256) {
        const int r = t / n, c = t % n;
        const int di = (c >> 1) % nx1 - (r >> 1) % nx1, dj = (c >> 1) / nx1 - (r >> 1) / nx1;
        float v = 0.f;
        if (di >= -1 && di <= 1 && dj >= -1 && dj <= 1)
            v = l.S[(long)(((dj + 1) * 3 + di + 1) * 4 + 2 * (r & 1) + (c & 1)) * l.nn + (r >> 1)];
        A[r][c] = r == c && !(v > 0.f) ? 1.f : v;
        B[r][c] = r == c ? 1.f : 0.f;
    }
    __syncthreads();
    for (int k = 0; k < n; ++k) {
        const float piv = 1.f / A[k][k];
        __syncthreads();
        for (int c = threadIdx.x; c < n; c += 256) {
            A[k][c] *= piv;
            B[k][c] *= piv;
        }
        __syncthreads();
        // every row but k: the column k of A is read by all of a row before it changes (last)
        for (int t = threadIdx.x; t < n * n; t += 256) {
            const int r = t / n, c = t % n;
            if (r == k) continue;
            const float m = A[r][k];
            B[r][c] -= m * B[k][c];
            if (c != k) A[r][c] -= m * A[k][c];
        }
        __syncthreads();
        for (int r = threadIdx.x; r < n; r += 256)
            if (r != k) A[r][k] = 0.f;
        __syncthreads();
    }
    for (int t = threadIdx.x; t < n * n; t += 256) {
        const int r = t / n, c = t % n;
        const bool dead = !(l.dinv[r] > 0.f) || !(l.dinv[c] > 0.f);
        inv[t] = dead ? 0.f : 0.5f * (B[r][c] + B[c][r]);
    }
}

// -------------------------------------------------------------------------------------- solve
__device__ __forceinline__ float2 ld2(const float *p, long n) { return __ldcg(reinterpret_cast<const float2 *>(p) + n); }
__device__ __forceinline__ float2 ldr(const double *p, long n)
{
    const double2 v = __ldcg(reinterpret_cast<const double2 *>(p) + n);
    return make_float2((float)v.x, (float)v.y);
}
__device__ __forceinline__ float2 ldr(const float *p, long n) { return ld2(p, n); }

// row n of the stencil applied to the neighbours' values val(k), k = 0 .. 8 (any finite value where the
// neighbour is off the grid: its coefficients are 0)
template <typename F> __device__ __forceinline__ float2 stencil(const float *S, F &&val)
{
    float2 s = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const float2 v = val(k);
        s.x += S[4 * k] * v.x + S[4 * k + 1] * v.y;
        s.y += S[4 * k + 2] * v.x + S[4 * k + 3] * v.y;
    }
    return s;
}
template <typename V> __device__ __forceinline__ void load_stencil(const V *S, int nn, long n, V *s)
{
#pragma unroll
    for (int k = 0; k < 36; ++k) s[k] = __ldg(S + (long)k * nn + n);
}

// bilinear interpolation of the coarse values get(I, J) at fine node (i, j): four values, some the same
template <typename F> __device__ __forceinline__ float2 interpolate(int i, int j, F &&get)
{
    const int I = i >> 1, J = j >> 1, I1 = I + (i & 1), J1 = J + (j & 1);
    const float2 a = get(I, J), b = get(I1, J), c = get(I, J1), d = get(I1, J1);
    return make_float2(0.25f * ((a.x + b.x) + (c.x + d.x)), 0.25f * ((a.y + b.y) + (c.y + d.y)));
}

// Phase down from level f to c: r_c = P^T (r - A (dinv r)) on tiles of f.cw x f.ch coarse nodes. rn(i, j, n,
// own) gives the residual of a fine node; `own` says that this block is the one the node belongs to.
template <typename F>
__device__ __forceinline__ void phase_down(const MgLevel &f, const MgLevel &c, float2 *sy, float2 *sr, F &&rn)
{
    const int nx1 = f.nx + 1, cw = f.cw, ch = f.ch;
    const int W = 2 * cw + 3, H = 2 * ch + 3, W1 = W - 2, H1 = H - 2;
    const int tx = (c.nx + cw) / cw, ty = (c.ny + ch) / ch;                  // ceil((nx + 1) / cw)
    for (int t = blockIdx.x; t < tx * ty; t += gridDim.x) {
        const int I0 = (t % tx) * cw, J0 = (t / tx) * ch;
        __syncthreads();
        for (int q = threadIdx.x; q < W * H; q += T) {
            const int li = q % W, lj = q / W, i = 2 * I0 - 2 + li, j = 2 * J0 - 2 + lj;
            float2 y = make_float2(0.f, 0.f);
            if (i >= 0 && j >= 0 && i <= f.nx && j <= f.ny) {
                const long n = (long)j * nx1 + i;
                const float2 d = __ldg(reinterpret_cast<const float2 *>(f.dinv) + n);
                const float2 r = rn(i, j, n, li >= 2 && lj >= 2 && li < 2 * cw + 2 && lj < 2 * ch + 2);
                y = make_float2(d.x * r.x, d.y * r.y);
                if (li >= 1 && lj >= 1 && li <= W1 && lj <= H1) sr[(lj - 1) * W1 + li - 1] = r;
            }
            sy[q] = y;
        }
        __syncthreads();
        for (int q = threadIdx.x; q < W1 * H1; q += T) {
            const int li = q % W1, lj = q / W1, i = 2 * I0 - 1 + li, j = 2 * J0 - 1 + lj;
            float2 v = make_float2(0.f, 0.f);
            if (i >= 0 && j >= 0 && i <= f.nx && j <= f.ny) {
                const long n = (long)j * nx1 + i;
                float S[36];
                load_stencil(f.S, f.nn, n, S);
                const float2 a = stencil(S, [&](int k) { return sy[(lj + k / 3) * W + li + k % 3]; });
                // clamped dofs and dofs without stiffness take no part
                const float2 d = __ldg(reinterpret_cast<const float2 *>(f.dinv) + n), r = sr[q];
                v = make_float2(d.x > 0.f ? r.x - a.x : 0.f, d.y > 0.f ? r.y - a.y : 0.f);
            }
            sr[q] = v;                                         // read by this thread alone until here
        }
        __syncthreads();
        for (int q = threadIdx.x; q < cw * ch; q += T) {
            const int li = q % cw, lj = q / cw, I = I0 + li, J = J0 + lj;
            if (I > c.nx || J > c.ny) continue;
            float2 s = make_float2(0.f, 0.f);
#pragma unroll
            for (int b = -1; b <= 1; ++b)
#pragma unroll
                for (int e = -1; e <= 1; ++e) {
                    const float w = (e ? 0.5f : 1.f) * (b ? 0.5f : 1.f);
                    const float2 v = sr[(2 * lj + 1 + b) * W1 + 2 * li + 1 + e];
                    s.x += w * v.x;
                    s.y += w * v.y;
                }
            const long n = (long)J * (c.nx + 1) + I;
            const float2 d = __ldg(reinterpret_cast<const float2 *>(c.dinv) + n);
            __stcg(reinterpret_cast<float2 *>(c.r) + n, make_float2(d.x > 0.f ? s.x : 0.f, d.y > 0.f ? s.y : 0.f));
        }
    }
}

// Phase up: z = y + dinv (r - A y), y = dinv r + P z_c, on tiles of f.tw x f.th nodes; returns the thread's
// share of r . z (FP64) on the finest level
template <typename R>
__device__ __forceinline__ double phase_up(const MgLevel &f, const MgLevel &c, const R *r, float2 *sy)
{
    const int nx1 = f.nx + 1, tw = f.tw, th = f.th, W = tw + 2, H = th + 2;
    const int tx = (f.nx + tw) / tw, ty = (f.ny + th) / th;
    double dot = 0.0;
    for (int t = blockIdx.x; t < tx * ty; t += gridDim.x) {
        const int i0 = (t % tx) * tw, j0 = (t / tx) * th;
        const int li = threadIdx.x % tw, lj = threadIdx.x / tw, i = i0 + li, j = j0 + lj;
        const bool mine = lj < th && i <= f.nx && j <= f.ny;
        const long n = (long)j * nx1 + i;
        float S[36];
        if (mine) load_stencil(f.S, f.nn, n, S);
        __syncthreads();
        for (int q = threadIdx.x; q < W * H; q += T) {
            const int ni = i0 - 1 + q % W, nj = j0 - 1 + q / W;
            float2 y = make_float2(0.f, 0.f);
            if (ni >= 0 && nj >= 0 && ni <= f.nx && nj <= f.ny) {
                const long m = (long)nj * nx1 + ni;
                const float2 rr = ldr(r, m), d = __ldg(reinterpret_cast<const float2 *>(f.dinv) + m);
                const float2 p = interpolate(ni, nj, [&](int I, int J) { return ld2(c.z, (long)J * (c.nx + 1) + I); });
                y = make_float2(d.x > 0.f ? d.x * rr.x + p.x : 0.f, d.y > 0.f ? d.y * rr.y + p.y : 0.f);
            }
            sy[q] = y;
        }
        __syncthreads();
        if (mine) {
            const float2 a = stencil(S, [&](int k) { return sy[(lj + k / 3) * W + li + k % 3]; });
            const float2 rr = ldr(r, n), d = __ldg(reinterpret_cast<const float2 *>(f.dinv) + n), y = sy[(lj + 1) * W + li + 1];
            const float2 z = make_float2(y.x + d.x * (rr.x - a.x), y.y + d.y * (rr.y - a.y));
            __stcg(reinterpret_cast<float2 *>(f.z) + n, z);
            if constexpr (sizeof(R) == 8) {
                const double2 rd = __ldcg(reinterpret_cast<const double2 *>(r) + n);
                dot += rd.x * z.x + rd.y * z.y;
            }
        }
    }
    return dot;
}

// one damped Jacobi sweep inside a block: dst = src + dinv (r - A src)
__device__ __forceinline__ void small_sweep(const MgLevel &f, const float2 *r, const float2 *src, float2 *dst)
{
    const int nx1 = f.nx + 1;
    for (int n = threadIdx.x; n < f.nn; n += T) {
        const int i = n % nx1, j = n / nx1;
        float S[36];
        load_stencil(f.S, f.nn, n, S);
        const float2 s = stencil(S, [&](int k) {
            return src[min(max(j + k / 3 - 1, 0), f.ny) * nx1 + min(max(i + k % 3 - 1, 0), f.nx)];
        });
        const float2 d = __ldg(reinterpret_cast<const float2 *>(f.dinv) + n), v = src[n];
        dst[n] = make_float2(v.x + d.x * (r[n].x - s.x), v.y + d.y * (r[n].y - s.y));
    }
    __syncthreads();
}

// the levels from first_small down, inside one block, on the residual r: sr / sz hold each level's
// residual and correction, tmp a level's scratch
template <typename R>
__device__ __forceinline__ void small_cycle(const MgArgs &a, const R *r, float2 *sr, float2 *sz, float2 *tmp)
{
    static_assert(kSweeps % 2 == 0, "an even number of sweeps ends in the buffer it began in");
    const int l0 = a.first_small;
    __syncthreads();
    for (int n = threadIdx.x; n < a.lv[l0].nn; n += T) sr[n] = ldr(r, n);
    __syncthreads();
    float2 *R_ = sr, *Z_ = sz;
    int l = l0;
    for (; l + 1 < a.levels; ++l) {
        const MgLevel &f = a.lv[l], &c = a.lv[l + 1];
        const int nx1 = f.nx + 1;
        // sweeps from zero: the first is the scaled residual, the last lands in Z_
        for (int n = threadIdx.x; n < f.nn; n += T) {
            const float2 d = __ldg(reinterpret_cast<const float2 *>(f.dinv) + n);
            tmp[n] = make_float2(d.x * R_[n].x, d.y * R_[n].y);
        }
        __syncthreads();
        for (int k = 1; k < kSweeps; ++k) small_sweep(f, R_, k & 1 ? tmp : Z_, k & 1 ? Z_ : tmp);
        for (int n = threadIdx.x; n < f.nn; n += T) {
            const int i = n % nx1, j = n / nx1;
            float S[36];
            load_stencil(f.S, f.nn, n, S);
            const float2 s = stencil(S, [&](int k) {
                return Z_[min(max(j + k / 3 - 1, 0), f.ny) * nx1 + min(max(i + k % 3 - 1, 0), f.nx)];
            });
            const float2 d = __ldg(reinterpret_cast<const float2 *>(f.dinv) + n);
            tmp[n] = make_float2(d.x > 0.f ? R_[n].x - s.x : 0.f, d.y > 0.f ? R_[n].y - s.y : 0.f);
        }
        __syncthreads();
        float2 *Rc = R_ + f.nn;
        for (int n = threadIdx.x; n < c.nn; n += T) {
            const int I = n % (c.nx + 1), J = n / (c.nx + 1);
            float2 s = make_float2(0.f, 0.f);
#pragma unroll
            for (int b = -1; b <= 1; ++b)
#pragma unroll
                for (int e = -1; e <= 1; ++e) {
                    const int i = 2 * I + e, j = 2 * J + b;
                    const bool in = i >= 0 && j >= 0 && i <= f.nx && j <= f.ny;
                    const float w = in ? (e ? 0.5f : 1.f) * (b ? 0.5f : 1.f) : 0.f;
                    const float2 v = tmp[in ? j * nx1 + i : 0];
                    s.x += w * v.x;
                    s.y += w * v.y;
                }
            const float2 d = __ldg(reinterpret_cast<const float2 *>(c.dinv) + n);
            Rc[n] = make_float2(d.x > 0.f ? s.x : 0.f, d.y > 0.f ? s.y : 0.f);
        }
        __syncthreads();
        R_ = Rc;
        Z_ += f.nn;
    }
    {
        const int n2 = 2 * a.lv[l].nn;
        const float *rc = reinterpret_cast<const float *>(R_);
        for (int t = threadIdx.x; t < n2; t += T) {
            float s = 0.f;
#pragma unroll 8
            for (int k = 0; k < n2; ++k) s += __ldg(a.inv + k * n2 + t) * rc[k];
            reinterpret_cast<float *>(Z_)[t] = s;
        }
        __syncthreads();
    }
    for (--l; l >= l0; --l) {
        const MgLevel &f = a.lv[l], &c = a.lv[l + 1];
        const float2 *Zc = Z_;
        Z_ -= f.nn;
        R_ -= f.nn;
        for (int n = threadIdx.x; n < f.nn; n += T) {
            const int i = n % (f.nx + 1), j = n / (f.nx + 1);
            const float2 p = interpolate(i, j, [&](int I, int J) { return Zc[J * (c.nx + 1) + I]; });
            const float2 d = __ldg(reinterpret_cast<const float2 *>(f.dinv) + n);
            if (d.x > 0.f) Z_[n].x += p.x;
            if (d.y > 0.f) Z_[n].y += p.y;
        }
        __syncthreads();
        for (int k = 0; k < kSweeps; ++k) small_sweep(f, R_, k & 1 ? tmp : Z_, k & 1 ? Z_ : tmp);
    }
    const MgLevel &f = a.lv[l0];
    for (int n = threadIdx.x; n < f.nn; n += T) __stcg(reinterpret_cast<float2 *>(f.z) + n, sz[n]);
}

struct __align__(16) Shared {            // sr also holds a tile of double2
    float2 sr[kSmallSum], sz[kSmallSum], tmp[kMgSmall];
};

// z = M^-1 r after the finest phase down (or from r itself when every level is small); adds r . z to *rz.
// false after a barrier that gave up.
__device__ __forceinline__ bool v_cycle(const MgArgs &a, GridBarrier &g, Shared &sh, const double *r, double *red, double *rz)
{
    const int m = a.first_small;
    for (int l = 1; l < m; ++l) {
        phase_down(a.lv[l], a.lv[l + 1], sh.sr, sh.sz, [&](int, int, long n, bool) { return ld2(a.lv[l].r, n); });
        if (!g.wait()) return false;
    }
    if (blockIdx.x == 0) {
        if (m == 0) small_cycle(a, r, sh.sr, sh.sz, sh.tmp);
        else small_cycle(a, a.lv[m].r, sh.sr, sh.sz, sh.tmp);
    }
    if (!g.wait()) return false;
    for (int l = m - 1; l > 0; --l) {
        phase_up(a.lv[l], a.lv[l + 1], a.lv[l].r, sh.sr);
        if (!g.wait()) return false;
    }
    double dot = 0.0;
    if (m > 0) {
        dot = phase_up(a.lv[0], a.lv[1], r, sh.sr);
    } else {
        for (int n = blockIdx.x * T + threadIdx.x; n < a.lv[0].nn; n += gridDim.x * T) {
            const double2 v = __ldcg(reinterpret_cast<const double2 *>(r) + n);
            const float2 z = ld2(a.lv[0].z, n);
            dot += v.x * z.x + v.y * z.y;
        }
    }
    dot = block_sum(dot, red);
    if (threadIdx.x == 0) atomicAdd(rz, dot);
    return g.wait();
}

__global__ void __launch_bounds__(T, 1) mg_solve_kernel(const __grid_constant__ MgArgs a)
{
    __shared__ Shared sh;
    __shared__ double red[T / 32], one;
    static_assert(sizeof(float2) * kSmallSum >= sizeof(double2) * kHalo, "a staged tile fits one buffer");
    static_assert(alignof(Shared) % alignof(double2) == 0, "and is aligned for it");
    GridBarrier g;
    g.bar = a.bar;
    const MgLevel &f = a.lv[0];
    const int nx1 = f.nx + 1, step = gridDim.x * T, first = blockIdx.x * T + threadIdx.x;
    const bool small = a.first_small == 0;
    double2 *x = reinterpret_cast<double2 *>(a.x), *q = reinterpret_cast<double2 *>(a.q);
    const double *b = a.force;               // the caller's: any FP64 alignment
    double *sc = a.sc;
    // x = 0, r = f on the free dofs, p = 0
    double ff = 0.0;
    for (int n = first; n < f.nn; n += step) {
        double2 v = make_double2(b[2 * (long)n], b[2 * (long)n + 1]);
        if (a.fixed[2 * n]) v.x = 0.0;
        if (a.fixed[2 * n + 1]) v.y = 0.0;
        __stcg(reinterpret_cast<double2 *>(a.r0) + n, v);
        __stcg(x + n, make_double2(0.0, 0.0));
        __stcg(q + n, make_double2(0.0, 0.0));
        __stcg(reinterpret_cast<double2 *>(a.p0) + n, make_double2(0.0, 0.0));
        __stcg(reinterpret_cast<double2 *>(a.p1) + n, make_double2(0.0, 0.0));
        ff += v.x * v.x + v.y * v.y;
    }
    ff = block_sum(ff, red);
    if (threadIdx.x == 0) atomicAdd(sc + kScFf, ff);
    if (!g.wait()) return;
    ff = __ldcg(sc + kScFf);
    const double stop = a.tol2 * ff;
    bool done = ff == 0.0;
    double rr = ff, rz = 1.0, alpha = 0.0;
    double best = ff;                        // |r|^2 that the last halving of |r| reached, and when
    int it = 0, best_it = 0;                 // iterations done
    // Pass k applies iteration k's step to x and r (none in pass 0), then z = M^-1 r, then the next direction
    // and its product with the operator. r and p alternate between two buffers: neighbours read the old ones.
    while (!done) {
        double2 *pn = reinterpret_cast<double2 *>(it & 1 ? a.p0 : a.p1), *po = reinterpret_cast<double2 *>(it & 1 ? a.p1 : a.p0);
        const double2 *ro = reinterpret_cast<const double2 *>(it & 1 ? a.r0 : a.r1);
        double2 *rn = reinterpret_cast<double2 *>(it & 1 ? a.r1 : a.r0);
        // r -= alpha q, x += alpha p (po: the direction of the step), rr
        rr = 0.0;
        auto step_node = [&](long n, bool own) {
            if (!it) return __ldcg(rn + n);
            const double2 w = __ldcg(q + n);
            double2 v = __ldcg(ro + n);
            v.x -= alpha * w.x;
            v.y -= alpha * w.y;
            if (own) {
                const double2 p = __ldcg(po + n);
                double2 xn = __ldcg(x + n);
                xn.x += alpha * p.x;
                xn.y += alpha * p.y;
                __stcg(x + n, xn);
                __stcg(rn + n, v);
                rr += v.x * v.x + v.y * v.y;
            }
            return v;
        };
        if (small) {
            for (int n = first; n < f.nn; n += step) step_node(n, true);
        } else {
            phase_down(a.lv[0], a.lv[1], sh.sr, sh.sz, [&](int, int, long n, bool own) {
                const double2 v = step_node(n, own);
                return make_float2((float)v.x, (float)v.y);
            });
        }
        if (it) {
            rr = block_sum(rr, red);
            if (threadIdx.x == 0) atomicAdd(sc + kScRr + it % 3, rr);
        }
        if (!g.wait()) return;
        if (it) {
            rr = __ldcg(sc + kScRr + it % 3);
            done = rr <= stop;
            if (done || it >= a.max_iter) break;
            if (it % 16 == 0) {
                if (rr < 0.25 * best) {
                    best = rr;
                    best_it = it;
                } else if (it - best_it >= a.patience) {
                    break;                   // stalled: leave it to the plain iteration
                }
            }
        }
        // the sums of the pass before are free again: nobody reads them past the barrier above
        if (first == 0) {
            __stcg(sc + kScRr + (it + 2) % 3, 0.0);
            __stcg(sc + kScPq + (it + 2) % 3, 0.0);
            __stcg(sc + kScRz + (it + 2) % 3, 0.0);
        }
        if (!v_cycle(a, g, sh, reinterpret_cast<const double *>(rn), red, sc + kScRz + it % 3)) return;
        const double rz_new = __ldcg(sc + kScRz + it % 3);
        if (!(rz_new > 0.0)) break;          // also NaN: leave it to the plain iteration
        const double beta = scalar([&]() { return it ? rz_new / rz : 0.0; }, &one);
        rz = rz_new;
        // p = z + beta p and q = A p on tiles; the halo's p is formed here too
        double pq = 0.0;
        {
            double2 *sp = reinterpret_cast<double2 *>(sh.sr);
            const int tw = f.tw, th = f.th, W = tw + 2, H = th + 2, tx = (f.nx + tw) / tw, ty = (f.ny + th) / th;
            for (int t = blockIdx.x; t < tx * ty; t += gridDim.x) {
                const int i0 = (t % tx) * tw, j0 = (t / tx) * th;
                const int li = threadIdx.x % tw, lj = threadIdx.x / tw, i = i0 + li, j = j0 + lj;
                const bool mine = lj < th && i <= f.nx && j <= f.ny;
                const long n = (long)j * nx1 + i;
                double S[36];
                if (mine) load_stencil(a.S64, f.nn, n, S);
                __syncthreads();
                for (int e = threadIdx.x; e < W * H; e += T) {
                    const int ni = i0 - 1 + e % W, nj = j0 - 1 + e / W;
                    double2 v = make_double2(0.0, 0.0);
                    if (ni >= 0 && nj >= 0 && ni <= f.nx && nj <= f.ny) {
                        const long m = (long)nj * nx1 + ni;
                        const float2 z = ld2(f.z, m);
                        const double2 p = __ldcg(po + m);
                        v = make_double2(z.x + beta * p.x, z.y + beta * p.y);
                    }
                    sp[e] = v;
                }
                __syncthreads();
                if (!mine) continue;
                double qx = 0.0, qy = 0.0;
#pragma unroll
                for (int k = 0; k < 9; ++k) {
                    const double2 u = sp[(lj + k / 3) * W + li + k % 3];
                    qx += S[4 * k] * u.x;
                    qx += S[4 * k + 1] * u.y;
                    qy += S[4 * k + 2] * u.x;
                    qy += S[4 * k + 3] * u.y;
                }
                const double2 p = sp[(lj + 1) * W + li + 1];
                __stcg(pn + n, p);
                __stcg(q + n, make_double2(qx, qy));
                pq += p.x * qx + p.y * qy;
            }
        }
        pq = block_sum(pq, red);
        if (threadIdx.x == 0) atomicAdd(sc + kScPq + it % 3, pq);
        if (!g.wait()) return;
        pq = __ldcg(sc + kScPq + it % 3);
        if (!(pq > 0.0)) break;
        alpha = scalar([&]() { return rz / pq; }, &one);
        ++it;
    }
    // compliance f . u
    double c = 0.0;
    for (int n = first; n < f.nn; n += step) {
        const double2 u = __ldcg(x + n);
        c += b[2 * (long)n] * u.x + b[2 * (long)n + 1] * u.y;
    }
    c = block_sum(c, red);
    if (threadIdx.x == 0) atomicAdd(sc + kScC, c);
    if (first == 0) {
        sc[kScIt] = it;
        sc[kScDone] = done ? 1.0 : 0.0;
        sc[kScLast] = rr;
    }
}

// ------------------------------------------------------------------------- optimality criteria
__global__ void __launch_bounds__(T) oc_solve_kernel(const __grid_constant__ OcArgs a)
{
    __shared__ double red[T / 32], one;
    GridBarrier g;
    g.bar = a.bar;
    const long first = blockIdx.x * (long)T + threadIdx.x, step = (long)gridDim.x * T;
    const double eb = exp(-a.beta);
    double cnt = 0.0;
    for (long i = first; i < a.n; i += step) {
        const double s = fmax((double)a.S[i], 0.0);
        a.xs[i] = a.xi[i] * (a.eta == 0.5 ? sqrt(s) : pow(s, a.eta));
        if (!(a.passive && a.passive[i])) cnt += 1.0;
    }
    cnt = block_sum(cnt, red);
    if (threadIdx.x == 0) atomicAdd(a.sc + 6, cnt);
    if (!g.wait()) return;
    const double target = a.volfrac * __ldcg(a.sc + 6);
    // the update at the multiplier whose power lam^-eta is li: xi (S / lam)^eta within the move limit and
    // [0, 1]; the sum of the projected densities of the free elements and its slope in log lam, and with
    // `write` also xi_new and sum |xi_new - xi| (in place of the slope)
    auto sum = [&](double li, bool write, double &second) {
        double vol = 0.0;
        second = 0.0;
        for (long i = first; i < a.n; i += step) {
            const bool pas = a.passive && a.passive[i];
            const double x = a.xi[i], w = a.xs[i] * li;
            double v = fmin(w, fmin(1.0, x + a.move));
            v = fmax(v, fmax(0.0, x - a.move));
            if (write) a.out[i] = pas ? 1.f : (float)v;
            if (pas) continue;
            const double e = exp(-a.beta * v);
            vol += 1.0 - e + v * eb;
            if (write) second += fabs(v - x);
            else if (v == w) second -= a.eta * v * (a.beta * e + eb);
        }
        return vol;
    };
    // Root of volume = target in u = log lam on the bracket [log 1e-12, log 1e12]: Newton steps, halving the
    // bracket where a step leaves it, the slope vanishes or the step is not half the one before; done when
    // a step is below 2e-10 or the bracket below 1e-9 (the bisection on the host ends at the latter). About
    // eight sums where bisection takes 36. A volume that stays above (below) the target ends at the bracket's
    // upper (lower) end, as there.
    double lo = -27.631021115928547, hi = 27.631021115928547, u = 0.0, last = 1e300;
    for (int k = 0; k < 200; ++k) {
        const double li = scalar([&]() { return exp(-a.eta * u); }, &one);
        double slope;
        double part = sum(li, false, slope);
        part = block_sum(part, red);
        slope = block_sum(slope, red);
        if (threadIdx.x == 0) {
            atomicAdd(a.sc + 2 * (k % 3), part);
            atomicAdd(a.sc + 2 * (k % 3) + 1, slope);
        }
        if (!g.wait()) return;
        const double f = __ldcg(a.sc + 2 * (k % 3)) - target, d = __ldcg(a.sc + 2 * (k % 3) + 1);
        // the sums of the step before are free again: nobody reads them past the barrier above
        if (first == 0) {
            __stcg(a.sc + 2 * ((k + 2) % 3), 0.0);
            __stcg(a.sc + 2 * ((k + 2) % 3) + 1, 0.0);
        }
        if (f > 0.0) lo = u;
        else hi = u;
        const double newton = scalar([&]() { return d < 0.0 ? u - f / d : 1e300; }, &one), move = fabs(newton - u);
        const bool take = newton > lo && newton < hi && move < 0.5 * last;
        const double to = take ? newton : 0.5 * (lo + hi);
        last = take ? move : 1e300;
        u = to;
        if ((take && move < 2e-10) || hi - lo < 1e-9) break;
    }
    double chg;
    const double li = scalar([&]() { return exp(-a.eta * u); }, &one);
    double vol = sum(li, true, chg);
    vol = block_sum(vol, red);
    chg = block_sum(chg, red);
    if (threadIdx.x == 0) {
        atomicAdd(a.sc + 8, vol);
        atomicAdd(a.sc + 7, chg);
    }
}

int blocks(long n) { return (int)std::max(1L, std::min((n + 127) / 128, 65535L)); }

} // namespace

size_t mg_plan(int nx, int ny, double nu, MgArgs &a)
{
    // Jacobi damping inside the spectrum of the diagonally scaled element matrix, whose largest eigenvalue
    // (dilation 1 / (1 - nu) or shear 1 / (1 + nu) over the diagonal (1/2 - nu/6) / (1 - nu^2)) bounds the operator's
    const double diag = (0.5 - nu / 6.0) / (1.0 - nu * nu), most = std::max(1.0 / (1.0 - nu), 1.0 / (1.0 + nu)) / diag;
    a.omega = (float)(1.9 / most);
    size_t bytes = 0;
    a.levels = 0;
    a.first_small = -1;
    while (true) {
        MgLevel &l = a.lv[a.levels];
        l = MgLevel{};
        l.nx = nx;
        l.ny = ny;
        l.nn = (nx + 1) * (ny + 1);
        // the tiles that leave the fewest of them: with a halo of one (up) or three fine nodes a side (down)
        long best_t = 1L << 60, best_c = 1L << 60;
        const int cx = (nx + 1) / 2 + 1, cy = (ny + 1) / 2 + 1;
        for (int w = 1; w <= T; ++w)
            for (int h = 1; w * h <= T; ++h) {
                const long t = (long)((nx + w) / w) * ((ny + h) / h), c = (long)((cx + w - 1) / w) * ((cy + h - 1) / h);
                if ((w + 2) * (h + 2) <= kHalo && (t < best_t || (t == best_t && w + h < l.tw + l.th))) {
                    best_t = t;
                    l.tw = w;
                    l.th = h;
                }
                if ((2 * w + 3) * (2 * h + 3) <= kHalo && (c < best_c || (c == best_c && w + h < l.cw + l.ch))) {
                    best_c = c;
                    l.cw = w;
                    l.ch = h;
                }
            }
        if (a.first_small < 0 && l.nn <= kMgSmall) a.first_small = a.levels;
        bytes += (size_t)l.nn * ((36 + 2 + 2 + 2) * 4 + 2) + 1024;
        if (!a.levels) bytes += (size_t)l.nn * (36 * 8 + 16) + 512;
        ++a.levels;
        if (l.nn <= kMgCoarse) break;
        if (a.levels == kMgMaxLevels) return 0;
        nx = (nx + 1) / 2;
        ny = (ny + 1) / 2;
    }
    return bytes + (size_t)4 * kMgCoarse * kMgCoarse * 4 + 128;
}

void mg_place(MgArgs &a, void *mem)
{
    char *p = static_cast<char *>(mem);
    auto take = [&](size_t bytes) {
        void *q = p;
        p += (bytes + 127) / 128 * 128;
        return q;
    };
    for (int l = 0; l < a.levels; ++l) {
        MgLevel &v = a.lv[l];
        v.S = static_cast<float *>(take((size_t)v.nn * 36 * 4));
        v.dinv = static_cast<float *>(take((size_t)v.nn * 8));
        v.r = static_cast<float *>(take((size_t)v.nn * 8));
        v.z = static_cast<float *>(take((size_t)v.nn * 8));
        v.fixed = static_cast<uint8_t *>(take((size_t)v.nn * 2));
    }
    a.S64 = static_cast<double *>(take((size_t)a.lv[0].nn * 36 * 8));
    a.r1 = static_cast<double *>(take((size_t)a.lv[0].nn * 16));
    a.inv = static_cast<float *>(take((size_t)4 * kMgCoarse * kMgCoarse * 4));
}

void mg_setup(const MgArgs &a, cudaStream_t s)
{
    mg_stencil_kernel<<<blocks(a.lv[0].nn), 128, 0, s>>>(a.lv[0], a.k0, a.E, a.fixed, a.S64, a.omega);
    for (int l = 1; l < a.levels; ++l) mg_rap_kernel<<<blocks(a.lv[l].nn), 128, 0, s>>>(a.lv[l - 1], a.lv[l], a.omega);
    mg_inverse_kernel<<<1, 256, 0, s>>>(a.lv[a.levels - 1], const_cast<float *>(a.inv));
}

cudaError_t mg_solve(const MgArgs &a, cudaStream_t s)
{
    const MgLevel &l = a.lv[0];
    return imf::launch_cooperative(mg_solve_kernel, a, T, (long)((l.nx + l.tw) / l.tw) * ((l.ny + l.th) / l.th), s);
}
cudaError_t oc_solve(const OcArgs &a, cudaStream_t s) { return imf::launch_cooperative(oc_solve_kernel, a, T, (a.n + T - 1) / T, s); }

} // namespace imf_to
