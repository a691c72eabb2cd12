// Host-only exports that run the kernels' building blocks (fft.cuh, fft2.cuh, erode_plan.h,
// fft_plan.h, orient_order.h, sweep_bits.cuh) on the CPU, for the CPU unit tests. Not part of
// libimf and never loaded by the product path.
#include <chrono>
#include <cmath>
#include <condition_variable>
#include <cstring>
#include <mutex>
#include <thread>
#include <vector>

#include "fft.cuh"
#include "fft2.cuh"
#include "erode_plan.h"
#include "erode_stream.h"
#include "fft_plan.h"
#include "fft_tma.cuh"
#include "grid_barrier.cuh"
#include "launch_errors.h"
#include "orient_order.h"
#include "sweep_bits.cuh"
#include "sweep_plan.h"
#include "topopt2d_mg.cuh"

extern "C" int imf_host_fft(int L, int sign, const float *in, float *out)
{
    imf::FftPlan p;
    if (L < 1 || !imf::make_plan(L, &p)) return -1;
    std::vector<float2> tw(L), a(L), b(L);
    for (int m = 0; m < L; ++m) {
        const double ang = -2.0 * M_PI * (double)m / (double)L;
        tw[m] = make_float2((float)std::cos(ang), (float)std::sin(ang));
        a[m] = make_float2(in[2 * m], in[2 * m + 1]);
    }
    float2 *r = sign < 0 ? imf::fft_pencil_host<-1>(p, a.data(), b.data(), tw.data())
                         : imf::fft_pencil_host<1>(p, a.data(), b.data(), tw.data());
    for (int m = 0; m < L; ++m) {
        out[2 * m] = r[m].x;
        out[2 * m + 1] = r[m].y;
    }
    return p.nrad;
}

// Number of (d, j) pairs, 2 <= d <= maxd, 0 <= j < maxj, where the stage reciprocal disagrees
// with integer division.
extern "C" long imf_host_check_div(int maxd, int maxj)
{
    long bad = 0;
    for (int d = 1; d <= maxd; ++d) {
        const unsigned mul = imf::div_magic((unsigned)d);
        for (int j = 0; j < maxj; ++j)
            if (imf::fast_div((unsigned)j, mul) != (unsigned)(j / d)) ++bad;
    }
    return bad;
}

// The two-pass register transform of fft2.cuh on one pencil. Returns 100 A + B for the split
// it used, or -1 when L has no supported split.
extern "C" int imf_host_fft2(int L, int sign, const float *in, float *out)
{
    int A = 0, B = 0;
    if (L < 4 || !imf::fft2::choose_split(L, &A, &B, imf::fft2::kMaxFactorBig)) return -1;
    std::vector<float2> tw(L), x(L), X(L), T(L);
    for (int m = 0; m < L; ++m) {
        const double ang = -2.0 * M_PI * (double)m / (double)L;
        tw[m] = make_float2((float)std::cos(ang), (float)std::sin(ang));
        x[m] = make_float2(in[2 * m], in[2 * m + 1]);
    }
    if (sign < 0) imf::fft2::fft2_pencil_host<-1>(A, B, x.data(), X.data(), T.data(), tw.data());
    else imf::fft2::fft2_pencil_host<1>(A, B, x.data(), X.data(), T.data(), tw.data());
    for (int m = 0; m < L; ++m) {
        out[2 * m] = X[m].x;
        out[2 * m + 1] = X[m].y;
    }
    return 100 * A + B;
}

// The plan of the tiled minimum over sharp points for one orientation's sharp offsets
// (n_pts triples x, y, z), window origin K and longest run maxL (16 or 31). Writes per chunk 44
// ints (run0, run1, txh, tyh, tzh, pitch_y, pitch_z, ox, oy, oz, lend[0..31], 0, 0) and per run
// 2 ints (tile offset, length). Returns the number of chunks, or -1 when the output arrays are
// too small; *smem gets the largest tile in bytes and *nruns the number of runs.
extern "C" int imf_host_plan_erode(const int *sh, int n_pts, const int *K, int maxL, int max_chunks, int *chunk_out,
                                   int max_runs, int *runs_out, long *smem, int *nruns)
{
    std::vector<int32_t> v(sh, sh + 3 * (size_t)n_pts);
    std::vector<imf::ErodeChunk> chunks;
    std::vector<int2> runs;
    size_t sm = 0;
    imf::plan_erode(v, K, chunks, runs, sm, maxL);
    *smem = (long)sm;
    *nruns = (int)runs.size();
    if ((int)chunks.size() > max_chunks || (int)runs.size() > max_runs) return -1;
    for (size_t c = 0; c < chunks.size(); ++c) {
        const imf::ErodeChunk &ch = chunks[c];
        int *o = chunk_out + 44 * c;
        const int head[10] = {ch.run0, ch.run1, ch.txh, ch.tyh, ch.tzh, ch.pitch_y, ch.pitch_z, ch.ox, ch.oy, ch.oz};
        for (int i = 0; i < 10; ++i) o[i] = head[i];
        for (int i = 0; i <= imf::kErMaxL3; ++i) o[10 + i] = ch.lend[i];
        o[42] = o[43] = 0;
    }
    for (size_t r = 0; r < runs.size(); ++r) {
        runs_out[2 * r] = runs[r].x;
        runs_out[2 * r + 1] = runs[r].y;
    }
    return (int)chunks.size();
}

// Tile geometry constants of the plan (kErTX, kErTY, kErTZ, kErXT, kErMaxL, budget bytes,
// runs per chunk).
extern "C" void imf_host_erode_constants(long *out)
{
    out[0] = imf::kErTX; out[1] = imf::kErTY; out[2] = imf::kErTZ; out[3] = imf::kErXT;
    out[4] = imf::kErMaxL; out[5] = (long)imf::kErodeBudget; out[6] = imf::kErMaxRunsPerChunk;
}

// One cutter run of the sweep as the kernels compute it (sweep_bits.cuh): the dilation levels
// of a row of wpr words, then the two windows of the run's descriptor for output word q at
// shift s >= 0 and length L (1 .. 32). Returns 1 for arguments out of range (reads past the row).
extern "C" int imf_host_sweep_run(const uint32_t *row, int wpr, int q, int s, int L, uint32_t *out)
{
    if (!row || !out || wpr < 2 || q < 0 || s < 0 || L < 1 || L > 32) return 1;
    const int4 d = imf::sweep_pair(0, s, L);
    if (q + d.x + d.y + 1 >= wpr) return 1;
    std::vector<uint32_t> lev((size_t)imf::kSweepLevels * wpr);
    for (int w = 0; w < wpr; ++w) {
        uint32_t l[imf::kSweepLevels - 1];
        imf::sweep_level_words(row[w], w + 1 < wpr ? row[w + 1] : 0u, l);
        lev[w] = row[w];
        for (int j = 1; j < imf::kSweepLevels; ++j) lev[(size_t)j * wpr + w] = l[j - 1];
    }
    *out = imf::sweep_pair_bits(lev.data() + (size_t)d.w * wpr + q + d.x, d);
    return 0;
}

// The x pass's packing of 32 free-flag bytes into one word (pack_flag_bytes).
extern "C" uint32_t imf_host_pack_flags(const uint8_t *bytes32)
{
    uint32_t g8[8];
    std::memcpy(g8, bytes32, sizeof g8);
    return imf::pack_flag_bytes(g8);
}

// The padded length the planner picks for a minimum length n with two-pass factors up to maxA,
// and the split it then uses (A, B; 0 when the length runs the radix-stage kernels).
extern "C" int imf_host_plan_length(int n, int maxA, int *A, int *B)
{
    const int L = imf::best_smooth(n, maxA);
    *A = *B = 0;
    if (!imf::fft2::choose_split(L, A, B, maxA)) *A = *B = 0;
    return L;
}

// The internal orientation order for n rotations (row-major 3 x 3 each): the nearest-neighbour
// chain, interleaved by spread_order when `spread` is set.
extern "C" void imf_host_orient_order(const double *R, int n, int spread, int *out)
{
    std::vector<double> r(R, R + 9 * (size_t)n);
    std::vector<int> o = imf::locality_order(r, n);
    if (spread) o = imf::spread_order(o);
    for (int i = 0; i < n; ++i) out[i] = o[i];
}

// The plan of the streamed minimum over sharp points (erode_stream.h) of one orientation's sharp
// offsets. head gets P, R, Q, stages, tile x, rows, W, plane groups, axis, lists, rows and 16-byte
// columns copied, ox, ou, ow; words the descriptor words. Returns the number of words, -1 where the
// plan refuses the points and -2 when the output array is too small.
extern "C" int imf_host_plan_stream(const int *sh, int n_pts, const int *K, int *head, int max_words,
                                    int *words_out)
{
    std::vector<std::vector<int32_t>> v(1, std::vector<int32_t>(sh, sh + 3 * (size_t)n_pts));
    std::vector<imf::EsOrient> h;
    std::vector<int> words;
    imf::EsGeometry g;
    if (!imf::es_plan(v, K, g, h, words)) return -1;
    const int out[15] = {g.P, g.R, g.Q, g.stages, imf::kEsTX, imf::kEsRows, imf::kEsW, imf::kEsNW,
                         h[0].axis, h[0].lists, h[0].rows, h[0].quads, h[0].ox, h[0].ou, h[0].ow};
    std::memcpy(head, out, sizeof out);
    if ((int)words.size() > max_words || h[0].words != (int)words.size() || g.words != h[0].words) return -2;
    std::memcpy(words_out, words.data(), words.size() * sizeof(int));
    return (int)words.size();
}

// The plan of the sweep on staged tiles (sweep_plan.h) of one orientation's cutter offsets. head gets nq, nl,
// planes per warp, row pitch, largest word shift, planes staged, bytes, axis, eu, ew, ou, ow; words the descriptors.
// Returns the number of words, -1 where the plan refuses the cutter and -2 when the output array is too small.
extern "C" int imf_host_plan_sweep(const int *rk, int n_pts, const int *K, const int *kmin, int nx, int *head, int max_words,
                                   int *words_out)
{
    std::vector<std::vector<int32_t>> v(1, std::vector<int32_t>(rk, rk + 3 * (size_t)n_pts));
    std::vector<imf::SwOrient> h;
    std::vector<int> words;
    imf::SwGeometry g;
    if (!imf::sw_plan(v, K, kmin, nx, g, h, words)) return -1;
    const int out[12] = {g.nq, g.nl, g.ppw, g.UP, g.somax, g.planes, (int)g.smem, h[0].axis, h[0].eu, h[0].ew, h[0].ou, h[0].ow};
    std::memcpy(head, out, sizeof out);
    if ((int)words.size() > max_words || h[0].words != (int)words.size()) return -2;
    std::memcpy(words_out, words.data(), words.size() * sizeof(int));
    return (int)words.size();
}

namespace {

// The producers of one block of the streamed minimum on host threads: late[t * total + n] != 0 makes thread t's
// wait for the n-th stage (over all orientations) run out.
struct HostRing {
    std::mutex m;
    std::condition_variable cv;
    int threads, arrived = 0, generation = 0;
    bool any = false, result = false, stuck = false;

    bool vote(bool late)
    {
        std::unique_lock<std::mutex> lock(m);
        any = any || late;
        const int mine = generation;
        if (++arrived == threads) {
            result = any;
            any = false;
            arrived = 0;
            ++generation;
            cv.notify_all();
        } else if (!cv.wait_for(lock, std::chrono::seconds(2), [&] { return generation != mine || stuck; }) || stuck) {
            stuck = true;                // some thread will never come: the device would wait for ever
            cv.notify_all();
            return true;
        }
        return result;
    }
};
struct HostProducer {
    HostRing &ring;
    const int *n_steps;
    const uint8_t *late;
    int stop_at, n = 0, copied = 0;

    int steps(int k) { return n_steps[k]; }
    bool wait(int, uint32_t) { return !late[n]; }
    imf::EsOpen open(int k, int, bool is_late)
    {
        if (ring.vote(is_late)) return imf::EsOpen::leave;
        return k == stop_at ? imf::EsOpen::done : imf::EsOpen::copy;
    }
    void copy(int, int, int) { ++n; ++copied; }
};

} // namespace

// Runs es_produce on `threads` host threads; how[t] gets 0 where thread t copied everything, 1 where it stopped at
// orientation stop_at, 2 where it left on a timeout, and copied[t] its stages. Returns 1 when a thread was
// left waiting at the producers' barrier, else 0.
extern "C" int imf_host_stream_producers(int threads, int orientations, const int *n_steps, int stages, int stop_at,
                                         const uint8_t *late, int total, int *how, int *copied)
{
    HostRing ring;
    ring.threads = threads;
    std::vector<std::thread> pool;
    for (int t = 0; t < threads; ++t)
        pool.emplace_back([&, t] {
            HostProducer io{ring, n_steps, late + (size_t)t * total, stop_at};
            how[t] = (int)imf::es_produce(io, orientations, stages);
            copied[t] = io.copied;
        });
    for (auto &p : pool) p.join();
    return ring.stuck;
}

// The choice of a cooperative launch's blocks (grid_barrier.cuh) against a launcher with room for `room` blocks that
// otherwise returns `error`. Returns the blocks launched, or minus the error; tries gets the calls made.
extern "C" int imf_host_launch_fitting(long want, long room, int error, int *tries)
{
    long got = 0;
    *tries = 0;
    const cudaError_t e = imf::launch_fitting(want, [&](long n) {
        ++*tries;
        if (n > room) return cudaErrorCooperativeLaunchTooLarge;
        got = n;
        return (cudaError_t)error;
    });
    return e == cudaSuccess ? (int)got : -(int)e;
}

// Whether the analysis takes the result of a multigrid solve that ended with `done` and this barrier error word.
extern "C" int imf_host_mg_converged(double done, unsigned barrier_error)
{
    double sc[imf_to::kScN] = {0};
    sc[imf_to::kScDone] = done;
    const unsigned bar[2] = {12345u, barrier_error};
    return imf_to::mg_converged(sc, bar);
}

// Whether an analysis handle takes a multigrid hierarchy of `bytes` where `room` bytes are free.
extern "C" int imf_host_mg_affordable(unsigned long long bytes, unsigned long long room)
{
    return imf_to::mg_affordable((size_t)bytes, (size_t)room);
}

// Whether a batch takes the streamed minimum (erode_stream.h): the sharp offsets of its orientations one after another,
// count[o] of them each. cost gets the plan's loads of a thread per orientation, kind the orientations with runs along
// y and along z. Returns -1 where the plan refuses the points.
extern "C" int imf_host_stream_faster(const int *sh, const int *count, int n_orient, const int *K, int nx, int ny, int nz,
                                      int nsm, double *cost, int *kind)
{
    std::vector<std::vector<int32_t>> v;
    for (int o = 0; o < n_orient; sh += 3 * (size_t)count[o], ++o) v.emplace_back(sh, sh + 3 * (size_t)count[o]);
    std::vector<imf::EsOrient> h;
    std::vector<int> words;
    imf::EsGeometry g;
    if (!imf::es_plan(v, K, g, h, words)) return -1;
    kind[0] = kind[1] = 0;
    for (const imf::EsOrient &e : h)
        if (e.axis >= 0) ++kind[e.axis];
    *cost = g.cost;
    return imf::es_faster(g, nx, ny, nz, kind, n_orient, nsm);
}

// Whether a batch takes the sweep on staged tiles (sweep_plan.h): the cutter offsets of its orientations one after
// another, count[o] of them each. runs gets the plan's runs along x. Returns -1 where the plan refuses the cutter.
extern "C" int imf_host_sweep_faster(const int *rk, const int *count, int n_orient, const int *K, const int *kmin, int nx, int ny,
                                     int nz, int nsm, double *runs)
{
    std::vector<std::vector<int32_t>> v;
    for (int o = 0; o < n_orient; rk += 3 * (size_t)count[o], ++o) v.emplace_back(rk, rk + 3 * (size_t)count[o]);
    std::vector<imf::SwOrient> h;
    std::vector<int> words;
    imf::SwGeometry g;
    if (!imf::sw_plan(v, K, kmin, nx, g, h, words)) return -1;
    int kind[2] = {0, 0};
    for (const imf::SwOrient &e : h)
        if (e.axis >= 0) ++kind[e.axis];
    *runs = g.runs;
    return imf::sw_faster(g, nx, ny, nz, kind, n_orient, nsm);
}

// Pencils per item of the copy-fed y and z passes (fft_tma.cuh), negative where no launch is compiled for them.
extern "C" int imf_host_tma_pencils(int big, int ws, int wide)
{
    const int W = imf::tma_fft::pencils(big != 0, ws != 0, wide != 0);
    return imf::tma_fft::compiled(big != 0, ws != 0, W) ? W : -W;
}

// Feeds n launch results to a call's record; returns what the call reports with `last` as the runtime's final word, and
// in next what a following call without errors reports.
extern "C" int imf_host_launch_errors(const int *results, int n, int last, int *next)
{
    imf::LaunchErrors e;
    for (int i = 0; i < n; ++i) e.note((cudaError_t)results[i]);
    const int got = (int)e.take((cudaError_t)last);
    *next = (int)e.take(cudaSuccess);
    return got;
}
