// Plan of the sweep on staged tiles (sweep_tile.cu): the cutter of an orientation as slices of equal x
// offset, each a set of runs along y or z. Shared by the library (imf_api.cu) and the CPU tests (hosttest.cu).
#pragma once
#include <algorithm>
#include <cmath>
#include <vector>

#include "sweep_tile.cuh"

namespace imf {

// rk = the cutter offsets (triples) of every orientation, K / kmin their largest and smallest, nx the grid's
// extent. Per orientation a header and descriptor words: per slice (whole-word shift falling) one word shift |
// bit shift << 8 | runs << 16, then per run its offset in the tile | length << 24. Returns false where the tile
// does not fit: the kernel on dilation levels takes those.
inline bool sw_plan(const std::vector<std::vector<int32_t>> &rk, const int K[3], const int kmin[3], int nx, SwGeometry &g,
                    std::vector<SwOrient> &head, std::vector<int> &words)
{
    const int n = (int)rk.size(), awords = (nx + 31) / 32;
    head.assign(n, SwOrient{});
    words.clear();
    g = SwGeometry{};
    g.somax = (K[0] - kmin[0]) >> 5;
    if (g.somax > 14) return false;
    // the words of a tile that leave the fewest lanes of a warp without an output
    double best_eff = 0;
    for (int q = 1; q <= std::min(awords, 31 - g.somax); ++q) {
        const int l = q + g.somax + 1, tiles = (awords + q - 1) / q;
        const double eff = (double)awords / tiles * (32 / l);
        if (eff > best_eff) {
            best_eff = eff;
            g.nq = q;
            g.nl = l;
            g.ppw = 32 / l;
        }
    }
    struct Run { int dx, du, dw, len; };
    std::vector<std::vector<Run>> runs(n);
    std::vector<int> top(3 * (size_t)n, 0);
    int eu = 0, ew = 0, with_cutter = 0;
    std::vector<uint8_t> in;
    for (int o = 0; o < n; ++o) {
        SwOrient &h = head[o];
        h.axis = -1;
        const std::vector<int32_t> &v = rk[o];
        if (v.empty()) continue;
        int mn[3] = {1 << 30, 1 << 30, 1 << 30}, mx[3] = {-(1 << 30), -(1 << 30), -(1 << 30)}, e[3];
        for (size_t m = 0; m < v.size(); m += 3)
            for (int c = 0; c < 3; ++c) { mn[c] = std::min(mn[c], v[m + c]); mx[c] = std::max(mx[c], v[m + c]); }
        for (int c = 0; c < 3; ++c) e[c] = mx[c] - mn[c] + 1;
        if (e[1] > 64 || e[2] > 64) return false;
        in.assign((size_t)e[0] * e[1] * e[2], 0);
        for (size_t m = 0; m < v.size(); m += 3)
            in[((size_t)(v[m + 2] - mn[2]) * e[1] + (v[m + 1] - mn[1])) * e[0] + (v[m] - mn[0])] = 1;
        ++with_cutter;
        for (size_t i = 0; i < in.size(); ++i) g.runs += in[i] && (i % e[0] == 0 || !in[i - 1]);
        const long step[3] = {1, e[0], (long)e[0] * e[1]};
        long best = 1L << 60;
        for (int u = 1; u <= 2; ++u) {
            const int w = 3 - u;
            std::vector<Run> r;
            long cost = 0;
            for (int ix = 0; ix < e[0]; ++ix)
                for (int iw = 0; iw < e[w]; ++iw) {
                    const uint8_t *line = in.data() + iw * step[w] + ix;
                    for (int i = 0, c = 0; i <= e[u]; ++i) {
                        const bool on = i < e[u] && line[i * step[u]];
                        c += on;
                        if (c && (!on || c == kSwMaxL)) {
                            cost += kSwX + c - 1;
                            r.push_back({mn[0] + ix, mn[u] + i - (on ? 0 : 1), mn[w] + iw, c});
                            c = 0;
                        }
                    }
                }
            if (cost < best) {
                best = cost;
                runs[o].swap(r);
                h.axis = u - 1;
                h.eu = e[u] - 1;
                h.ew = e[w] - 1;
                h.ou = K[u] - mx[u];
                h.ow = K[w] - mx[w];
                top[3 * o + 1] = mx[u];
                top[3 * o + 2] = mx[w];
            }
        }
        eu = std::max(eu, h.eu);
        ew = std::max(ew, h.ew);
        g.cost += best;
        g.stage += (double)(kSwRows + h.eu) * (g.ppw * kSwNP + h.ew) * g.nl;
    }
    for (double *v : {&g.cost, &g.stage, &g.runs}) *v /= std::max(with_cutter, 1);
    g.UP = (kSwRows + eu) | 1;
    g.planes = g.ppw * kSwNP + ew;
    for (int o = 0; o < n; ++o) {
        SwOrient &h = head[o];
        h.word0 = (int)words.size();
        if (h.axis < 0) continue;
        // slices by falling shift s = K - dx (words first), then by length inside a slice
        std::vector<Run> &r = runs[o];
        std::stable_sort(r.begin(), r.end(), [](const Run &a, const Run &b) { return a.dx != b.dx ? a.dx < b.dx : a.len < b.len; });
        for (size_t i = 0; i < r.size();) {
            size_t j = i;
            while (j < r.size() && r[j].dx == r[i].dx) ++j;
            const int s = K[0] - r[i].dx;
            words.push_back((s >> 5) | ((s & 31) << 8) | (int)(j - i) << 16);
            for (; i < j; ++i)
                words.push_back((top[3 * o + 2] - r[i].dw) * g.nl * g.UP + (top[3 * o + 1] - r[i].du) | r[i].len << 24);
        }
        h.words = (int)words.size() - h.word0;
        g.words = std::max(g.words, h.words);
    }
    g.smem = ((size_t)g.planes * g.nl * g.UP + g.words) * 4;
    return g.smem <= kSwMaxSmem;
}

// Whether the staged tiles take a batch of nb orientations, kind[a] of them with runs along axis a, of a planned tool.
// Both kernels' times, in us, to 13 and 10 % over 440 measurements (the grids, cutters and orientations named in
// erode_stream.h, 3 to 64 of these): the levels and their sweep pay for every output word and run along x, a
// staged block for its words, and for all its runs one after another, whose latency is the whole time where few
// blocks share an SM. Taken without this line (us, levels and staged): 40^3 x 3, radius 11 and length 30, 82 and 238;
// 200 x 100 x 8 x 64, radius 8, 153 and 265; 128^3 x 32, radius 11, 796 and 1195. Chosen by it, at most 1.22
// (398 and 485, 96^3 x 64 with radius 8) in those measurements, and 55 of 440 faster by up to 0.6.
inline bool sw_faster(const SwGeometry &g, int nx, int ny, int nz, const int kind[2], int nb, int nsm)
{
    const int awords = (nx + 31) / 32, tp = g.ppw * kSwNP;
    auto up = [](int n, int d) { return (double)((n + d - 1) / d); };
    const double words = (double)awords * ny * nz * nb / nsm;
    const double blocks = up(awords, g.nq) * (kind[0] * up(ny, kSwRows) * up(nz, tp) + kind[1] * up(nz, kSwRows) * up(ny, tp)) / nsm;
    const double bps = std::min(8.0, std::floor(227.0 * 1024 / (g.smem + 1024)));
    const double levels = 6.8 + 0.105 * g.runs + words * (0.00098 + 0.000188 * std::pow(g.runs, 0.878) * (1 + 0.66 / awords));
    const double staged = 10.4 + 0.082 * std::pow(g.cost, 0.8136) +
                          std::max(0.0, blocks - 1) * (0.52 + 0.00367 * g.cost * (1 + 0.9 / bps) + 0.0009 * g.stage);
    return staged < 0.95 * levels;
}

} // namespace imf
