// Plan of the streamed minimum over sharp points (erode_stream.cu): runs of sharp points along y
// or z per orientation, listed by the source plane they read. Shared by the library (imf_api.cu)
// and the CPU tests (hosttest.cu).
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <vector>

#include "erode.cuh"
#include "erode_stream.cuh"

namespace imf {

struct EsRun {
    int dx, du, dw, len;             // du: last offset of the run along its axis
};

// Runs (at most kEsMaxL long) along axis u (1 = y, 2 = z) of the points marked in the box `in`
// ([z][y][x], extents e, first offset mn); returns the window loads of one thread, kEsX + L - 1
// per run.
inline long es_runs(const std::vector<uint8_t> &in, const int e[3], const int mn[3], int u, std::vector<EsRun> *out)
{
    const int w = 3 - u;
    const long step[3] = {1, e[0], (long)e[0] * e[1]};
    long cost = 0;
    for (int iw = 0; iw < e[w]; ++iw)
        for (int ix = 0; ix < e[0]; ++ix) {
            const uint8_t *line = in.data() + iw * step[w] + ix;
            for (int i = 0, n = 0; i <= e[u]; ++i) {
                const bool on = i < e[u] && line[i * step[u]];
                n += on;
                if (n && (!on || n == kEsMaxL)) {
                    cost += kEsX + n - 1;
                    if (out) out->push_back({mn[0] + ix, mn[u] + i - (on ? 0 : 1), mn[w] + iw, n});
                    n = 0;
                }
            }
        }
    return cost;
}

// Plans a tool: `sh` = the sharp points (offset triples) of every orientation, K = kmax of its
// cutter offsets. Per orientation a header and its descriptor words: first where each list starts, then the lists. List m holds the runs that read
// source planes 4 m .. 4 m + 3 counted from the output's own first one: 16 bytes with the runs of
// each length, then the byte offsets of the runs from the output's place in plane 4 m, by length
// (lengths taken two or four at a time start at multiples of that). Returns false where no kernel instance has rows wide enough, too few stages
// fit or a length has too many runs: the tiled kernel (erode.cu) takes those.
inline bool es_plan(const std::vector<std::vector<int32_t>> &sh, const int K[3], EsGeometry &g,
                    std::vector<EsOrient> &head, std::vector<int> &words)
{
    const int n = (int)sh.size();
    std::vector<EsRun> runs;
    std::vector<int> first(n + 1, 0), top(3 * (size_t)n, 0);
    head.assign(n, EsOrient{});
    words.clear();
    int need = 0, eu = 0, with_points = 0;
    long loads = 0;
    std::vector<uint8_t> in;
    for (int o = 0; o < n; ++o) {
        EsOrient &h = head[o];
        h.axis = -1;
        first[o + 1] = (int)runs.size();
        const std::vector<int32_t> &v = sh[o];
        if (v.empty()) continue;
        int mn[3] = {1 << 30, 1 << 30, 1 << 30}, mx[3] = {-(1 << 30), -(1 << 30), -(1 << 30)}, e[3];
        for (size_t m = 0; m < v.size(); m += 3)
            for (int c = 0; c < 3; ++c) { mn[c] = std::min(mn[c], v[m + c]); mx[c] = std::max(mx[c], v[m + c]); }
        for (int c = 0; c < 3; ++c) e[c] = mx[c] - mn[c] + 1;
        if (!es_pitch(kEsTX + e[0] - 1 + 3) || e[1] > 128 || e[2] > 128) return false;
        in.assign((size_t)e[0] * e[1] * e[2], 0);
        for (size_t m = 0; m < v.size(); m += 3)
            in[((size_t)(v[m + 2] - mn[2]) * e[1] + (v[m + 1] - mn[1])) * e[0] + (v[m] - mn[0])] = 1;
        const long along_y = es_runs(in, e, mn, 1, nullptr), along_z = es_runs(in, e, mn, 2, nullptr);
        const int u = along_y <= along_z ? 1 : 2, w = 3 - u;
        es_runs(in, e, mn, u, &runs);
        loads += std::min(along_y, along_z);
        ++with_points;
        first[o + 1] = (int)runs.size();
        for (int c = 0; c < 3; ++c) top[3 * o + c] = mx[c];
        const int shift = (K[0] - mx[0]) & 3;                  // copies start at multiples of 4 columns
        h.axis = u == 1 ? 0 : 1;
        h.lists = (e[w] + 3) / 4;
        h.rows = kEsRows + e[u] - 1;
        h.quads = (kEsTX + e[0] - 1 + shift + 3) / 4;
        h.ox = K[0] - mx[0] - shift;
        h.ou = K[u] - mx[u];
        h.ow = K[w] - mx[w];
        need = std::max(need, 4 * h.quads);
        eu = std::max(eu, e[u] - 1);
    }
    g.cost = (double)loads / std::max(with_points, 1);
    g.P = es_pitch(need);
    g.R = kEsRows + eu;
    g.Q = g.R * g.P;
    while (g.Q % 32 != 8) g.Q += 4;                            // four planes of 8 columns: 32 banks
    if (!g.P) return false;
    std::vector<int> by_len[kEsMaxL + 1];
    for (int o = 0; o < n; ++o) {
        EsOrient &h = head[o];
        h.word0 = (int)words.size();
        if (h.axis < 0) continue;
        const int u = h.axis ? 2 : 1, w = 3 - u, *mx = &top[3 * o], shift = (K[0] - mx[0]) & 3;
        words.resize(words.size() + (h.lists + 3) / 4 * 4, 0);
        for (int m = 0; m < h.lists; ++m) {
            words[h.word0 + m] = (int)words.size() - h.word0;
            for (auto &b : by_len) b.clear();
            for (int r = first[o]; r < first[o + 1]; ++r) {
                const int k = mx[w] - runs[r].dw - 4 * m;      // plane of the list the run reads
                if (k < 0 || k >= 4) continue;
                by_len[runs[r].len].push_back(4 * (k * g.Q + (mx[u] - runs[r].du) * g.P + (mx[0] - runs[r].dx) + shift));
            }
            uint32_t count[4] = {0, 0, 0, 0};
            const size_t at = words.size();
            words.resize(at + 4, 0);
            for (int L = 1; L <= kEsMaxL; ++L) {
                std::vector<int> &b = by_len[L];
                if (b.size() > 255) return false;
                while (!b.empty() && words.size() % es_unroll(L)) words.push_back(0);
                count[(L - 1) / 4] |= (uint32_t)b.size() << (8 * ((L - 1) % 4));
                words.insert(words.end(), b.begin(), b.end());
            }
            for (int i = 0; i < 4; ++i) words[at + i] = (int)count[i];
            while (words.size() % 4) words.push_back(0);
        }
        h.words = (int)words.size() - h.word0;
        g.words = std::max(g.words, h.words);
    }
    const size_t slots = (size_t)kEsSlots * g.words * 4, stage = (size_t)16 * g.Q;
    if (slots > kEsBudget) return false;
    g.stages = (int)std::min<size_t>(kEsMaxStages, (kEsBudget - slots) / stage);
    return g.stages >= 3;
}

// Whether the streamed kernel takes a batch of nb orientations, kind[a] of them with runs along axis a, of a planned tool.
// Its time over the tiled kernel's follows, to 11 % over 208 measurements (grids 40^3 to 128^3 and flat and
// long ones, cutters of radius 1 to 11, 8 to 64 orientations),
//   sqrt(V) (0.715 + (1.14 + 2.1 min(1, 300 / cost)) / p):
// V is the volume of its tiles with their orientations over that of the tiled kernel's, p the pairs of a tile and an
// orientation an SM gets, cost the loads of a thread per orientation. Its blocks fill a ring before they reduce, which
// few pairs or cheap cutters do not pay for, and its tiles of 24 rows along z waste a flat grid. With the line at
// twelve tiles x orientations of either kind an SM alone (us, tiled and streamed): 200 x 100 x 8 x 16, radius 1, 40 and 64;
// 400 x 60 x 32 x 8, radius 1, 78 and 98; 200 x 100 x 8 x 32, radius 8, 690 and 766; 40^3 x 64, radius 2, 92 and 109.
// Chosen by this, at most 1.07 (558 and 597) in those measurements. Grids of one plane use an eighth of its
// tiles and stay with the tiled kernel.
inline bool es_faster(const EsGeometry &g, int nx, int ny, int nz, const int kind[2], int nb, int nsm)
{
    const EsTiles t = es_tile_counts(nx, ny, nz);
    const double pairs = (double)t.kind(0) * kind[0] + (double)t.kind(1) * kind[1];
    if (nz < 2 || !(pairs > 0) || (double)(t.kind(0) + t.kind(1)) * nb < 12.0 * nsm) return false;
    auto up = [](int n, int d) { return (double)((n + d - 1) / d); };
    const double tiled = up(nx, kErTX) * up(ny, kErTY) * up(nz, kErTZ) * nb;
    const double V = pairs * (kEsTX * kEsRows * kEsW) / (tiled * (kErTX * kErTY * kErTZ));
    return std::sqrt(V) * (0.715 + (1.14 + 2.1 * std::min(1.0, 300.0 / std::max(g.cost, 1.0))) * nsm / pairs) < 1.0;
}

} // namespace imf
