// What the CUDA-core backward pass lays out in the caller's scratch for groups of chunks, group by group, on a machine without a GPU
// (linked with the library's objects and fake_runtime.c).
#include <algorithm>
#include <utility>
#include <vector>

#include "backward.h"
#include "handle.h"

using namespace lococo;

// Floats that the groups of a call of L tokens in chunks of B, where there is room for `room` floats, take beyond what is reserved for them:
// the most of any group (0: all fit; -1: no groups at these sizes; -2: two arrays overlap). *chunks: of a whole group.
extern "C" long long fake_group_overrun(const lococo_config* cfg, int L, int B, size_t room, int* chunks) {
    lococo_handle* h = nullptr;
    if (lococo_create(cfg, &h) != LOCOCO_OK) return -3;
    size_t floats = 0;
    const int most = simt_group_chunks(h, L, B, room, &floats), units = h->units;
    lococo_destroy(h);
    *chunks = most;
    if (most == 0) return -1;
    BwdGroup G{};
    BwdStep& p = G.first;
    p.units = units; p.heads = cfg->heads; p.d = cfg->head_dim; p.M = cfg->M; p.k = cfg->k; p.c_in = cfg->c_in;
    G.L = L; G.B = std::min(B, L);
    G.S = p.M + G.B; G.Sr = (G.S + 3) / 4 * 4;
    float* base = reinterpret_cast<float*>(4096);
    const long long rows = (long long)units * p.M, d2 = 2 * p.d;
    long long worst = 0;
    for (int n = (L + B - 1) / B; n > 0; n -= G.count) {
        G.count = std::min(n, most);
        G.n0 = n - G.count;
        simt_group_layout(G, base, floats);
        std::vector<std::pair<float*, long long>> arrays = {
            {G.attn, (long long)G.count * units * G.S * d2}, {G.R, G.count * (long long)G.splits * rows * G.Sr}, {G.dA, G.count * rows * G.Sr},
            {G.g, (G.count + 1) * rows * d2}, {G.last, rows * d2}, {G.s, G.count * rows}, {G.inner, G.count * rows}};
        std::sort(arrays.begin(), arrays.end());
        for (size_t i = 0; i + 1 < arrays.size(); ++i)
            if (arrays[i].first + arrays[i].second > arrays[i + 1].first) return -2;
        worst = std::max(worst, (long long)(arrays.back().first + arrays.back().second - base) - (long long)floats);
    }
    return worst;
}
