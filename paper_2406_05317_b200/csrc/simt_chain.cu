// The backward pass of a group of chunks in fp32, the part that is a chain: from the gradient w.r.t. the cache after each compress
// step to the one before it. All that the chain needs of the convolution and the attention is there before it starts; what only
// this chunk's rows and the weights need comes after it (simt_backward.cu). Per step, for the M rows of the cache alone,
//   dw = gK X_K^T + gV X_V^T (positions 0 .. c + pad),  <dw_i, w_i> = g_i . (row i of the new cache),  dA = [R > 0] (dw - <dw, w>) / s
//   g' = attention's share + sum over slots of (R / s)^T g + dA (*) G
//
// A cluster of 1 to 16 CTAs of 512 threads owns one unit; a CTA owns some of its slots: their g, their rows of R and their weights stay
// in its shared memory. The contraction of g' runs over slots, so every CTA makes partial rows for all of the cache and writes each
// into the shared memory of the CTA that owns it; after a cluster barrier the owner adds them up in a fixed order. Rows of the next step are
// on their way meanwhile. Bound: latencies, as in the forward loop (simt_loop.cu).
// 8 units, M = 48, d = 64, k = 5 in clusters of ten: 4.2 us per step; with one round of tiles per warp of 32 lanes, four positions per
// thread and the fetch ahead of everything 6.6.
#include <algorithm>
#include <type_traits>

#include "backward.h"
#include "handle.h"
#include "simt.cuh"

namespace lococo {
namespace {

using namespace simt;

constexpr int kThreads = 512, kWarps = kThreads / 32;
constexpr int kMaxSmem = 232448 - 128;
constexpr int kShareWarps = 12;          // make a CTA's share of g'; the others fetch
constexpr int kTA = 3, kTP = 4;          // slots x positions of a tile of dw: with the three <dw, w>, fifteen sums over the lanes

__host__ __device__ inline int round4(int x) { return (x + 3) / 4 * 4; }
// Shared memory, in floats. Rows of 2 d channels (keys, then values) lie 2 d + 4 apart.
struct ChainLayout {
    int rows, RR, DR, slots;             // rows of X; row strides of R and of dA (position j at pad + j); slots per CTA
    int w, x, r, kn, at, s, g, da, recv, owner, total;
};
__host__ __device__ inline ChainLayout chain_layout(int d, int M, int k, int c_in, int ctas) {
    ChainLayout l;
    const int pad = (k - 1) / 2, row = 2 * d + 4;
    l.slots = (M + ctas - 1) / ctas;
    l.rows = round4(M + pad);
    l.RR = round4(M + pad) + 4;
    l.DR = round4(round4(M) + k - 1 + 4);
    int off = 0;
    l.w = off;     off += l.slots * k * c_in;
    l.x = off;     off += 2 * l.rows * row;
    l.r = off;     off += 2 * l.slots * l.RR;
    l.kn = off;    off += 2 * l.slots * row;
    l.at = off;    off += 2 * l.slots * row;
    l.s = off;     off += 2 * round4(l.slots);
    l.g = off;     off += l.slots * row;
    l.da = off;    off += l.slots * l.DR;
    l.recv = off;  off += 2 * ctas * l.slots * 2 * d;
    l.owner = off; off += round4(M);
    l.total = off;
    return l;
}

template <int D>
__global__ void __launch_bounds__(kThreads, 1) chain_kernel(const __grid_constant__ BwdGroup G) {
    extern __shared__ __align__(16) float smem[];
    constexpr int kQ = D / 2, RS = 2 * D + 4;                     // quads of channels per row [keys | values]
    const BwdStep& F = G.first;
    const int ctas = G.ctas, rank = blockIdx.x % ctas, u = blockIdx.x / ctas, n = u / F.heads, h = u % F.heads;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int M = F.M, k = F.k, C = F.c_in, pad = (k - 1) / 2;
    const int i_begin = M * rank / ctas, slots = M * (rank + 1) / ctas - i_begin;
    const ChainLayout lay = chain_layout(D, M, k, C, ctas);
    float *Ws = smem + lay.w, *gs = smem + lay.g, *dAs = smem + lay.da;
    auto Xs = [&](int b) { return smem + lay.x + b * lay.rows * RS; };
    auto Rs = [&](int b) { return smem + lay.r + b * lay.slots * lay.RR; };
    auto Kn = [&](int b) { return smem + lay.kn + b * lay.slots * RS; };
    auto At = [&](int b) { return smem + lay.at + b * lay.slots * RS; };
    auto Ss = [&](int b) { return smem + lay.s + b * round4(lay.slots); };
    auto cache_before = [&](int nn) { return min(M, G.c0 + nn * G.B); };
    auto chunk_rows = [&](int nn) { return min(G.B, G.L - nn * G.B); };
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (int x = tid; x < lay.slots * lay.DR; x += kThreads) dAs[x] = 0.f;
    // where this CTA's share of row j goes (in the first of the two receive buffers of the CTA that owns the row)
    uint32_t* owner = reinterpret_cast<uint32_t*>(smem + lay.owner);
    for (int j = tid; j < M; j += kThreads) {
        const int to = ((j + 1) * ctas - 1) / M;
        owner[j] = remote((uint32_t)__cvta_generic_to_shared(smem + lay.recv + (rank * lay.slots + j - M * to / ctas) * 2 * D), to);
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");

    const int row0 = tid / kQ, ch0 = 4 * (tid % kQ), ch = ch0 < D ? ch0 : ch0 - D;      // a thread has the same channels of every kStep-th row
    constexpr int kStep = kThreads / kQ;
    // Rows of step G.n0 + i into buffers b: X (cache, and as far into the chunk as the convolution reaches), own rows of R, of the
    // attention's share and of the cache after the step. By `threads` threads (a multiple of kQ); this is thread t of them.
    const float* snap_base = reinterpret_cast<const float*>((ch0 < D ? F.xk : F.xv).cache.ptr) + (int64_t)u * M * D + ch;
    const float* chunk_base = unit_base<float>((ch0 < D ? F.xk : F.xv).chunk, n, h) + ch;
    const int64_t chunk_st = (ch0 < D ? F.xk : F.xv).chunk.st;
    auto fetch = [&](int i, int b, int t, int threads) {
        const int nn = G.n0 + i, c = cache_before(nn), S = c + chunk_rows(nn), first = t / kQ, step = threads / kQ;
        const float* snap = snap_base + nn * G.snap_step;
        if (S > M) {
            const float* src = chunk_base + (int64_t)nn * G.B * chunk_st;
            float* dst = Xs(b) + ch0;
            for (int j = first; j < c; j += step) cp_async16(dst + j * RS, snap + j * D, true);
            for (int j = c + first; j < lay.rows; j += step) cp_async16(dst + j * RS, j < S ? src + (j - c) * chunk_st : snap, j < S);
            const float* r = G.R + ((int64_t)i * G.splits * F.units + u) * M * G.Sr + (int64_t)i_begin * G.Sr;
            for (int a = t >> 5; a < slots; a += threads >> 5)
                for (int j = 4 * (t & 31); j < lay.rows; j += 128) cp_async16(Rs(b) + a * lay.RR + j, j < G.Sr ? r + (int64_t)a * G.Sr + j : r, j < G.Sr);
            const bool final_cache = nn * G.B + G.B >= G.L;
            const float* next = final_cache ? G.last + ((int64_t)u * M + i_begin) * (2 * D) + ch0 : snap + G.snap_step + i_begin * D;
            for (int a = first; a < slots; a += step) cp_async16(Kn(b) + a * RS + ch0, next + a * (final_cache ? 2 * D : D), true);
            for (int a = t; a < slots; a += threads) Ss(b)[a] = G.s[((int64_t)i * F.units + u) * M + i_begin + a];
        }
        const float* at = G.attn + ((int64_t)i * F.units * G.S + (int64_t)u * S + i_begin) * (2 * D) + ch0;
        for (int a = first; a < slots; a += step) {
            const bool live = i_begin + a < c;
            cp_async16(At(b) + a * RS + ch0, live ? at + a * (2 * D) : G.attn, live);
        }
        cp_async_commit();
    };
    fetch(G.count - 1, (G.count - 1) & 1, tid, kThreads);
    {
        const float* w = reinterpret_cast<const float*>(F.g_reverse) + ((int64_t)(F.weights_per_head ? h * M : 0) + i_begin) * k * C;
        for (int x = tid; x < slots * k * C / 4; x += kThreads) cp_async16(Ws + 4 * x, w + 4 * x, true);
        cp_async_commit();
    }
    // g: the caller's gradient w.r.t. the final cache, or what the group behind this one left
    const bool first = (G.n0 + G.count) * (int64_t)G.B >= G.L;
    const int64_t g_step = (int64_t)F.units * M * 2 * D, g_row = ((int64_t)u * M + i_begin) * (2 * D) + ch0;      // between steps; this thread's channels of row i_begin
    for (int a = row0; a < slots; a += kStep) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (first) {
            const View& f = ch0 < D ? G.gk_final : G.gv_final;
            if (f.ptr) v = load4(unit_base<float>(f, n, h) + (int64_t)(i_begin + a) * f.st + ch);
        } else {
            v = load4((ch0 < D ? G.gK : G.gV) + ((int64_t)u * M + i_begin + a) * D + ch);
        }
        store4(gs + a * RS + ch0, v);
        store4(G.g + G.count * g_step + g_row + (int64_t)a * (2 * D), v);
    }
    cp_async_wait<0>();
    if (ctas > 1) cluster_sync();
    else __syncthreads();
    int exchanged = 0;                   // compress steps so far
#pragma unroll 1
    for (int i = G.count - 1; i >= 0; --i) {
        const int b = i & 1, nn = G.n0 + i, c = cache_before(nn), S = c + chunk_rows(nn);
        const bool compress = S > M;
        if (compress) {
            // ---- dw, <dw, w>, dA of this CTA's slots: two tiles per warp, every sixteenth quad of channels per lane. (Zeros behind a
            // short chunk; with no cache and no padding one round of tiles all the same, for <dw, w>.)
            const int it = (slots + kTA - 1) / kTA, positions = min(c + pad, S), jt = max(1, (c + pad + kTP - 1) / kTP), tiles = it * jt;
            const uint32_t magic = 0xffffffffu / jt + 1;                       // t / jt = the upper half of t magic (jt > 1)
#pragma unroll 1
            for (int t0 = 2 * warp; t0 < tiles; t0 += 2 * kWarps) {
                const int t = min(t0 + (lane >> 4), tiles - 1), ti = jt == 1 ? t : __umulhi(t, magic), a0 = kTA * ti, j0 = kTP * (t - ti * jt);
                const float *x = Xs(b) + j0 * RS + 4 * (lane & 15), *gr = gs + 4 * (lane & 15), *kr = Kn(b) + 4 * (lane & 15);
                int row[kTA];
#pragma unroll
                for (int a = 0; a < kTA; ++a) row[a] = min(a0 + a, slots - 1) * RS;
                f32x2 acc[kTA][kTP + 1];
#pragma unroll
                for (int a = 0; a < kTA; ++a)
#pragma unroll
                    for (int p = 0; p <= kTP; ++p) acc[a][p] = 0ull;
#pragma unroll
                for (int q = 0; q < kQ / 16; ++q) {
                    f32x4 z[kTP];
#pragma unroll
                    for (int p = 0; p < kTP; ++p) z[p] = load_pairs(x + p * RS + 64 * q);
#pragma unroll
                    for (int a = 0; a < kTA; ++a) {
                        const f32x4 g = load_pairs(gr + row[a] + 64 * q), kn = load_pairs(kr + row[a] + 64 * q);
#pragma unroll
                        for (int p = 0; p < kTP; ++p) { fma2(g.lo, z[p].lo, acc[a][p]); fma2(g.hi, z[p].hi, acc[a][p]); }
                        fma2(g.lo, kn.lo, acc[a][kTP]);
                        fma2(g.hi, kn.hi, acc[a][kTP]);
                    }
                }
                float v[16];
                v[15] = 0.f;
#pragma unroll
                for (int a = 0; a < kTA; ++a) {
#pragma unroll
                    for (int p = 0; p < kTP; ++p) { const float2 f = unpair(acc[a][p]); v[kTP * a + p] = f.x + f.y; }
                    const float2 f = unpair(acc[a][kTP]);
                    v[kTA * kTP + a] = f.x + f.y;
                }
                reduce_lanes<16, 16>(v, lane & 15);
                const int idx = lane & 15, a = min(idx / kTP, kTA - 1), j = j0 + idx % kTP;
                const float inner = __shfl_sync(0xffffffffu, v[0], (lane & 16) + kTA * kTP + a);
                if (idx < kTA * kTP && a0 + a < slots) {
                    const int slot = i_begin + a0 + a;
                    const float inv = 1.f / Ss(b)[a0 + a];
                    // (a protected slot's row has no gradient)
                    dAs[(a0 + a) * lay.DR + pad + j] = j < positions && slot >= G.prot && Rs(b)[(a0 + a) * lay.RR + j] > 0.f ? (v[0] - inner) * inv : 0.f;
                    if (j == 0) G.inner[((int64_t)i * F.units + u) * M + slot] = inner;
                }
            }
            __syncthreads();
            // ---- this CTA's share of all rows of g': two positions x four channels per thread, first the channels that the
            // convolution reaches; beside it the last four warps ask for the next step's rows
            if (warp >= kShareWarps) {
                if (i > 0) fetch(i - 1, b ^ 1, tid - 32 * kShareWarps, 32 * (kWarps - kShareWarps));
            } else {
                const uint32_t parity = (exchanged & 1) * ctas * lay.slots * 2 * D * 4;
                auto share = [&](auto conv_quads, auto first_quad, auto quads) {
                    constexpr bool kConv = decltype(conv_quads)::value;
                    constexpr int kFirst = decltype(first_quad)::value, kPer = decltype(quads)::value;
#pragma unroll 1
                    for (int x = tid; x < (c + 1) / 2 * kPer; x += 32 * kShareWarps) {
                        const int q = kFirst + x % kPer, j0 = 2 * (x / kPer);
                        f32x4 acc0{0ull, 0ull}, acc1{0ull, 0ull};
                        const float *w = Ws + 4 * q, *da = dAs + j0, *r = Rs(b) + j0, *g = gs + 4 * q;
#pragma unroll 1
                        for (int a = 0; a < slots; ++a, r += lay.RR, g += RS, da += lay.DR) {
                            const float inv = 1.f / Ss(b)[a];
                            const float2 rr = *reinterpret_cast<const float2*>(r);
                            const f32x4 gq = load_pairs(g);
                            fma4(pair(rr.x * inv, rr.x * inv), gq, acc0);
                            fma4(pair(rr.y * inv, rr.y * inv), gq, acc1);
                            if (kConv) {
                                f32x2 z0 = pair(da[0], da[0]);
#pragma unroll 4
                                for (int t = 1; t <= k; ++t, w += C) {
                                    const f32x2 z1 = pair(da[t], da[t]);
                                    const f32x4 wt = load_pairs(w);
                                    fma4(z0, wt, acc0);
                                    fma4(z1, wt, acc1);
                                    z0 = z1;
                                }
                            }
                        }
#pragma unroll
                        for (int p = 0; p < 2; ++p) {
                            if (j0 + p >= c) break;
                            const float4 v = to_float4(p ? acc1 : acc0);
                            st_remote(owner[j0 + p] + parity + 16 * q, make_uint4(__float_as_uint(v.x), __float_as_uint(v.y), __float_as_uint(v.z), __float_as_uint(v.w)));
                        }
                    }
                };
                using Zero = std::integral_constant<int, 0>;
                if (C == D) {
                    share(std::true_type{}, Zero{}, std::integral_constant<int, kQ / 2>{});
                    share(std::false_type{}, std::integral_constant<int, kQ / 2>{}, std::integral_constant<int, kQ / 2>{});
                } else {
                    share(std::true_type{}, Zero{}, std::integral_constant<int, kQ>{});
                }
            }
        } else if (i > 0) {
            fetch(i - 1, b ^ 1, tid, kThreads);
        }
        cp_async_wait<0>();
        if (ctas > 1 && compress) cluster_sync();
        else __syncthreads();
        // ---- the rows of g' that this CTA owns
        const float* recv = smem + lay.recv + (exchanged & 1) * ctas * lay.slots * 2 * D;
        if (compress) ++exchanged;
        for (int a = row0; a < slots; a += kStep) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (i_begin + a < c) {                                             // (rows that the cache did not have before get none)
                v = compress ? make_float4(0.f, 0.f, 0.f, 0.f) : load4(gs + a * RS + ch0);
                if (compress) {
#pragma unroll 4
                    for (int r = 0; r < ctas; ++r) {
                        const float4 w = load4(recv + (r * lay.slots + a) * 2 * D + ch0);
                        v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
                    }
                }
                const float4 w = load4(At(b) + a * RS + ch0);
                v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
            }
            store4(gs + a * RS + ch0, v);
            store4(G.g + i * g_step + g_row + (int64_t)a * (2 * D), v);
            if (i == 0) store4((ch0 < D ? G.gK : G.gV) + ((int64_t)u * M + i_begin + a) * D + ch, v);
        }
        __syncthreads();
    }
    if (ctas > 1) cluster_sync();        // (nobody leaves while others may still write to it)
}

ClusterKernel chain_state[2];

// CTAs per unit (0: none fits) by the fewest estimated microseconds per step, and how many of these are not the step's work spread over all SMs.
// resident[ctas]: how many clusters of that many CTAs run at once.
struct ChainPlan { int ctas; double us, idle_us; };
template <typename Count>
ChainPlan chain_plan(int units, int M, int d, int k, int c_in, const Count* resident) {
    ChainPlan best{0, 1e30, 0};
    for (int ctas = 1; resident && ctas <= std::min(kMaxCluster, M); ctas = next_cluster(ctas)) {
        const ChainLayout lay = chain_layout(d, M, k, c_in, ctas);
        if ((double)lay.slots * k * c_in * 4 > kMaxSmem || (size_t)lay.total * 4 > kMaxSmem) continue;
        const int clusters = resident[ctas];
        if (clusters == 0) continue;
        const double per_slot = (double)M * (4.0 * d + (double)c_in * k) / 90e3;
        const double us = (units + clusters - 1) / clusters * (2.0 + 0.03 * ctas + lay.slots * per_slot);
        if (us < best.us) best = {ctas, us, us - per_slot * M * units / kSMs};
    }
    return best;
}

}  // namespace

// What a group saves is the latency of a step's four launches, about 28 us; what it costs is the chip's time while units wait for others' clusters or
// for one another's rows, and the attention's blocks (per SM) no longer hide anything where they alone fill the chip. The weights are a
// least-squares fit to 78 sizes (6 us per step off). d = 128, B = 100, a training step in groups / a step at a time, us: 32 units, M = 32, k = 5
// 560 / 643; 96, M = 16 1029 / 1047; 24, M = 32, k = 11 612 / 667, 48 1083 / 984; 16, M = 48, k = 5 497 / 527, 32 830 / 781, 96 2178 / 1706.
static bool group_pays(const ChainPlan& plan, int units, int M, int B, int d) {
    const int attention_blocks = ((M + B + 31) / 32 + (B + 31) / 32) * units;
    return plan.ctas > 0 && 1.9 * plan.idle_us + 4.6 * attention_blocks / kSMs * d / 128 <= 28.0;
}
int simt_group_clusters(const BwdGroup& G) {
    const BwdStep& p = G.first;
    const std::atomic<int>* resident = p.d == 128 ? resident_clusters(chain_state[1], chain_kernel<128>, kMaxSmem, kThreads)
                                     : resident_clusters(chain_state[0], chain_kernel<64>, kMaxSmem, kThreads);
    const ChainPlan plan = chain_plan(p.units, p.M, p.d, p.k, p.c_in, resident);
    return group_pays(plan, p.units, p.M, G.B, p.d) ? plan.ctas : 0;
}
bool simt_group_possible(const lococo_handle* h, int B) {
    const lococo_config& c = h->cfg;
    int most[kMaxCluster + 1];
    for (int ctas = 1; ctas <= kMaxCluster; ++ctas) most[ctas] = kSMs / ctas;
    return group_pays(chain_plan(h->units, c.M, c.head_dim, c.k, c.c_in, most), h->units, c.M, B, c.head_dim);
}

int simt_backward_chain(const BwdGroup& G, cudaStream_t st) {
    const BwdStep& p = G.first;
    const size_t smem = (size_t)chain_layout(p.d, p.M, p.k, p.c_in, G.ctas).total * 4;
    return (p.d == 128 ? launch_clusters(chain_state[1], chain_kernel<128>, kMaxSmem, G.ctas, p.units, kThreads, smem, st, G)
                       : launch_clusters(chain_state[0], chain_kernel<64>, kMaxSmem, G.ctas, p.units, kThreads, smem, st, G)) ? 1 : -1;
}

}  // namespace lococo
