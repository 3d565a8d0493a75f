// The backward pass of one step of Algorithm 2 on the CUDA cores, in fp32 (storage type float, or bf16 under
// LOCOCO_PATH_SIMT). Four launches:
//   1. what depends on nothing else of the step, side by side: the attention gradient (Eq. 1 reversed: dQ, and the keys' and
//      values' share of dX into a part of its own), the forward's convolution recomputed (Eq. 6, partial sums), and
//      dw = gK X_K^T + gV X_V^T
//   2. row by row: R = bias and ReLU of the convolution, the denominators s, dA = [R > 0] (dw - <dw, w>) / s
//   3. dX's compress share, w^T g + dA (*) G, as one or more partial sums, and dG += dA (*) Z beside it
//   4. the parts of dX are added: rows of the cache become the gradient handed to the step before, rows of the chunk dK, dV
// A fill step has 1 (attention only) and 4. No sum of several blocks meets in memory except dG's and dbias's.
#include <algorithm>

#include "backward.h"
#include "handle.h"
#include "simt.cuh"

namespace lococo {
namespace {

using namespace simt;

// ------------------------------------------------------------------ Eq. 1 reversed
// A block of 256 threads owns 32 rows of one side (kKeys: keys, else queries); its two groups of 128 take every other tile of
// 32 rows of the other and add up at the end:
//   s = F1 S1^T, dp = F2 S2^T     (F1, S1: keys and queries; F2, S2: values and output gradients)
//   p = exp(scale s - lse), ds = scale p (dp - delta)     under the causal mask
//   dF1 += ds S1,  dF2 += p S2 (keys' side only)
// A thread computes 4 x 2 scores and 4 rows x D/16 channels of each gradient. The next tile is on its way while one is computed
// (fp32: asynchronous copies into the other of two stages).
template <int D>
struct GradSmem {
    static constexpr int kRow = D + 4;
    static constexpr int kTile = 32 * kRow;
    static constexpr int kStage = 2 * kTile + 2 * 32;                 // streamed rows, and lse and delta of queries
    static constexpr int kGroup = 2 * kStage + 2 * 32 * 36;           // two stages
    static constexpr int kFloats = 2 * kTile + 2 * kGroup;
};

template <typename T, int D, bool kKeys>
__device__ __forceinline__ void attention_grad(const BwdStep& p, float* dx_attn, float* smem, int tile, int u) {
    constexpr int RS = GradSmem<D>::kRow, NC = D / 64;
    const int group = threadIdx.x >> 7;
    float *F1 = smem, *F2 = F1 + GradSmem<D>::kTile, *stages = F2 + GradSmem<D>::kTile + group * GradSmem<D>::kGroup;
    float *Ds = stages + 2 * GradSmem<D>::kStage, *Ps = Ds + 32 * 36;        // [32 fixed rows][32 streamed rows], row stride 36
    const int n = u / p.heads, h = u % p.heads;
    const int tid = threadIdx.x & 127, ts = tid & 15, tf = tid >> 4;
    const int f0 = tile * 32;
    const float sc2 = p.scale * 1.4426950408889634f;
    // rows r0 .. r0 + 31 of the queries and their output gradients, or of the keys and values; rows past the end are zeros
    auto stage = [&](bool keys, int r0, float* a, float* b, int first, int threads) {
        for (int e = first; e < 32 * (D / 4); e += threads) {
            const int r = e / (D / 4), q4 = e % (D / 4), row = r0 + r;
            const bool live = row < (keys ? p.S : p.b);
            const T* va = live ? (keys ? cat_row<T>(p.xk, n, h, row) : unit_base<T>(p.q, n, h) + (int64_t)row * p.q.st) + 4 * q4 : unit_base<T>(p.q, n, h);
            const T* vb = live ? (keys ? cat_row<T>(p.xv, n, h, row) : unit_base<T>(p.d_o, n, h) + (int64_t)row * p.d_o.st) + 4 * q4 : unit_base<T>(p.q, n, h);
            if constexpr (sizeof(T) == 4) {
                cp_async16(a + r * RS + 4 * q4, va, live);
                cp_async16(b + r * RS + 4 * q4, vb, live);
            } else {
                const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
                *reinterpret_cast<float4*>(a + r * RS + 4 * q4) = live ? load4(va) : zero;
                *reinterpret_cast<float4*>(b + r * RS + 4 * q4) = live ? load4(vb) : zero;
            }
        }
    };
    auto stage_vectors = [&](int r0, float* to) {      // lse, delta
        if (tid < 64) {
            const int r = r0 + (tid & 31);
            const float* src = tid < 32 ? p.lse + (int64_t)u * p.lse_stride : p.delta + (int64_t)u * p.delta_stride;
            cp_async4(to + tid, r < p.b ? src + r : src, r < p.b);
        }
    };
    stage(kKeys, f0, F1, F2, threadIdx.x, 256);
    if (!kKeys) stage_vectors(f0, stages + 2 * GradSmem<D>::kTile);
    f32x4 g1[4][NC], g2[4][NC];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int c = 0; c < NC; ++c) g1[a][c] = g2[a][c] = f32x4{0ull, 0ull};
    // streamed rows that meet the fixed ones: queries from the first that sees key f0, keys up to the last query's limit
    const int s_begin = kKeys ? max(0, f0 - p.c) / 32 * 32 : 0;
    const int s_end = kKeys ? p.b : p.c + min(f0 + 31, p.b - 1) + 1;
    auto stream = [&](int s0, int which) {
        float* to = stages + which * GradSmem<D>::kStage;
        stage(!kKeys, s0, to, to + GradSmem<D>::kTile, tid, 128);
        if (kKeys) stage_vectors(s0, to + 2 * GradSmem<D>::kTile);
    };
    const int s_first = s_begin + 32 * group;
    if (s_first < s_end) stream(s_first, 0);
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    int at = 0;
#pragma unroll 1
    for (int s0 = s_first; s0 < s_end; s0 += 64, at ^= 1) {
        if (s0 > s_first) {
            cp_async_wait<0>();
            group_sync(1 + group);                                  // this tile is there, and nobody reads the other stage any more
        }
        if (s0 + 64 < s_end) {
            stream(s0 + 64, at ^ 1);
            cp_async_commit();
        }
        const float *S1 = stages + at * GradSmem<D>::kStage, *S2 = S1 + GradSmem<D>::kTile;
        const float *lse_s = (kKeys ? S1 : stages) + 2 * GradSmem<D>::kTile, *delta_s = lse_s + 32;      // of the 32 queries at hand
        f32x2 s2[4][2], dp2[4][2];                                  // sums over the even and over the odd channels
#pragma unroll
        for (int a = 0; a < 4; ++a) s2[a][0] = s2[a][1] = dp2[a][0] = dp2[a][1] = 0ull;
        auto scores = [&](const float* fixed, const float* streamed, int d4, f32x2 (&acc)[4][2]) {
            f32x4 f[4], w[2];
#pragma unroll
            for (int b = 0; b < 2; ++b) w[b] = load_pairs(streamed + (ts + 16 * b) * RS + 4 * d4);
#pragma unroll
            for (int a = 0; a < 4; ++a) f[a] = load_pairs(fixed + (4 * tf + a) * RS + 4 * d4);
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 2; ++b) { fma2(f[a].lo, w[b].lo, acc[a][b]); fma2(f[a].hi, w[b].hi, acc[a][b]); }
        };
#pragma unroll 2
        for (int d4 = 0; d4 < D / 4; ++d4) {
            scores(F1, S1, d4, s2);
            scores(F2, S2, d4, dp2);
        }
        float s[4][2], dp[4][2];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const float2 x = unpair(s2[a][b]), y = unpair(dp2[a][b]);
                s[a][b] = x.x + x.y;
                dp[a][b] = y.x + y.y;
            }
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const int fr = 4 * tf + a, sr = ts + 16 * b;
                const int key = kKeys ? f0 + fr : s0 + sr, query = kKeys ? s0 + sr : f0 + fr, q = kKeys ? sr : fr;
                const float pr = (key < p.S && query < p.b && key <= p.c + query) ? exp2f(fmaf(s[a][b], sc2, -1.4426950408889634f * lse_s[q])) : 0.f;
                Ds[fr * 36 + sr] = pr * (dp[a][b] - delta_s[q]) * p.scale;
                if (kKeys) Ps[fr * 36 + sr] = pr;
            }
        group_sync(1 + group);
#pragma unroll 1
        for (int k4 = 0; k4 < 8; ++k4) {
            float4 ds[4], pr[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                ds[a] = *reinterpret_cast<const float4*>(Ds + (4 * tf + a) * 36 + 4 * k4);
                if (kKeys) pr[a] = *reinterpret_cast<const float4*>(Ps + (4 * tf + a) * 36 + 4 * k4);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e)
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    auto add = [&](const float* rows, const float4 (&w)[4], f32x4 (&g)[4][NC]) {
                        const f32x4 v = load_pairs(rows + (4 * k4 + e) * RS + 64 * c + 4 * ts);
#pragma unroll
                        for (int a = 0; a < 4; ++a) {
                            const float x = e == 0 ? w[a].x : e == 1 ? w[a].y : e == 2 ? w[a].z : w[a].w;
                            fma4(pair(x, x), v, g[a][c]);
                        }
                    };
                    add(S1, ds, g1);
                    if (kKeys) add(S2, pr, g2);
                }
        }
    }
    // the second group's sums through its own buffers
    group_sync(1 + group);
    float *G1 = F2 + GradSmem<D>::kTile + GradSmem<D>::kGroup, *G2 = G1 + GradSmem<D>::kTile;      // (its stages)
    if (group == 1) {
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                *reinterpret_cast<float4*>(G1 + (4 * tf + a) * RS + 64 * c + 4 * ts) = to_float4(g1[a][c]);
                if (kKeys) *reinterpret_cast<float4*>(G2 + (4 * tf + a) * RS + 64 * c + 4 * ts) = to_float4(g2[a][c]);
            }
    }
    __syncthreads();
    if (group == 1) return;
    auto plus = [](const f32x4& a, const float* b) {
        const float4 x = to_float4(a), y = *reinterpret_cast<const float4*>(b);
        return make_float4(x.x + y.x, x.y + y.y, x.z + y.z, x.w + y.w);
    };
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const int row = f0 + 4 * tf + a;
        if (row >= (kKeys ? p.S : p.b)) continue;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const int at = (4 * tf + a) * RS + 64 * c + 4 * ts;
            if (kKeys) {
                float* dst = dx_attn + ((int64_t)u * p.S + row) * (2 * D) + 64 * c + 4 * ts;
                store4(dst, plus(g1[a][c], G1 + at));
                store4(dst + D, plus(g2[a][c], G2 + at));
            } else {
                store4(unit_base_mut<T>(p.dq, n, h) + (int64_t)row * p.dq.st + 64 * c + 4 * ts, plus(g1[a][c], G1 + at));
            }
        }
    }
}

// ------------------------------------------------------------------ dw
// dw[u][i][j] = <gK[u][i], XK[j]> + <gV[u][i], XV[j]>: 64 slots x 64 positions per group of 128 threads (8 x 4 each), sixteen
// channels per stage, both operands transposed on their way into shared memory.
// `out(u, i, j, v)` takes v = dw[u][i][j .. j + 3].
constexpr int kDwFloats = 2 * 16 * 68;
template <typename T, typename Out>
__device__ __forceinline__ void dw_body(const BwdStep& p, float* smem, int block, int tid, int group, const Out& out) {
    float (*As)[68] = reinterpret_cast<float (*)[68]>(smem), (*Xs)[68] = As + 16;
    const int pos_tiles = (p.S + 63) / 64, slot_tiles = (p.M + 63) / 64;
    const int j0 = block % pos_tiles * 64; block /= pos_tiles;
    const int i0 = block % slot_tiles * 64, u = block / slot_tiles, n = u / p.heads, h = u % p.heads;
    const int ti = tid & 7, tj = tid >> 3;
    const int row = tid & 63, half = tid >> 6;
    float acc[8][4];
#pragma unroll
    for (int x = 0; x < 8; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) acc[x][y] = 0.f;
    float4 a[2], b[2];
    auto fetch = [&](int ch0) {
        const bool is_v = ch0 >= p.d;
        const int c0 = (is_v ? ch0 - p.d : ch0) + 8 * half;
        a[0] = a[1] = b[0] = b[1] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i0 + row < p.M) {
            const float* g = (is_v ? p.gV : p.gK) + ((int64_t)u * p.M + i0 + row) * p.g_st + c0;
            a[0] = load4(g);
            a[1] = load4(g + 4);
        }
        if (j0 + row < p.S) {
            const T* x = cat_row<T>(is_v ? p.xv : p.xk, n, h, j0 + row) + c0;
            b[0] = load4(x);
            b[1] = load4(x + 4);
        }
    };
    fetch(0);
#pragma unroll 1
    for (int ch0 = 0; ch0 < 2 * p.d; ch0 += 16) {
        group_sync(1 + group);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int c = 8 * half + 4 * e;
            As[c][row] = a[e].x; As[c + 1][row] = a[e].y; As[c + 2][row] = a[e].z; As[c + 3][row] = a[e].w;
            Xs[c][row] = b[e].x; Xs[c + 1][row] = b[e].y; Xs[c + 2][row] = b[e].z; Xs[c + 3][row] = b[e].w;
        }
        group_sync(1 + group);
        if (ch0 + 16 < 2 * p.d) fetch(ch0 + 16);
#pragma unroll
        for (int c = 0; c < 16; ++c) {
            const float4 g0 = *reinterpret_cast<const float4*>(&As[c][4 * ti]), g1 = *reinterpret_cast<const float4*>(&As[c][32 + 4 * ti]);
            const float4 z4 = *reinterpret_cast<const float4*>(&Xs[c][4 * tj]);
            const float g[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w}, z[4] = {z4.x, z4.y, z4.z, z4.w};
#pragma unroll
            for (int x = 0; x < 8; ++x)
#pragma unroll
                for (int y = 0; y < 4; ++y) acc[x][y] = fmaf(g[x], z[y], acc[x][y]);
        }
    }
#pragma unroll
    for (int x = 0; x < 8; ++x) out(u, i0 + (x < 4 ? 4 * ti + x : 32 + 4 * ti + x - 4), j0 + 4 * tj, make_float4(acc[x][0], acc[x][1], acc[x][2], acc[x][3]));
}

template <typename T, int D, int OT>
__global__ void __launch_bounds__(256) front_kernel(const __grid_constant__ BwdStep p, const __grid_constant__ CompressParams fwd, float* dx_attn, int n_attn, int n_conv, int n_dw) {
    extern __shared__ __align__(16) float smem[];
    wait_for_previous();
    const int key_tiles = (p.S + 31) / 32, n_keys = key_tiles * p.units;
    const int group = threadIdx.x >> 7, tid = threadIdx.x & 127;
    int x = blockIdx.x;
    if (x < n_attn) {
        // the tiles with the most work first: early keys (every query sees them), late queries
        if (x < n_keys) attention_grad<T, D, true>(p, dx_attn, smem, x / p.units, x % p.units);
        else attention_grad<T, D, false>(p, dx_attn, smem, (p.b + 31) / 32 - 1 - (x - n_keys) / p.units, (x - n_keys) % p.units);
        return;
    }
    x = 2 * (x - n_attn) + group;                      // two tiles per block from here on
    const int n_conv2 = (n_conv + 1) / 2 * 2;
    if (x < n_conv2) {
        if (x < n_conv) conv_body<T, OT>(fwd, smem + group * (WindowConv<T, OT>::smem_bytes(p.k) / 4), x, tid, group);
    } else if (x - n_conv2 < n_dw) {
        dw_body<T>(p, smem + group * kDwFloats, x - n_conv2, tid, group, [&](int u, int i, int j, const float4& v) {
            if (i < p.M && j < p.S) store4(p.dA + ((int64_t)u * p.M + i) * p.Sr + j, v);
        });
    }
}

// One warp per (unit, slot) row: R from the partial convolutions, s = sum R + eps, inner = <dw, R>/s;
// dA = [R>0] (dw - inner)/s;  dbias += sum_j dA. (Columns from S on are zeros in R and in dA.)
__global__ void __launch_bounds__(256) rows_kernel(const __grid_constant__ BwdStep p, const __grid_constant__ CompressParams fwd) {
    wait_for_previous();
    const int row = blockIdx.x * 8 + threadIdx.x / 32;
    if (row >= p.units * p.M) return;
    const int lane = threadIdx.x % 32;
    const int u = row / p.M, i = row % p.M, h = u % p.heads;
    const LogitRow L(fwd, row);
    float4* R = reinterpret_cast<float4*>(p.R + (int64_t)row * p.Sr);
    float4* dA = reinterpret_cast<float4*>(p.dA + (int64_t)row * p.Sr);
    const int n4 = p.Sr / 4;
    float inner = 0.f, sum = 0.f;
    for (int j = lane; j < n4; j += 32) {
        const float4 r = L.at4(4 * j), w = dA[j];
        R[j] = r;
        sum += r.x + r.y + r.z + r.w;
        if (r.x > 0.f) inner = fmaf(w.x, r.x, inner);
        if (r.y > 0.f) inner = fmaf(w.y, r.y, inner);
        if (r.z > 0.f) inner = fmaf(w.z, r.z, inner);
        if (r.w > 0.f) inner = fmaf(w.w, r.w, inner);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        inner += __shfl_xor_sync(0xffffffffu, inner, o);
        sum += __shfl_xor_sync(0xffffffffu, sum, o);
    }
    const float s = i < fwd.prot ? 1.f : sum + fwd.eps, inv_s = 1.f / s;
    if (lane == 0) p.s[row] = s;
    inner *= inv_s;
    float bsum = 0.f;
    for (int j = lane; j < n4; j += 32) {
        const float4 r = R[j];
        float4 w = dA[j];
        w.x = r.x > 0.f ? (w.x - inner) * inv_s : 0.f;
        w.y = r.y > 0.f ? (w.y - inner) * inv_s : 0.f;
        w.z = r.z > 0.f ? (w.z - inner) * inv_s : 0.f;
        w.w = r.w > 0.f ? (w.w - inner) * inv_s : 0.f;
        dA[j] = w;
        bsum += w.x + w.y + w.z + w.w;
    }
    if (p.dbias) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) bsum += __shfl_xor_sync(0xffffffffu, bsum, o);
        if (lane == 0) atomicAdd(p.dbias + (p.weights_per_head ? h * p.M : 0) + i, bsum);
    }
}

// ------------------------------------------------------------------ dX (compress share)
// dX[j][ch] = sum_i (R[i][j] / s_i) g[i][ch]  +  (ch < c_in)  sum_i sum_t dA[i][j - t + pad] G[i][ch][t]
// Both sums are window convolutions over the slots: the second with the taps reversed, the first with a single tap.
struct SlotRows {      // rows [slot][position] of a unit, scaled row by row where `s` is given
    const float* rows;
    const float* s;
    int M, S, Sr;
    __device__ __forceinline__ void load8(int i0, int j, float (&v)[8]) const {
        const bool in = j >= 0 && j < S;
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = (in && i0 + e < M) ? rows[(int64_t)(i0 + e) * Sr + j] * (s ? 1.f / s[i0 + e] : 1.f) : 0.f;
    }
};

// Positions j0 .. j0 + 63, channels 64 ct .. 64 ct + 63 of [keys | values], slots 8 c_begin .. 8 c_end - 1; `out(j, ch, v)` takes four
// consecutive channels of row j. kSums: sixteen slots at a time (where the slots are not split over blocks).
template <typename T, bool kSums, typename Out>
__device__ __forceinline__ void dx_tile(const BwdStep& p, int u, int j0, int ct, int c_begin, int c_end, float* smem, const Out& out) {
    const int h = u % p.heads, pad = (p.k - 1) / 2, ch0 = ct * 64;
    ConvAcc acc, total;
    acc.clear();
    if (kSums) total.clear();
    if (ch0 < p.c_in) {
        const T* w = reinterpret_cast<const T*>(p.g_reverse) + (p.weights_per_head ? (int64_t)h * p.k * p.M * p.c_in : 0);
        const SlotRows in{p.dA + (int64_t)u * p.M * p.Sr, nullptr, p.M, p.S, p.Sr};
        WindowConv<T, 64>::template run<kSums>(w, p.M, p.c_in, p.k, ch0, j0 - pad, c_begin, c_end, in, smem, acc, threadIdx.x, 0, &total);
        __syncthreads();
    }
    const float* g = (ch0 < p.d ? p.gK : p.gV) + (int64_t)u * p.M * p.g_st;
    const SlotRows in{p.R + (int64_t)u * p.M * p.Sr, p.s + (int64_t)u * p.M, p.M, p.S, p.Sr};
    WindowConv<float, 64>::run<kSums>(g, p.M, p.g_st, 1, ch0 < p.d ? ch0 : ch0 - p.d, j0, c_begin, c_end, in, smem, acc, threadIdx.x, 0, &total);
    const ConvAcc& sum = kSums ? total : acc;
    const int ti = threadIdx.x & 7, tj = threadIdx.x >> 3;
#pragma unroll
    for (int y = 0; y < 4; ++y) {
        const int j = j0 + 4 * tj + y;
        if (j >= p.S) break;
        out(j, ch0 + 4 * ti, make_float4(sum.get(0, y), sum.get(1, y), sum.get(2, y), sum.get(3, y)));
        out(j, ch0 + 4 * ti + 32, make_float4(sum.get(4, y), sum.get(5, y), sum.get(6, y), sum.get(7, y)));
    }
}
template <typename T>
__device__ __forceinline__ void dx_body(const BwdStep& p, float* parts, int splits, float* smem, int block) {
    const int pos_tiles = (p.S + 63) / 64;
    const int jt = block % pos_tiles; block /= pos_tiles;
    const int u = block % p.units; block /= p.units;
    const int split = block % splits, ct = block / splits;
    const int chunks = (p.M + 7) / 8;
    float* dst = parts + ((int64_t)split * p.units + u) * p.S * (2 * p.d);
    dx_tile<T, false>(p, u, 64 * jt, ct, chunks * split / splits, chunks * (split + 1) / splits, smem,
                      [&](int j, int ch, const float4& v) { store4(dst + (int64_t)j * 2 * p.d + ch, v); });
}

// ------------------------------------------------------------------ dG
// dG[set][i][ch][t] += sum over the set's units, sum_j dA[u][i][j] * Z_u[j+t-pad][ch].
// A block of 128 threads takes 16 slots x 32 channels x up to 8 taps and one stretch of positions of one unit: a lane owns a
// channel, a warp four slots; eight positions at a time, the 15 inputs they and eight taps touch sit in registers and serve
// 256 FMAs together with eight vector loads of dA. Blocks of the same set meet in atomics.
constexpr int kGTaps = 8, kGPos = 64, kGSlots = 16;
// Taps per block: at most eight, as few as cover k in as many blocks (kT, what the code is unrolled for: 5 to 8, no fewer).
__host__ __device__ inline int g_taps(int k) { const int tiles = (k + kGTaps - 1) / kGTaps; return (k + tiles - 1) / tiles; }
// `stage(q, dA, xk, xv, S, j0)`: the q-th stretch of 64 positions (of all that are to be summed: one chunk's, or several chunks').
template <typename T, int kT, typename Stage>
__device__ __forceinline__ void dg_tile(const BwdStep& p, int pieces, int stages, float* smem, int block, const Stage& stage) {
    float* As = smem;                        // [16 slots][64 positions], row stride 68
    float* Zs = smem + kGSlots * 68;         // [64 + 8 positions][32 channels], row stride 33
    const int slot_tiles = (p.M + kGSlots - 1) / kGSlots, ch_tiles = p.c_in / 32;
    const int piece = block % pieces; block /= pieces;
    const int u = block % p.units; block /= p.units;
    const int ch0 = (block % ch_tiles) * 32; block /= ch_tiles;
    const int i0 = (block % slot_tiles) * kGSlots, taps = g_taps(p.k), t0 = (block / slot_tiles) * taps;
    const int n = u / p.heads, h = u % p.heads, set = p.weights_per_head ? h : 0, pad = (p.k - 1) / 2;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float acc[4][kT];
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int t = 0; t < kT; ++t) acc[x][t] = 0.f;
#pragma unroll 1
    for (int st = stages * piece / pieces; st < stages * (piece + 1) / pieces; ++st) {
        const float* dA;
        CatView xk, xv;
        int S, j0;
        if (!stage(st, dA, xk, xv, S, j0)) continue;
        dA += (int64_t)u * p.M * p.Sr;
        __syncthreads();
        for (int x = tid; x < kGSlots * (kGPos / 4); x += 128) {
            const int r = x / (kGPos / 4), q = 4 * (x % (kGPos / 4));
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (i0 + r < p.M && j0 + q < p.Sr) v = load4(dA + (int64_t)(i0 + r) * p.Sr + j0 + q);
            *reinterpret_cast<float4*>(As + r * 68 + q) = v;
        }
        for (int x = tid; x < (kGPos + kGTaps) * 8; x += 128) {
            const int r = x >> 3, q = 4 * (x & 7), j = j0 + r + t0 - pad, ch = ch0 + q;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (j >= 0 && j < S) v = load4(ch < p.d ? cat_row<T>(xk, n, h, j) + ch : cat_row<T>(xv, n, h, j) + ch - p.d);
            float* d = Zs + r * 33 + q;
            d[0] = v.x; d[1] = v.y; d[2] = v.z; d[3] = v.w;
        }
        __syncthreads();
#pragma unroll 1
        for (int j = 0; j < kGPos; j += 8) {
            float z[8 + kT - 1];
#pragma unroll
            for (int e = 0; e < 8 + kT - 1; ++e) z[e] = Zs[(j + e) * 33 + lane];
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const float4 a0 = *reinterpret_cast<const float4*>(As + (4 * warp + x) * 68 + j), a1 = *reinterpret_cast<const float4*>(As + (4 * warp + x) * 68 + j + 4);
                const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
                for (int e = 0; e < 8; ++e)
#pragma unroll
                    for (int t = 0; t < kT; ++t) acc[x][t] = fmaf(a[e], z[e + t], acc[x][t]);
            }
        }
    }
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        const int i = i0 + 4 * warp + x;
        if (i >= p.M) break;
        float* out = p.dG + (((int64_t)set * p.M + i) * p.c_in + ch0 + lane) * p.k + t0;
#pragma unroll
        for (int t = 0; t < kT; ++t)
            if (t < taps && t0 + t < p.k) atomicAdd(out + t, acc[x][t]);
    }
}

template <typename T, typename Stage>
__device__ __forceinline__ void dg_body(const BwdStep& p, int pieces, int stages, float* smem, int block, const Stage& stage) {
    switch (g_taps(p.k)) {
        case 8: return dg_tile<T, 8>(p, pieces, stages, smem, block, stage);
        case 7: return dg_tile<T, 7>(p, pieces, stages, smem, block, stage);
        case 6: return dg_tile<T, 6>(p, pieces, stages, smem, block, stage);
        default: return dg_tile<T, 5>(p, pieces, stages, smem, block, stage);
    }
}

template <typename T>
__global__ void __launch_bounds__(128) dx_dg_kernel(const __grid_constant__ BwdStep p, float* parts, int splits, int n_dx, int pieces) {
    extern __shared__ __align__(16) float smem[];
    wait_for_previous();
    if ((int)blockIdx.x < n_dx) dx_body<T>(p, parts, splits, smem, blockIdx.x);
    else dg_body<T>(p, pieces, (p.S + kGPos - 1) / kGPos, smem, blockIdx.x - n_dx, [&](int q, const float*& dA, CatView& xk, CatView& xv, int& S, int& j0) {
        dA = p.dA; xk = p.xk; xv = p.xv; S = p.S; j0 = q * kGPos;
        return true;
    });
}

// ------------------------------------------------------------------ split
// dX = attention share + compress share (or, after a fill step, the gradient of the filled cache itself). Rows 0..c-1 become
// the gradient w.r.t. the cache before this step (rows >= c: zero); rows c..S-1 are this chunk's dK, dV.
template <typename T>
__global__ void __launch_bounds__(256) split_kernel(const __grid_constant__ BwdStep p, const float* attn, const float* parts, int n_parts) {
    wait_for_previous();
    const int u = blockIdx.y, n = u / p.heads, h = u % p.heads;
    const int per_row = p.d / 2, rows = max(p.M, p.S);           // float4 pieces of a [key | value] row
    const int64_t step = (int64_t)p.units * p.S * (2 * p.d);
    for (int x = blockIdx.x * 256 + threadIdx.x; x < rows * per_row; x += gridDim.x * 256) {
        const int row = x / per_row, c2 = 4 * (x % per_row);
        const bool is_v = c2 >= p.d;
        const int ch = is_v ? c2 - p.d : c2;
        float* g = (is_v ? p.gV : p.gK) + ((int64_t)u * p.M + row) * p.d + ch;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (row < p.S) {
            const int64_t at = ((int64_t)u * p.S + row) * (2 * p.d) + c2;
            v = load4(attn + at);
            if (n_parts == 0) {
                const float4 w = load4(g);
                v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
            }
            for (int s = 0; s < n_parts; ++s) {
                const float4 w = load4(parts + s * step + at);
                v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
            }
        }
        if (row < p.M) store4(g, row < p.c ? v : make_float4(0.f, 0.f, 0.f, 0.f));
        if (row >= p.c && row < p.S) store4(unit_base_mut<T>(is_v ? p.dv : p.dk, n, h) + (int64_t)(row - p.c) * (is_v ? p.dv : p.dk).st + ch, v);
    }
}

// Partial sums of dX: one per block sharing a 64 x 64 tile's slots; few tiles are split so that they fill the machine
// (three blocks per SM), each keeping at least two chunks of eight slots.
int dx_splits(int units, int S, int M, int d) {
    const int64_t tiles = (int64_t)units * ((S + 63) / 64) * (2 * d / 64);
    return (int)std::max<int64_t>(1, std::min<int64_t>(3 * kSMs / tiles, M / 16));
}

template <typename T, int D, int OT>
int launch_front(const BwdStep& p, const CompressParams& fwd, float* dx_attn, int n_conv, int n_dw, cudaStream_t st) {
    static bool done[64] = {};
    const size_t attn = sizeof(float) * GradSmem<D>::kFloats, conv = 2 * WindowConv<T, OT>::smem_bytes(p.k), dw = sizeof(float) * 2 * kDwFloats;
    if (!smem_limit(front_kernel<T, D, OT>, 200 * 1024, done)) return -1;
    const int n_attn = ((p.S + 31) / 32 + (p.b + 31) / 32) * p.units, blocks = n_attn + (n_conv + 1) / 2 + (n_dw + 1) / 2;
    return launch_after(front_kernel<T, D, OT>, dim3(blocks), dim3(256), std::max(attn, n_conv ? std::max(conv, dw) : (size_t)0), st, p, fwd, dx_attn, n_attn, n_conv, n_dw) ? 1 : -1;
}
template <typename T, int D>
int launch_front_tiles(const BwdStep& p, const CompressParams& fwd, float* dx_attn, int n_conv, int n_dw, cudaStream_t st) {
    switch (slot_tile(p.M)) {
        case 64: return launch_front<T, D, 64>(p, fwd, dx_attn, n_conv, n_dw, st);
        case 32: return launch_front<T, D, 32>(p, fwd, dx_attn, n_conv, n_dw, st);
        default: return launch_front<T, D, 16>(p, fwd, dx_attn, n_conv, n_dw, st);
    }
}

template <typename T>
int step_typed(const BwdStep& p, CompressParams fwd, float* parts, cudaStream_t st) {
    float* attn = parts;
    float* comp = parts + (int64_t)p.units * p.S * (2 * p.d);
    const bool compress = p.S > p.M;
    fwd.splits = conv_splits(fwd);
    const int n_conv = compress ? conv_tiles(fwd) : 0, n_dw = compress ? (p.S + 63) / 64 * ((p.M + 63) / 64) * p.units : 0;
    int n = p.d == 128 ? launch_front_tiles<T, 128>(p, fwd, attn, n_conv, n_dw, st) : launch_front_tiles<T, 64>(p, fwd, attn, n_conv, n_dw, st);
    if (n < 0) return -1;
    int splits = 0;
    if (compress) {
        if (!launch_after(rows_kernel, dim3((p.units * p.M + 7) / 8), dim3(256), 0, st, p, fwd)) return -1;
        splits = dx_splits(p.units, p.S, p.M, p.d);
        const int n_dx = (p.S + 63) / 64 * (2 * p.d / 64) * p.units * splits;
        // dG: position stretches per unit, so that about six blocks per SM exist, none shorter than a stage
        const int tiles = (p.k + kGTaps - 1) / kGTaps * ((p.M + kGSlots - 1) / kGSlots) * (p.c_in / 32) * p.units;
        const int pieces = std::max(1, std::min((p.S + kGPos - 1) / kGPos, 6 * kSMs / std::max(1, tiles)));
        const size_t smem = std::max(WindowConv<T, 64>::smem_bytes(p.k), sizeof(float) * (kGSlots * 68 + (kGPos + kGTaps) * 33));
        static bool done[64] = {};
        if (!smem_limit(dx_dg_kernel<T>, 64 * 1024, done)) return -1;
        if (!launch_after(dx_dg_kernel<T>, dim3(n_dx + tiles * pieces), dim3(128), smem, st, p, comp, splits, n_dx, pieces)) return -1;
        n += 2;
    }
    const int total = std::max(p.M, p.S) * (p.d / 2);
    if (!launch_after(split_kernel<T>, dim3((total + 255) / 256, p.units), dim3(256), 0, st, p, attn, comp, splits)) return -1;
    return n + 1;
}

// ------------------------------------------------------------------ groups of chunks
// Of a step's work only the cache rows' dw, dA and dX wait for the step behind it. For problems of which one chunk does not fill the chip,
// everything else is done for a whole group of chunks at a time:
//   group_front   attention gradients (dQ, shares of dX) and the recomputed convolution, all chunks side by side
//   group_rows    R, s; the cache after the call's last chunk
//   (simt_chain)  the chain through the cache gradient, one launch for all steps
//   group_logits  dA (and dbias) at all positions
//   group_out     dK, dV of the chunks' rows, and dG
// 8 units, M = 48, B = 100, d = 64, k = 5, 8 chunks: 171 us where the four launches of every step took 380 (front 59, rows 9, chain 36, logits 17, out 49).
__device__ __forceinline__ void step_of(const BwdGroup& G, int i, BwdStep& p) {
    p = G.first;
    const int n = G.n0 + i, t0 = n * G.B;
    p.c = min(p.M, G.c0 + t0);
    p.b = min(G.B, G.L - t0);
    p.S = p.c + p.b;
    p.Sr = G.Sr;
    auto tokens = [&](View& v) { v.ptr += (int64_t)t0 * v.st * 4; };
    tokens(p.xk.chunk); tokens(p.xv.chunk); tokens(p.q); tokens(p.o); tokens(p.d_o); tokens(p.dq); tokens(p.dk); tokens(p.dv);
    p.xk.cache.ptr += n * G.snap_step * 4;
    p.xv.cache.ptr += n * G.snap_step * 4;
    p.xk.c = p.xv.c = p.c;
    p.xk.b = p.xv.b = p.b;
    p.lse += t0;
    p.delta += t0;
    const int64_t rows = (int64_t)i * p.units * p.M;
    p.R = G.R + rows * G.splits * G.Sr;
    p.s = G.s + rows;
    p.dA = G.dA + rows * G.Sr;
    p.gK = G.g + (rows + (int64_t)p.units * p.M) * (2 * p.d);        // the gradient w.r.t. the cache after the step
    p.gV = p.gK + p.d;
    p.g_st = 2 * p.d;
}
__device__ __forceinline__ void logits_of(const BwdGroup& G, const BwdStep& p, CompressParams& f) {
    f.xk = p.xk; f.xv = p.xv;
    f.heads = p.heads; f.units = p.units; f.d = p.d; f.M = p.M; f.k = p.k; f.c_in = p.c_in;
    f.S = p.S; f.Sr = p.Sr; f.splits = G.splits; f.weights_per_head = p.weights_per_head;
    f.g_packed = G.g_packed; f.bias = G.bias; f.eps = G.eps; f.prot = G.prot; f.R = p.R; f.s = p.s;
}

template <int D, int OT>
__global__ void __launch_bounds__(256) group_front_kernel(const __grid_constant__ BwdGroup G, int n_conv) {
    extern __shared__ __align__(16) float smem[];
    __shared__ BwdStep p;
    __shared__ __align__(16) unsigned char fwd_bytes[sizeof(CompressParams)];
    CompressParams& fwd = *reinterpret_cast<CompressParams*>(fwd_bytes);
    wait_for_previous();
    const int units = G.first.units, each = units * G.count;
    const int n_keys = (G.S + 31) / 32 * each, n_queries = (G.B + 31) / 32 * each;
    const int group = threadIdx.x >> 7, tid = threadIdx.x & 127;
    int x = blockIdx.x;
    const int kind = x < n_keys ? 0 : (x < n_keys + n_queries ? 1 : 2);
    x -= kind == 0 ? 0 : (kind == 1 ? n_keys : n_keys + n_queries);
    const int conv_blocks = (n_conv + 1) / 2;
    const int i = kind == 2 ? x / conv_blocks : x % each / units;
    if (threadIdx.x == 0) {
        step_of(G, i, p);
        if (kind == 2) logits_of(G, p, fwd);
    }
    __syncthreads();
    if (kind < 2) {
        // the tiles with the most work first: early keys (every query sees them), late queries
        const int tile = x / each, u = x % units;
        if (kind == 0) {
            if (32 * tile < p.S) attention_grad<float, D, true>(p, G.attn + (int64_t)i * units * G.S * (2 * D), smem, tile, u);
        } else {
            const int last = (p.b + 31) / 32 - 1;
            if (tile <= last) attention_grad<float, D, false>(p, nullptr, smem, last - tile, u);
        }
        return;
    }
    constexpr int PT = WindowConv<float, OT>::PT;
    const int tile = 2 * (x % conv_blocks) + group, tiles = (p.S + PT - 1) / PT * ((p.M + OT - 1) / OT) * G.splits * units;
    if (p.S > p.M && tile < tiles) conv_body<float, OT>(fwd, smem + group * (WindowConv<float, OT>::smem_bytes(p.k) / 4), tile, tid, group);
}

// R from the partial convolutions and s = sum R + eps, a warp per (chunk, unit, slot); for the last chunk of the call, the first
// `last_blocks` blocks, also the new cache: a block takes four slots of a unit, two warps each for R, all warps a share of the
// positions for the blends. (A block per slot read the chunk's rows four times as often: 100 us at 96 units, M = 32, B = 142.)
__global__ void __launch_bounds__(256) group_rows_kernel(const __grid_constant__ BwdGroup G, int last_blocks) {
    __shared__ float sums[8];
    __shared__ __align__(16) float blend[8][4][128];
    wait_for_previous();
    const int M = G.first.M, rows = G.first.units * M, per_chunk = (rows + 7) / 8, warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const bool wide = (int)blockIdx.x < last_blocks;
    const int x = (int)blockIdx.x - last_blocks, i = wide ? G.count - 1 : x / per_chunk, per_unit = (M + 3) / 4;
    const int u4 = blockIdx.x / per_unit, i4 = 4 * (blockIdx.x % per_unit), slot4 = min(i4 + warp / 2, M - 1);
    const int row = wide ? u4 * M + slot4 : x % per_chunk * 8 + warp;
    BwdStep p;
    CompressParams fwd;
    step_of(G, i, p);
    logits_of(G, p, fwd);
    if (p.S <= M || row >= rows) return;
    const LogitRow L(fwd, row);
    float* R = p.R + (int64_t)row * p.Sr;
    float sum = 0.f;
    const bool twice = wide && i4 + warp / 2 >= M;                 // (another pair of warps has this row)
    for (int j = 4 * (wide ? lane + 32 * (warp & 1) : lane); j < p.Sr && !twice; j += wide ? 256 : 128) {
        const float4 r = L.at4(j);
        store4(R + j, r);
        sum += (r.x + r.y) + (r.z + r.w);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (!wide) {
        if (lane == 0) p.s[row] = row % M < G.prot ? 1.f : sum + G.eps;
        return;
    }
    if (lane == 0) sums[warp] = sum;
    __syncthreads();
    const int n = u4 / p.heads, h = u4 % p.heads;
    const float* rows4[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) rows4[a] = p.R + (int64_t)(u4 * M + min(i4 + a, M - 1)) * p.Sr;
#pragma unroll 1
    for (int ch0 = 0; ch0 < 2 * p.d; ch0 += 128) {
        const int ch = ch0 + 4 * lane;
        float4 acc[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) acc[a] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
        for (int j = warp; j < p.S; j += 8) {
            const float4 v = load4(ch < p.d ? cat_row<float>(p.xk, n, h, j) + ch : cat_row<float>(p.xv, n, h, j) + ch - p.d);
#pragma unroll
            for (int a = 0; a < 4; ++a) axpy4(rows4[a][j], v, acc[a]);
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) store4(&blend[warp][a][4 * lane], acc[a]);
        __syncthreads();
        for (int e = threadIdx.x; e < 512; e += 256) {
            const int a = e / 128, c = e % 128, slot = i4 + a;
            if (slot >= M || ch0 + c >= 2 * p.d) continue;
            float v[4];
#pragma unroll
            for (int w = 0; w < 4; ++w) v[w] = blend[2 * w][a][c] + blend[2 * w + 1][a][c];
            const float s = slot < G.prot ? 1.f : sums[2 * a] + sums[2 * a + 1] + G.eps;
            if (ch0 + c == 0) p.s[u4 * M + slot] = s;
            G.last[((int64_t)u4 * M + slot) * (2 * p.d) + ch0 + c] = ((v[0] + v[1]) + (v[2] + v[3])) * (1.f / s);
        }
        __syncthreads();
    }
}

// dw at all positions, and dA: a block of 256 threads takes 16 or 32 slots (32 where that leaves fewer than 16 idle: the rows are then
// read half as often) x 128 positions of a unit, 2 or 4 x 4 per thread; keys and values with their
// gradients come whole (asynchronous copies, the values while the keys' half is summed). (With 64 x 64 tiles by groups of 128
// threads, sixteen channels per barrier: 32 us at 8 units, M = 48, B = 100, 8 chunks; now 17.)
template <int D, int kSlots>
struct DwSmem {
    static constexpr int kRow = D + 4, kRows = 128 + kSlots, kHalf = kRows * kRow, kFloats = 2 * kHalf;
};
template <int D, int kSlots>
__global__ void __launch_bounds__(256) group_logits_kernel(const __grid_constant__ BwdGroup G) {
    extern __shared__ __align__(16) float smem[];
    __shared__ float bias_part[8][kSlots];
    wait_for_previous();
    using Smem = DwSmem<D, kSlots>;
    constexpr int RS = Smem::kRow, kA = kSlots / 8;      // slots per thread: ti, ti + 8, ...
    const int tid = threadIdx.x, lane = tid & 31, ti = tid & 7, tj = tid >> 3;
    const int pos_tiles = (G.S + 127) / 128, slot_tiles = (G.first.M + kSlots - 1) / kSlots;
    int x = blockIdx.x;
    const int j0 = 128 * (x % pos_tiles); x /= pos_tiles;
    const int i0 = kSlots * (x % slot_tiles); x /= slot_tiles;
    const int u = x % G.first.units, i = x / G.first.units;
    BwdStep p;
    step_of(G, i, p);
    if (p.S <= p.M || j0 >= p.S) return;
    const int n = u / p.heads, h = u % p.heads;
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
        const CatView& xs = half ? p.xv : p.xk;
        const float *cache = unit_base<float>(xs.cache, n, h), *chunk = unit_base<float>(xs.chunk, n, h);
        const float* g = (half ? p.gV : p.gK) + ((int64_t)u * p.M + i0) * p.g_st;
        float* dst = smem + half * Smem::kHalf;
        const int ch = 4 * (tid % (D / 4));
        for (int r = tid / (D / 4); r < Smem::kRows; r += 256 / (D / 4)) {
            const int j = j0 + r;
            const bool live = r < 128 ? j < p.S : i0 + r - 128 < p.M;
            const float* src = r >= 128 ? g + (int64_t)(r - 128) * p.g_st : (j < p.c ? cache + (int64_t)j * xs.cache.st : chunk + (int64_t)(j - p.c) * xs.chunk.st);
            cp_async16(dst + r * RS + ch, live ? src + ch : cache, live);
        }
        cp_async_commit();
    }
    f32x2 acc[kA][4];
#pragma unroll
    for (int a = 0; a < kA; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = 0ull;
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
        if (half) cp_async_wait<0>();
        else cp_async_wait<1>();
        __syncthreads();
        const float *xr = smem + half * Smem::kHalf + tj * RS, *gr = smem + half * Smem::kHalf + (128 + ti) * RS;
#pragma unroll 2
        for (int q = 0; q < D / 4; ++q) {
            f32x4 z[4];
#pragma unroll
            for (int b = 0; b < 4; ++b) z[b] = load_pairs(xr + 32 * b * RS + 4 * q);
#pragma unroll
            for (int a = 0; a < kA; ++a) {
                const f32x4 w = load_pairs(gr + 8 * a * RS + 4 * q);
#pragma unroll
                for (int b = 0; b < 4; ++b) { fma2(w.lo, z[b].lo, acc[a][b]); fma2(w.hi, z[b].hi, acc[a][b]); }
            }
        }
    }
    const float* inner = G.inner + ((int64_t)i * p.units + u) * p.M;
#pragma unroll
    for (int a = 0; a < kA; ++a) {
        const int slot = i0 + ti + 8 * a, row = u * p.M + slot;
        float sum = 0.f;
        if (slot < p.M) {
            const float inv = 1.f / p.s[row], in = inner[slot];
            const float* R = p.R + (int64_t)row * p.Sr;
            float* dA = p.dA + (int64_t)row * p.Sr;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int j = j0 + tj + 32 * b;
                if (j >= p.Sr) break;
                const float2 f = unpair(acc[a][b]);
                const float v = slot >= G.prot && R[j] > 0.f ? (f.x + f.y - in) * inv : 0.f;      // (a protected slot's row has no gradient)
                dA[j] = v;
                sum += v;
            }
        }
        if (p.dbias) {                                   // lanes ti, ti + 8, ... hold positions of the same slot
#pragma unroll
            for (int o = 8; o < 32; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            if (lane < 8) bias_part[tid >> 5][ti + 8 * a] = sum;
        }
    }
    if (!p.dbias) return;
    __syncthreads();
    if (tid < kSlots && i0 + tid < p.M) {
        float v[4];
#pragma unroll
        for (int w = 0; w < 4; ++w) v[w] = bias_part[2 * w][tid] + bias_part[2 * w + 1][tid];
        atomicAdd(p.dbias + (p.weights_per_head ? h * p.M : 0) + i0 + tid, (v[0] + v[1]) + (v[2] + v[3]));
    }
}

__global__ void __launch_bounds__(128) group_out_kernel(const __grid_constant__ BwdGroup G, int n_dx, int pieces) {
    extern __shared__ __align__(16) float smem[];
    wait_for_previous();
    const BwdStep& F = G.first;
    int x = blockIdx.x;
    if (x >= n_dx) {
        const int per = (G.S + kGPos - 1) / kGPos;
        dg_body<float>(F, pieces, per * G.count, smem, x - n_dx, [&](int q, const float*& dA, CatView& xk, CatView& xv, int& S, int& j0) {
            const int i = q / per, n = G.n0 + i, t0 = n * G.B, c = min(F.M, G.c0 + t0);
            j0 = (q - i * per) * kGPos;
            S = c + min(G.B, G.L - t0);
            if (S <= F.M || j0 >= S) return false;
            dA = G.dA + (int64_t)i * F.units * F.M * G.Sr;
            xk = F.xk; xv = F.xv;
            xk.cache.ptr += n * G.snap_step * 4; xv.cache.ptr += n * G.snap_step * 4;
            xk.chunk.ptr += (int64_t)t0 * xk.chunk.st * 4; xv.chunk.ptr += (int64_t)t0 * xv.chunk.st * 4;
            xk.c = xv.c = c;
            return true;
        });
        return;
    }
    const int tiles = (G.B + 63) / 64, jt = x % tiles; x /= tiles;
    const int ct = x % (F.d / 32); x /= F.d / 32;
    const int u = x % F.units, i = x / F.units;
    BwdStep p;
    step_of(G, i, p);
    if (64 * jt >= p.b) return;
    const int n = u / p.heads, h = u % p.heads;
    const float* attn = G.attn + ((int64_t)i * p.units * G.S + (int64_t)u * p.S) * (2 * p.d);
    auto put = [&](int j, int ch, const float4& v) {
        const bool is_v = ch >= p.d;
        const View& out = is_v ? p.dv : p.dk;
        const float4 a = load4(attn + (int64_t)j * (2 * p.d) + ch);
        store4(unit_base_mut<float>(out, n, h) + (int64_t)(j - p.c) * out.st + (is_v ? ch - p.d : ch), make_float4(v.x + a.x, v.y + a.y, v.z + a.z, v.w + a.w));
    };
    const int j0 = p.c + 64 * jt;
    if (p.S > p.M) {
        dx_tile<float, true>(p, u, j0, ct, 0, (p.M + 7) / 8, smem, put);
        return;
    }
    // a fill step: the gradient of the filled cache itself
    for (int e = threadIdx.x; e < 64 * 16; e += 128) {
        const int j = j0 + e / 16, ch = 64 * ct + 4 * (e % 16);
        if (j < p.S) put(j, ch, load4(p.gK + ((int64_t)u * p.M + j) * p.g_st + ch));
    }
}

template <int D, int OT>
int launch_group_front(const BwdGroup& G, cudaStream_t st) {
    static bool done[64] = {};
    if (!smem_limit(group_front_kernel<D, OT>, 200 * 1024, done)) return -1;
    const int each = G.first.units * G.count, pt = WindowConv<float, OT>::PT;
    const int n_conv = (G.S + pt - 1) / pt * ((G.first.M + OT - 1) / OT) * G.splits * G.first.units;
    const size_t smem = std::max(sizeof(float) * (size_t)GradSmem<D>::kFloats, 2 * WindowConv<float, OT>::smem_bytes(G.first.k));
    const int64_t blocks = (int64_t)((G.S + 31) / 32 + (G.B + 31) / 32) * each + (int64_t)(n_conv + 1) / 2 * G.count;
    return launch_after(group_front_kernel<D, OT>, dim3((unsigned)blocks), dim3(256), smem, st, G, n_conv) ? 1 : -1;
}
template <int D>
int launch_group_front_tiles(const BwdGroup& G, cudaStream_t st) {
    switch (slot_tile(G.first.M)) {
        case 64: return launch_group_front<D, 64>(G, st);
        case 32: return launch_group_front<D, 32>(G, st);
        default: return launch_group_front<D, 16>(G, st);
    }
}

template <int D, int kSlots>
int launch_group_logits(const BwdGroup& G, cudaStream_t st) {
    static bool done[64] = {};
    const int smem = sizeof(float) * DwSmem<D, kSlots>::kFloats, blocks = (G.S + 127) / 128 * ((G.first.M + kSlots - 1) / kSlots) * G.first.units * G.count;
    if (!smem_limit(group_logits_kernel<D, kSlots>, smem, done)) return -1;
    return launch_after(group_logits_kernel<D, kSlots>, dim3(blocks), dim3(256), smem, st, G) ? 1 : -1;
}
template <int D>
int launch_group_logits_tiles(const BwdGroup& G, cudaStream_t st) {
    return (G.first.M + 31) / 32 * 32 - G.first.M < 16 ? launch_group_logits<D, 32>(G, st) : launch_group_logits<D, 16>(G, st);
}

// Partial sums per tile of the recomputed convolution, as in conv_splits, for the tiles of all chunks together.
int group_splits(int units, int M, int S, int c_in, int chunks) {
    const int OT = slot_tile(M), PT = 4096 / OT;
    const int64_t tiles = (int64_t)((S + PT - 1) / PT) * ((M + OT - 1) / OT) * units * chunks;
    return (int)std::max<int64_t>(1, std::min<int64_t>(6 * kSMs / tiles, c_in / 32));
}
size_t group_floats(int units, int M, int S, int d, int splits, int chunks) {
    const size_t rows = (size_t)units * M, Sr = (S + 3) / 4 * 4;
    return chunks * ((size_t)units * S * 2 * d + rows * Sr * (splits + 1) + 2 * ((rows + 3) / 4 * 4)) + (chunks + 2) * rows * 2 * d;
}

}  // namespace

size_t simt_backward_parts_floats(int units, int M, int B, int d) {
    // the attention share, and the partial sums of the compress share (splits * tiles <= three tiles of 64 x 64 per SM)
    const size_t one = (size_t)units * (M + B) * 2 * d;
    return one + std::min(one * std::max(1, M / 16), std::max(one, (size_t)3 * kSMs * 4096));
}

int simt_backward_fill_split(int dtype, const BwdStep& p, const float* attn, cudaStream_t st) {
    const dim3 grid((std::max(p.M, p.S) * (p.d / 2) + 255) / 256, p.units);
    const float* none = nullptr;
    return (dtype == LOCOCO_F32 ? launch_after(split_kernel<float>, grid, dim3(256), 0, st, p, attn, none, 0)
                                : launch_after(split_kernel<__nv_bfloat16>, grid, dim3(256), 0, st, p, attn, none, 0)) ? 1 : -1;
}

int simt_backward_step(int dtype, const BwdStep& p, const CompressParams& fwd, float* parts, cudaStream_t st) {
    return dtype == LOCOCO_F32 ? step_typed<float>(p, fwd, parts, st) : step_typed<__nv_bfloat16>(p, fwd, parts, st);
}

int simt_group_chunks(const lococo_handle* h, int L, int B, size_t room, size_t* floats) {
    const lococo_config& c = h->cfg;
    B = std::min(B, L);
    const int chunks = (L + B - 1) / B;
    *floats = 0;
    if (c.dtype != LOCOCO_F32 || chunks < 2 || (size_t)c.M * c.head_dim > 6144 || !simt_group_possible(h, B)) return 0;      // (larger caches: not in simt_chain.cu's shared memory)
    // Where the attention's blocks of one chunk alone are more than six per SM, single steps are as fast and take less memory (96 units,
    // M = 32, B = 142: 571 us a step at a time, 588 in one group). simt_group_clusters draws a narrower line, by what the device runs at once.
    if ((int64_t)((c.M + B + 31) / 32 + (B + 31) / 32) * h->units > 6 * kSMs) return 0;
    // as many chunks as 128 MB hold, or the caller's scratch
    auto need = [&](int n) { return group_floats(h->units, c.M, c.M + B, c.head_dim, group_splits(h->units, c.M, c.M + B, c.c_in, n), n); };
    room = std::min(room, (size_t)32 << 20);
    int n = std::min(chunks, 4096);
    while (n > 1 && need(n) > room) n = std::min(n - 1, (n * 7 + 7) / 8);
    if (n < 2) return 0;
    *floats = need(n);
    return n;
}

size_t simt_group_layout(BwdGroup& G, float* scratch, size_t floats) {
    const BwdStep& p = G.first;
    const size_t rows = (size_t)p.units * p.M;
    // The group that is left over at the front of a call may have fewer chunks than the others, and with fewer tiles its convolution is split
    // further: only as far as the room goes. (As far as a whole group's always fits.)
    G.splits = group_splits(p.units, p.M, G.S, p.c_in, G.count);
    while (G.splits > 1 && group_floats(p.units, p.M, G.S, p.d, G.splits, G.count) > floats) --G.splits;
    float* at = scratch;
    auto take = [&](size_t n) { float* r = at; at += n; return r; };
    G.attn = take((size_t)G.count * p.units * G.S * 2 * p.d);
    G.R = take(G.count * rows * G.Sr * G.splits);
    G.dA = take(G.count * rows * G.Sr);
    G.g = take((G.count + 1) * rows * 2 * p.d);
    G.last = take(rows * 2 * p.d);
    G.s = take(G.count * ((rows + 3) / 4 * 4));
    G.inner = take(G.count * ((rows + 3) / 4 * 4));
    return at - scratch;
}

int simt_backward_group(const BwdGroup& G, cudaStream_t st) {
    const BwdStep& p = G.first;
    const int rows = p.units * p.M;
    static bool done[64] = {};
    if ((p.d == 128 ? launch_group_front_tiles<128>(G, st) : launch_group_front_tiles<64>(G, st)) < 0) return -1;
    const int last = (G.n0 + G.count) * (int64_t)G.B >= G.L, last_blocks = last ? (p.M + 3) / 4 * p.units : 0;
    if (!launch_after(group_rows_kernel, dim3(last_blocks + (rows + 7) / 8 * (G.count - last)), dim3(256), 0, st, G, last_blocks)) return -1;
    if (simt_backward_chain(G, st) < 0) return -1;
    if ((p.d == 128 ? launch_group_logits_tiles<128>(G, st) : launch_group_logits_tiles<64>(G, st)) < 0) return -1;
    const int n_dx = (G.B + 63) / 64 * (p.d / 32) * p.units * G.count;
    // dG: stretches of the group's positions per unit, so that about six blocks per SM exist, none shorter than a stage
    const int tiles = (p.k + kGTaps - 1) / kGTaps * ((p.M + kGSlots - 1) / kGSlots) * (p.c_in / 32) * p.units;
    const int stages = (G.S + kGPos - 1) / kGPos * G.count, most = std::max(1, std::min(stages, 6 * kSMs / std::max(1, tiles)));
    const int pieces = (stages + (stages + most - 1) / most - 1) / ((stages + most - 1) / most);      // (as many stages each)
    const size_t smem = std::max(WindowConv<float, 64>::smem_bytes(p.k), sizeof(float) * (kGSlots * 68 + (kGPos + kGTaps) * 33));
    if (!smem_limit(group_out_kernel, 64 * 1024, done)) return -1;
    if (!launch_after(group_out_kernel, dim3(n_dx + tiles * pieces), dim3(128), smem, st, G, n_dx, pieces)) return -1;
    return 5;
}

}  // namespace lococo
