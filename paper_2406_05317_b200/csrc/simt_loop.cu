// Algorithm 2's whole chunk loop in one launch, for small fp32 problems: a cluster of 1 to 16 CTAs of 512 threads owns one
// (sequence, head) unit; every CTA keeps the unit's whole [cache; chunk] in shared memory.
//
// Such a problem is all latency: with M = B = 16, d = 64, k = 5 a chunk is 280 thousand FMAs, a microsecond of one SM,
// and through the per-chunk launches (three per chunk, 2 to 3 us each on the host alone) 256 tokens took 252 us.
// The CTAs of a cluster share the slots and the chunk's queries: a CTA convolves for its own slots over all positions, so that
// their rows of R, their denominators and their new cache rows are its own affair, and it writes those rows into the shared
// memory of all CTAs; one cluster barrier per chunk is all the exchange there is. Within a CTA two groups of warps work side by side:
//   the chain   convolution of Eq. 6 with bias and ReLU -> barrier of these warps -> new rows R [X_K | X_V] / (sum R + eps), into the
//               other of two row buffers, of every CTA
//   attention   a warp takes up to four queries from scores to output, with no barrier at all; before that these warps ask for the
//               next chunk's rows (asynchronous copies into the other buffer)
// The convolution is tiles of 2 to 4 slots x 4 or 8 positions whose channels are spread over the lanes of a group, so that few
// results occupy many warps; the lanes' sums meet in shuffles. Positions of a blend are spread over up to eight lanes likewise.
// Bound: the latencies of the chain (dependent loads and FMAs at about 3 cycles per instruction, 12 warps or 24 alike).
// us per call, a block per unit with four rounds of block barriers -> now: 256 tokens, M = B = 16, d = 64, k = 5 76 -> 41 (8 CTAs per unit;
// of 4 47, of 2 56, one 66; 148 units, one each 81 -> 69); 777 tokens of 8 units, M = 48, B = 100 180 (launches) -> 72 (10 CTAs).
#include <algorithm>
#include <atomic>
#include <cmath>
#include <type_traits>

#include "common.cuh"
#include "handle.h"
#include "simt.cuh"

namespace lococo {
namespace {

using namespace simt;

constexpr int kThreads = 512, kWarps = kThreads / 32;
constexpr int kMaxSmem = 232448 - 128;   // dynamic shared memory: 227 KB less the kernel's few static words

struct LoopParams {
    View q, k, v, o, k_cache, v_cache;
    int heads, d, M, k_taps, c_in, L, B, c0, weights_per_head, prot;
    const float* g_reverse;      // [sets][M][k][c_in], taps reversed
    const float* bias;           // [sets][M] or nullptr
    float eps, scale;
    float *snap_k, *snap_v;      // optional: [chunk][units][M][d]
    int64_t snap_step;           // floats between chunks
    float* lse;                  // optional: [units][L]
    int ctas;                    // CTAs per unit
    int chain_warps;             // warps 0 .. chain_warps - 1 update the cache, the others (an even number) attend
    int tile;                    // slots x positions of a convolution tile: 0, 1, 2: 4, 3, 2 x 8; 3: 2 x 4
};

__host__ __device__ inline int round4(int x) { return (x + 3) / 4 * 4; }
// Shared memory, in floats. A buffer of rows holds [zeros | cache | chunk | zeros], keys and values side by side, so that a
// row of [cache; chunk] and the convolution's padding are plain offsets; while a compress step reads one buffer the CTAs write
// the new cache into the other, where the next chunk is on its way. Row strides are padded by four so that lanes that take
// consecutive rows meet different banks.
template <int D>
struct Strides {
    static constexpr int kRow = 2 * D + 4, kQuery = D + 4;
};
struct LoopLayout {
    int MS;                      // row stride of R^T (this CTA's slots along the row)
    int rows;                    // per buffer
    int queries;                 // per buffer
    int g, x, q, p, r, total;
};
__host__ __device__ inline LoopLayout loop_layout(int d, int M, int B, int k, int c_in, int ctas, int attention_warps) {
    LoopLayout l;
    const int slots = round4((M + ctas - 1) / ctas);
    l.MS = slots + 4;
    l.rows = M + B + k - 1 + 8;
    l.queries = (B + ctas - 1) / ctas;
    int off = 0;
    l.g = off;      off += slots * k * c_in;
    l.x = off;      off += 2 * l.rows * (2 * d + 4);
    l.q = off;      off += 2 * l.queries * (d + 4);
    l.p = off;      off += attention_warps * (M + B) * 4;  // [warp][key][up to four queries]
    l.r = off;      off += (M + B + 7) * l.MS;
    l.total = off;
    return l;
}

// One row of a tile of dot products: acc[b] += over this lane's four channels x . y[(b + first) % NB]
template <int NB>
__device__ __forceinline__ void row_fma(const f32x4& x, const f32x4 (&y)[NB], int first, f32x2* acc) {
#pragma unroll
    for (int b = 0; b < NB; ++b) { fma2(x.lo, y[(b + first) % NB].lo, acc[b]); fma2(x.hi, y[(b + first) % NB].hi, acc[b]); }
}

// N floats at dst, in all CTAs of the cluster
template <int N>
__device__ __forceinline__ void store_everywhere(float* dst, const float* v, int rank, int ctas) {
    const uint32_t at = (uint32_t)__cvta_generic_to_shared(dst);
#pragma unroll 4
    for (int c = 0; c < ctas; ++c) {
        const uint32_t r = remote(at, rank + c < ctas ? rank + c : rank + c - ctas);
        if constexpr (N == 4) asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(r), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]) : "memory");
        else if constexpr (N == 2) asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(r), "f"(v[0]), "f"(v[1]) : "memory");
        else st_remote(r, v[0]);
    }
}

// N floats at an address that is a multiple of their size
template <int N>
__device__ __forceinline__ void get(const float* src, float (&v)[N]) {
    if constexpr (N == 4) *reinterpret_cast<float4*>(v) = *reinterpret_cast<const float4*>(src);
    else if constexpr (N == 2) *reinterpret_cast<float2*>(v) = *reinterpret_cast<const float2*>(src);
    else v[0] = src[0];
}
template <int N>
__device__ __forceinline__ void put(float* dst, const float (&v)[N]) {
    if constexpr (N == 4) *reinterpret_cast<float4*>(dst) = *reinterpret_cast<const float4*>(v);
    else if constexpr (N == 2) *reinterpret_cast<float2*>(dst) = *reinterpret_cast<const float2*>(v);
    else dst[0] = v[0];
}

// kLC: lanes that share a small convolution tile's channels (c_in / 4, at most 32); half as many share a large one's
template <int D, int kLC>
__global__ void __launch_bounds__(kThreads, 1) small_loop_kernel(const __grid_constant__ LoopParams P) {
    extern __shared__ __align__(16) float smem[];
    constexpr int kLD = D / 4, RS = Strides<D>::kRow, RQ = Strides<D>::kQuery;
    const int ctas = P.ctas, rank = blockIdx.x % ctas, u = blockIdx.x / ctas, n = u / P.heads, h = u % P.heads;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int M = P.M, B = P.B, k = P.k_taps, C = P.c_in, pad = (k - 1) / 2;
    const int i_begin = M * rank / ctas, slots = M * (rank + 1) / ctas - i_begin;      // this CTA's slots
    const int chain_warps = P.chain_warps, chain_threads = 32 * chain_warps;
    const LoopLayout lay = loop_layout(D, M, B, k, C, ctas, kWarps - chain_warps);
    const int MS = lay.MS;
    float *Gs = smem + lay.g, *Ps = smem + lay.p + (warp - chain_warps) * (M + B) * 4, *Rs = smem + lay.r;
    auto rows_of = [&](int buf) { return smem + lay.x + (buf * lay.rows + pad) * RS; };      // row 0 of [cache; chunk]
    auto everybody = [&] {
        if (ctas == 1) __syncthreads();
        else cluster_sync();
    };
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (int x = tid; x < 2 * lay.rows * RS / 4; x += kThreads) store4(smem + lay.x + 4 * x, make_float4(0.f, 0.f, 0.f, 0.f));
    asm volatile("griddepcontrol.wait;" ::: "memory");
    __syncthreads();

    // The attention's threads bring the chunk's keys and values into rows c .. of row buffer `buf` (zeros behind a short one), and this
    // CTA's queries (every ctas-th, so that all CTAs have early and late ones) into query buffer `qbuf`. A thread copies the
    // same four channels of every step-th row.
    const int at = tid - chain_threads, step = (kThreads - chain_threads) / (2 * kLD);
    const int row0 = at / (2 * kLD), ch0 = 4 * (at % (2 * kLD)), q_row0 = at / kLD, q_ch0 = 4 * (at % kLD);
    const View& kv = ch0 < D ? P.k : P.v;
    const float* kv_src = unit_base<float>(kv, n, h) + row0 * kv.st + (ch0 < D ? ch0 : ch0 - D);
    const float* q_src = unit_base<float>(P.q, n, h) + (rank + q_row0 * ctas) * P.q.st + q_ch0;
    const int64_t kv_step = step * kv.st, q_step = (int64_t)2 * step * ctas * P.q.st;
    auto fetch = [&](int t0, int c, int buf, int qbuf) {
        const int b = min(B, P.L - t0);
        float *rows = rows_of(buf) + c * RS, *dst = rows + row0 * RS + ch0;
        const float* src = kv_src + t0 * kv.st;
        for (int r = row0; r < b; r += step, dst += step * RS, src += kv_step) cp_async16(dst, src, true);
        dst = smem + lay.q + (qbuf * lay.queries + q_row0) * RQ + q_ch0;
        src = q_src + t0 * P.q.st;
        for (int q = rank + q_row0 * ctas; q < b; q += 2 * step * ctas, dst += 2 * step * RQ, src += q_step) cp_async16(dst, src, true);
        cp_async_commit();
        if (c + b < M + B)
            for (int x = at; x < pad * RS / 4; x += kThreads - chain_threads) store4(rows + b * RS + 4 * x, make_float4(0.f, 0.f, 0.f, 0.f));
    };
    if (at >= 0) fetch(0, P.c0, 0, 0);
    {
        const float* g = P.g_reverse + ((int64_t)(P.weights_per_head ? h * M : 0) + i_begin) * k * C;
        const int live = slots * k * C / 4, all = (MS - 4) * k * C / 4;
        for (int x = tid; x < all; x += kThreads) cp_async16(Gs + 4 * x, x < live ? g + 4 * x : g, x < live);
        for (int x = tid; x < P.c0 * 2 * kLD; x += kThreads) {
            const int r = x / (2 * kLD), q4 = x % (2 * kLD), c = 4 * (q4 % kLD);
            const View& v = q4 < kLD ? P.k_cache : P.v_cache;
            cp_async16(rows_of(0) + r * RS + 4 * q4, unit_base<float>(v, n, h) + (int64_t)r * v.st + c, true);
        }
        cp_async_commit();
    }
    const int full_queries = (B - rank + ctas - 1) / ctas, tail_queries = ((P.L - 1) % B + ctas - rank) / ctas;
    const float sc2 = P.scale * 1.4426950408889634f;
    const int n_chunks = (P.L + B - 1) / B;
    int c = P.c0, cur = 0;
    cp_async_wait<0>();
    everybody();
#pragma unroll 1
    for (int ch = 0; ch < n_chunks; ++ch) {
        // (this chunk is there, and nobody, here or in another CTA, reads the other buffers any more)
        const int t0 = ch * B, b = min(B, P.L - t0), S = c + b;
        const bool compress = S > M;
        float* X = rows_of(cur);
        if (at >= 0) {
            if (ch + 1 < n_chunks) fetch(t0 + B, compress ? M : S, compress ? cur ^ 1 : cur, (ch + 1) & 1);
            if (P.snap_k) {
                float* snap = (ch0 < D ? P.snap_k : P.snap_v - D) + ch * P.snap_step + (int64_t)u * M * D + ch0;
                for (int r = rank * step + row0; r < c; r += ctas * step) store4(snap + r * D, load4(X + r * RS + ch0));
            }
            // ---- attention: scores (in base-2 units, masked entries -inf), maximum, exponentials, O = P V / sum P
            const int queries = b == B ? full_queries : tail_queries;
            const float* qs = smem + lay.q + (ch & 1) * lay.queries * RQ;
            auto attend = [&](auto per_warp) {
                constexpr int Q = decltype(per_warp)::value;
#pragma unroll 1
                for (int g = warp - chain_warps; g * Q < queries; g += kWarps - chain_warps) {
                    const int q0 = rank + g * Q * ctas;                              // (then every ctas-th)
                    const int keys = c + min(q0 + (Q - 1) * ctas, b - 1) + 1;        // that the last of them sees
                    const float* q_row[Q];                                           // (the last query again where there are fewer)
                    float top[Q], sum[Q];
#pragma unroll
                    for (int a = 0; a < Q; ++a) { q_row[a] = qs + min(g * Q + a, queries - 1) * RQ; top[a] = -INFINITY; sum[a] = 0.f; }
#pragma unroll 1
                    for (int j = lane; j < keys; j += 32) {
                        const float* x = X + j * RS;
                        f32x2 acc[Q][2];
#pragma unroll
                        for (int a = 0; a < Q; ++a) acc[a][0] = acc[a][1] = 0ull;
#pragma unroll 4
                        for (int c4 = 0; c4 < kLD; ++c4) {
                            const f32x4 y = load_pairs(x + 4 * c4);
#pragma unroll
                            for (int a = 0; a < Q; ++a) {
                                const f32x4 w = load_pairs(q_row[a] + 4 * c4);
                                fma2(w.lo, y.lo, acc[a][0]);
                                fma2(w.hi, y.hi, acc[a][1]);
                            }
                        }
                        float s[Q];
#pragma unroll
                        for (int a = 0; a < Q; ++a) {
                            const float2 lo = unpair(acc[a][0]), hi = unpair(acc[a][1]);
                            s[a] = j <= c + q0 + a * ctas ? ((lo.x + lo.y) + (hi.x + hi.y)) * sc2 : -INFINITY;
                            top[a] = fmaxf(top[a], s[a]);
                        }
                        put<Q>(Ps + j * Q, s);
                    }
#pragma unroll
                    for (int a = 0; a < Q; ++a)
#pragma unroll
                        for (int of = 16; of; of >>= 1) top[a] = fmaxf(top[a], __shfl_xor_sync(0xffffffffu, top[a], of));
                    for (int j = lane; j < keys; j += 32) {
                        float s[Q];
                        get<Q>(Ps + j * Q, s);
#pragma unroll
                        for (int a = 0; a < Q; ++a) sum[a] += s[a] = exp2f(s[a] - top[a]);
                        put<Q>(Ps + j * Q, s);
                    }
#pragma unroll
                    for (int a = 0; a < Q; ++a)
#pragma unroll
                        for (int of = 16; of; of >>= 1) sum[a] += __shfl_xor_sync(0xffffffffu, sum[a], of);
                    __syncwarp();
                    constexpr int kParts = 32 / kLD;                         // lanes that share a channel quad take every other key
                    const int c4 = lane % kLD, part = lane / kLD;
                    f32x4 acc[Q];
#pragma unroll
                    for (int a = 0; a < Q; ++a) acc[a] = f32x4{0ull, 0ull};
                    const float *x = X + part * RS + D + 4 * c4, *pr = Ps + part * Q;
#pragma unroll 4
                    for (int j = part; j < keys; j += kParts, x += kParts * RS, pr += kParts * Q) {
                        const f32x4 v = load_pairs(x);
                        float w[Q];
                        get<Q>(pr, w);
#pragma unroll
                        for (int a = 0; a < Q; ++a) fma4(pair(w[a], w[a]), v, acc[a]);
                    }
#pragma unroll
                    for (int a = 0; a < Q; ++a) {
                        float4 v = to_float4(acc[a]);
                        if (kParts == 2) {
                            v.x += __shfl_xor_sync(0xffffffffu, v.x, 16); v.y += __shfl_xor_sync(0xffffffffu, v.y, 16);
                            v.z += __shfl_xor_sync(0xffffffffu, v.z, 16); v.w += __shfl_xor_sync(0xffffffffu, v.w, 16);
                        }
                        if (g * Q + a >= queries || part != a % kParts) continue;
                        const int q = t0 + q0 + a * ctas;
                        const float s = 1.f / sum[a];
                        store4(unit_base_mut<float>(P.o, n, h) + (int64_t)q * P.o.st + 4 * c4, make_float4(v.x * s, v.y * s, v.z * s, v.w * s));
                        if (P.lse && c4 == 0) P.lse[(int64_t)u * P.L + q] = (top[a] + log2f(sum[a])) * 0.6931471805599453f;
                    }
                    __syncwarp();
                }
            };
            // as few queries per warp as keep every warp busy once, up to four (a warp's loads of keys and values serve them all)
            const int warps = kWarps - chain_warps;
            if (queries <= warps) attend(std::integral_constant<int, 1>{});
            else if (queries <= 2 * warps) attend(std::integral_constant<int, 2>{});
            else attend(std::integral_constant<int, 4>{});
        } else if (compress) {
            // ---- Eq. 6, bias, ReLU: R^T[position][slot]
            auto convolve = [&](auto tile_slots, auto tile_positions, auto tile_lanes) {
                constexpr int TA = decltype(tile_slots)::value, TP = decltype(tile_positions)::value, kL = decltype(tile_lanes)::value;
                constexpr int kPerWarp = 32 / kL, kAll = TA == 3 ? 4 * TP : TA * TP, kOut = kAll > kL ? kAll / kL : 1;      // (powers of two)
                const int it = (slots + TA - 1) / TA, jt = (S + TP - 1) / TP, tiles = it * jt, gl = tid % kL;
                const uint32_t magic = 0xffffffffu / jt + 1;                 // t / jt = the upper half of t magic (jt > 1)
#pragma unroll 1
                for (int t0w = warp * kPerWarp; t0w < tiles; t0w += chain_warps * kPerWarp) {
                    const int t = min(t0w + lane / kL, tiles - 1);           // (the last tile twice rather than none)
                    const int ti = jt == 1 ? t : __umulhi(t, magic), i0 = TA * ti, j0 = TP * (t - ti * jt);
                    f32x2 acc[TA * TP];
#pragma unroll
                    for (int e = 0; e < TA * TP; ++e) acc[e] = 0ull;
#pragma unroll 1
                    for (int c4 = gl; c4 < C / 4; c4 += kL) {
                        const int slot = k * C;
                        const float* w = Gs + (i0 * k + k - 1) * C + 4 * c4;          // tap t of slot a: w + (a k - t) C
                        const float* x = X + (j0 - pad) * RS + 4 * c4;
                        f32x4 z[TP];                                                  // rows of the window, the first at tap % TP
#pragma unroll
                        for (int e = 0; e < TP - 1; ++e) z[e] = load_pairs(x + e * RS);
                        x += (TP - 1) * RS;
#pragma unroll 1
                        for (int tap = 0; tap < k; tap += TP) {
#pragma unroll
                            for (int e = 0; e < TP; ++e, w -= C, x += RS) {
                                if (tap + e >= k) break;
                                z[(e + TP - 1) % TP] = load_pairs(x);
#pragma unroll
                                for (int a = 0; a < TA; ++a) row_fma<TP>(load_pairs(w + a * slot), z, e, acc + TP * a);
                            }
                        }
                    }
                    float v[kAll];
#pragma unroll
                    for (int e = 0; e < kAll; ++e) { const float2 f = unpair(e < TA * TP ? acc[e] : 0ull); v[e] = f.x + f.y; }
                    reduce_lanes<kAll, kL>(v, gl);
                    const int idx = gl * kAll / kL, a = i0 + idx / TP, i = i_begin + a;
                    if (idx < TA * TP && a < slots) {
                        const float bias = P.bias ? P.bias[(P.weights_per_head ? h * M : 0) + i] : 0.f;
#pragma unroll
                        for (int e = 0; e < kOut; ++e) {
                            const int j = j0 + idx % TP + e;
                            if (j < S) Rs[j * MS + a] = i < P.prot ? (j == i ? 1.f : 0.f) : fmaxf(v[e] + bias, 0.f);
                        }
                    }
                }
            };
            using Two = std::integral_constant<int, 2>;
            using Four = std::integral_constant<int, 4>;
            using Eight = std::integral_constant<int, 8>;
            using Lanes = std::integral_constant<int, kLC>;
            using Fewer = std::integral_constant<int, kLC / 2>;
            if (P.tile == 0) convolve(Four{}, Eight{}, Fewer{});
            else if (P.tile == 1) convolve(std::integral_constant<int, 3>{}, Eight{}, Fewer{});
            else if (P.tile == 2) convolve(Two{}, Eight{}, Fewer{});
            else convolve(Two{}, Four{}, Lanes{});
            asm volatile("bar.sync 1, %0;" ::"r"(chain_threads) : "memory");
            // ---- the new rows of this CTA's slots: kRows rows x four channels per group of kParts lanes, which share the positions
            float* next = rows_of(cur ^ 1) + i_begin * RS;
            auto blend = [&](auto rows_per_group, auto lanes_per_group) {
                constexpr int kRows = decltype(rows_per_group)::value, kParts = decltype(lanes_per_group)::value;
                const int items = (slots + kRows - 1) / kRows * 2 * kLD;
#pragma unroll 1
                for (int t0w = 32 * warp; t0w < items * kParts; t0w += chain_threads) {
                    const int part = lane % kParts, t = min((t0w + lane) / kParts, items - 1);
                    const int r0 = kRows * (t / (2 * kLD)), ch4 = 4 * (t % (2 * kLD));
                    f32x4 acc[kRows];
                    float sum[kRows];
#pragma unroll
                    for (int a = 0; a < kRows; ++a) { acc[a] = f32x4{0ull, 0ull}; sum[a] = 0.f; }
                    const float *w = Rs + part * MS + r0, *x = X + part * RS + ch4;
#pragma unroll 4
                    for (int j = part; j < S; j += kParts, w += kParts * MS, x += kParts * RS) {
                        float r[kRows];
                        get<kRows>(w, r);
                        const f32x4 v = load_pairs(x);
#pragma unroll
                        for (int a = 0; a < kRows; ++a) { fma4(pair(r[a], r[a]), v, acc[a]); sum[a] += r[a]; }
                    }
                    float v[4 * kRows];
#pragma unroll
                    for (int a = 0; a < kRows; ++a) {
                        const float4 f = to_float4(acc[a]);
                        v[4 * a] = f.x; v[4 * a + 1] = f.y; v[4 * a + 2] = f.z; v[4 * a + 3] = f.w;
#pragma unroll
                        for (int m = kParts / 2; m; m >>= 1) sum[a] += __shfl_xor_sync(0xffffffffu, sum[a], m);
                    }
                    reduce_lanes<4 * kRows, kParts>(v, part);
                    constexpr int kOut = 4 * kRows / kParts, kVec = kOut < 4 ? kOut : 4;      // results of a lane, of one store
                    const int first = part * kOut;
#pragma unroll
                    for (int e = 0; e < kOut; e += kVec) {
                        const int a = (first + e) / 4, r = r0 + a;
                        float own = sum[0];                        // (no indexing by a variable)
#pragma unroll
                        for (int y = 1; y < kRows; ++y) own = a == y ? sum[y] : own;
                        if (r >= slots) break;
                        const float s = i_begin + r < P.prot ? 1.f : 1.f / (own + P.eps);
#pragma unroll
                        for (int y = 0; y < kVec; ++y) v[e + y] *= s;
                        float* dst = next + r * RS + ch4 + (first + e) % 4;
                        if (ctas > 1) store_everywhere<kVec>(dst, v + e, rank, ctas);
                        else {
#pragma unroll
                            for (int y = 0; y < kVec; ++y) dst[y] = v[e + y];
                        }
                    }
                }
            };
            // four rows per group where there are as many, and as many lanes per group as there are threads for
            auto lanes = [&](auto rows_per_group) {
                const int items = (slots + decltype(rows_per_group)::value - 1) / decltype(rows_per_group)::value * 2 * kLD;
                if (8 * items <= chain_threads) blend(rows_per_group, Eight{});
                else if (4 * items <= chain_threads) blend(rows_per_group, Four{});
                else if (2 * items <= chain_threads) blend(rows_per_group, Two{});
                else blend(rows_per_group, std::integral_constant<int, 1>{});
            };
            if (slots > 2) lanes(Four{});
            else lanes(Two{});
        }
        if (compress) {
            cur ^= 1;
            c = M;
        } else {
            c = S;                                          // fill: the chunk's rows are where they belong
        }
        cp_async_wait<0>();
        everybody();
    }
    const float* cache = rows_of(cur);
    for (int x = rank * kThreads + tid; x < c * 2 * kLD; x += ctas * kThreads) {
        const int r = x / (2 * kLD), q4 = x % (2 * kLD);
        const View& v = q4 < kLD ? P.k_cache : P.v_cache;
        store4(unit_base_mut<float>(v, n, h) + (int64_t)r * v.st + 4 * (q4 % kLD), load4(cache + r * RS + 4 * q4));
    }
}

template <int D, int kLC>
int launch_loop(const LoopParams& P, int units, size_t smem, cudaStream_t st) {
    static ClusterKernel state;
    return launch_clusters(state, small_loop_kernel<D, kLC>, kMaxSmem, P.ctas, units, kThreads, smem, st, P) ? 1 : -1;
}

ClusterKernel loop_state;      // of the kernel that is asked how many clusters fit (all forms need an SM per CTA)

}  // namespace

// The plan, and the rule: fp32, [cache; chunk] in one SM's shared memory, and a call estimated faster than as launches over the whole chip. A fill
// step is a short launch or two there, but here every cluster of a unit takes its turn; a compress step is mostly work that launches do in tiles
// of 4096 logits and blocks of 32 queries, however few are needed. Both estimates are in us:
//   here      3 + rounds of clusters x (2.6 for zeros and weights, 2.4 and the work's share per compress step, 1.5 and the attention per fill step)
//   launches  1.4 + per step the attention's rounds of one block per SM; per fill step 3.6, per compress step the convolution's and the blends' rounds
// A compress step here is fitted to 44 shapes with every cluster size each, the rest to 260 calls both ways (units 1 to 2000, M and B up to 110
// and 150, one to twelve chunks, from empty and full caches). Launches have to be estimated 15 % faster: of 220 other calls 213 went within 3 % of the
// faster way without that, the worst at twice its time, and 215 with it, the worst at 1.46 times (583 units, M = 8, one chunk of 132: 340 us by
// launches, 497 here). Launches / this, us per call: 256 tokens of one unit, M = B = 16, d = 64, k = 5 263 / 41; 777 tokens of 8 units, M = 48,
// B = 100 180 / 72; two chunks of 16 of 1600 units, M = 8, d = 128, k = 5 698 / 125; twelve chunks of 2 of 617 units, M = 54, d = 64, k = 9
// 3715 / 1759; and by launches: 8 tokens that fill a cache of 48, 32 units, d = 128 10.3 / 18.5; one of 310, M = 24 18.6 / 105.
LoopPlan simt_loop_plan(const lococo_handle* h, int L, int B, int c0) {
    const lococo_config& c = h->cfg;
    LoopPlan best{0, 0, 0};
    if (c.dtype != LOCOCO_F32) return best;
    B = std::min(B, L);
    const double S = (double)c.M + B, keys = c.M + 0.5 * B, d2 = 2.0 * c.head_dim, taps = (double)c.c_in * c.k;
    if (2.0 * S * d2 * 4 > kMaxSmem) return best;
    const int chunks = (L + B - 1) / B, fills = c0 + L <= c.M ? chunks : std::min(chunks, (c.M - c0) / B), compresses = chunks - fills;
    const double fill_keys = c0 + 0.5 * B * fills;
    double least;
    {
        const int OT = slot_tile(c.M), PT = 4096 / OT;
        const double tiles = (double)(((int)S + PT - 1) / PT) * ((c.M + OT - 1) / OT) * h->units, splits = std::max(1.0, std::min(std::floor(6 * kSMs / tiles), c.c_in / 32.0));
        const double conv = taps * std::max(1 / splits, tiles / (4 * kSMs)), blends = std::floor((S + 63) / 64) * std::max(1.0, (c.M + 15) / 16 * d2 / 64 * h->units / (6 * kSMs));
        auto attention = [&](double n) { return 3.2 * std::max(1.0, (double)h->units * ((B + 31) / 32) / kSMs) * (1 + std::floor(n / 64)) * c.head_dim / 64; };
        least = (1.4 + fills * (3.6 + attention(fill_keys)) + compresses * (0.094 * conv + 5.6 * blends + attention(S))) / 0.85;
    }
    const std::atomic<int>* resident = resident_clusters(loop_state, small_loop_kernel<64, 16>, kMaxSmem, kThreads);
    for (int ctas = 1; resident && ctas <= std::min(kMaxCluster, c.M); ctas = next_cluster(ctas)) {
        const int slots = (c.M + ctas - 1) / ctas, queries = (B + ctas - 1) / ctas, clusters = resident[ctas];
        const double conv = slots * S * taps, blends = slots * S * d2, attention = queries * keys * d2;
        LoopPlan p{ctas, std::min(12, std::max(4, 2 * (int)(0.5 * kWarps * (conv + blends) / (conv + blends + 1.3 * attention) + 0.5))), 3};
        const LoopLayout lay = loop_layout(c.head_dim, c.M, B, c.k, c.c_in, ctas, kWarps - p.chain_warps);
        if (clusters == 0 || (double)slots * taps * 4 > kMaxSmem || (size_t)lay.total * 4 > kMaxSmem) continue;
        const double compress = 2.4 + 0.025 * ctas + conv / 109e3 + blends / 240e3 + attention / 91e3, fill = 1.5 + queries * fill_keys * d2 / 9500;
        const double t = 3 + (h->units + clusters - 1) / clusters * (2.6 + compresses * compress + fills * fill);
        if (t >= least) continue;
        least = t;
        // Tiles of 2 x 4 while that is one round of the chain's lanes; else 8 positions wide, of as many slots as waste least
        const int lanes = c.head_dim == 64 && c.c_in == 64 ? 16 : 32, threads = 32 * p.chain_warps;
        if ((slots + 1) / 2 * (((int)S + 3) / 4) * lanes > threads) {
            double cost = 1e30;
            for (int a = 4; a >= 2; --a) {
                const double rounds = ((slots + a - 1) / a * (((int)S + 7) / 8) * (lanes / 2) + threads - 1) / threads;
                if (rounds * (a + 0.7) < cost) { cost = rounds * (a + 0.7); p.tile = 4 - a; }
            }
        }
        best = p;
    }
    return best;
}

int simt_loop(lococo_handle* h, const LoopPlan& plan, View q, View k, View v, int L, int B, View o, View kc, View vc, int c0, char* saved, size_t snap_step,
              size_t snap_all, cudaStream_t st) {
    const lococo_config& c = h->cfg;
    LoopParams P{};
    P.q = q; P.k = k; P.v = v; P.o = o; P.k_cache = kc; P.v_cache = vc;
    P.heads = c.heads; P.d = c.head_dim; P.M = c.M; P.k_taps = c.k; P.c_in = c.c_in; P.L = L; P.B = std::min(B, L); P.c0 = c0;
    P.weights_per_head = c.weights_per_head; P.prot = h->prot;
    P.g_reverse = reinterpret_cast<const float*>(h->ws + h->off_greverse);
    P.bias = h->has_bias ? reinterpret_cast<const float*>(h->ws + h->off_bias) : nullptr;
    P.eps = c.norm_eps;
    P.scale = h->scale;
    P.ctas = plan.ctas; P.chain_warps = plan.chain_warps; P.tile = plan.tile;
    if (saved) {
        P.snap_k = reinterpret_cast<float*>(saved);
        P.snap_v = reinterpret_cast<float*>(saved + snap_all);
        P.snap_step = (int64_t)(snap_step / sizeof(float));
        P.lse = reinterpret_cast<float*>(saved + 2 * snap_all);
    }
    const size_t smem = (size_t)loop_layout(P.d, P.M, P.B, P.k_taps, P.c_in, P.ctas, kWarps - P.chain_warps).total * 4;
    prof_begin(&h->prof, PROF_SEQUENCE, st);
    const int r = P.d == 128 ? launch_loop<128, 32>(P, h->units, smem, st)
                : P.c_in == 64 ? launch_loop<64, 16>(P, h->units, smem, st) : launch_loop<64, 32>(P, h->units, smem, st);
    prof_end(&h->prof, st);
    return r;
}

}  // namespace lococo
