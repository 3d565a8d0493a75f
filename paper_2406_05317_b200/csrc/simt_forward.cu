// CUDA-core (fp32 FMA) kernels of the LoCoCo chunk step. They serve the fp32
// storage type, whose 1e-4 tolerance rules out tensor-core input rounding, the static-scratch
// entry point and LOCOCO_PATH_SIMT. Storage type T is float or bf16; all arithmetic is fp32.
//
// A compress step is two launches: the convolution (in the chunk loop together with the step's attention, which
// does not depend on it) and the blends, which add up partial convolutions (where the channels were split over blocks),
// apply Eq. 6's bias and ReLU, form Eq. 7's denominators on the way and write the new cache. A row pass of its own in
// between runs only where somebody reads R afterwards (mixing weights on request).
#include <algorithm>

#include "common.cuh"
#include "simt.cuh"

namespace lococo {
namespace {

using namespace simt;

// ------------------------------------------------------------------ weight packing
// G [sets][M][C][k] -> Wf [set][channel][tap][slot] (the forward convolution contracts over channels and reads the slots of
// a block side by side): a plain transpose of [slot][channel, tap].
template <typename T>
__global__ void pack_forward_kernel(const T* __restrict__ G, T* __restrict__ out, int M, int rows) {
    __shared__ T tile[32][33];
    const int64_t plane = (int64_t)blockIdx.z * M * rows;
    const int r0 = blockIdx.x * 32, i0 = blockIdx.y * 32;
    for (int y = threadIdx.y; y < 32; y += blockDim.y)
        if (i0 + y < M && r0 + (int)threadIdx.x < rows) tile[y][threadIdx.x] = G[plane + (int64_t)(i0 + y) * rows + r0 + threadIdx.x];
    __syncthreads();
    for (int y = threadIdx.y; y < 32; y += blockDim.y)
        if (r0 + y < rows && i0 + (int)threadIdx.x < M) out[plane + (int64_t)(r0 + y) * M + i0 + threadIdx.x] = tile[threadIdx.x][y];
}
// G [sets][M][C][k] -> Wb [set][slot][k-1-tap][channel] (its gradient contracts over slots, with the taps reversed). A block
// takes one slot: its C x k values come in as they lie and leave transposed.
template <typename T>
__global__ void pack_reverse_kernel(const T* __restrict__ G, T* __restrict__ out, int C, int k) {
    extern __shared__ __align__(16) unsigned char raw[];
    T* tile = reinterpret_cast<T*>(raw);
    const int64_t base = (int64_t)blockIdx.x * C * k;
    for (int x = threadIdx.x; x < C * k; x += blockDim.x) tile[x] = G[base + x];
    __syncthreads();
    for (int x = threadIdx.x; x < C * k; x += blockDim.x) {
        const int ch = x % C, t = x / C;
        out[base + x] = tile[ch * k + k - 1 - t];
    }
}

template <typename T>
__global__ void to_f32_kernel(const T* __restrict__ in, float* __restrict__ out, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = to_f32(in[i]);
}

// ------------------------------------------------------------------ fill branch
template <typename T>
__global__ void fill_kernel(FillParams p) {
    if (!p.late) start_next();
    wait_for_previous();
    const int u = blockIdx.y, n = u / p.heads, h = u % p.heads;
    const int vec = 16 / sizeof(T), per_row = p.d / vec;
    const int total = p.b * per_row;
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < total; x += gridDim.x * blockDim.x) {
        const int r = x / per_row, v = x % per_row;
        const int4* sk = reinterpret_cast<const int4*>(unit_base<T>(p.src_k, n, h) + (int64_t)r * p.src_k.st) + v;
        const int4* sv = reinterpret_cast<const int4*>(unit_base<T>(p.src_v, n, h) + (int64_t)r * p.src_v.st) + v;
        int4* dk = reinterpret_cast<int4*>(unit_base_mut<T>(p.dst_k, n, h) + (int64_t)(p.c + r) * p.dst_k.st) + v;
        int4* dv = reinterpret_cast<int4*>(unit_base_mut<T>(p.dst_v, n, h) + (int64_t)(p.c + r) * p.dst_v.st) + v;
        *dk = *sk;
        *dv = *sv;
    }
}

// ------------------------------------------------------------------ Eq. 1, chunk form
// One block of 256 threads per 32 queries of a unit: two groups of 128 take every other tile of 48 keys, each with its own
// running maximum, sum and output, and meet at the end. A thread computes 4 queries x 3 keys of the scores
// (per 4 channels 7 vector loads from shared memory for 48 FMAs) and 4 queries x D/16 channels of the output; the sixteen
// threads of a query group meet in shuffles. Keys and values take turns in one buffer. (With one group
// per query tile the longest attention block of a step outlasted everything else on the chip: 8 heads of 128, 640 keys,
// 200 us for a launch whose FMAs take 60.)
// (Four threads per query, each with a quarter of its channels, needed one vector load per 4 FMAs.)
template <int D>
struct AttnSmem {
    static constexpr int kKeys = 48, kPRow = kKeys + 4;
    static constexpr int kQ = 32 * (D + 4), kKV = kKeys * (D + 4), kP = 32 * kPRow;
    static constexpr int kFloats = kQ + 2 * (kKV + kP);
};

template <typename T, int D>
__device__ __forceinline__ void attention_body(const AttnParams& p, float* smem, int qtile, int u) {
    constexpr int RS = D + 4;                  // row stride: rows of consecutive threads fall into different banks
    constexpr int NC = D / 64;                 // float4 groups of output channels per thread
    constexpr int KT = AttnSmem<D>::kKeys, PR = AttnSmem<D>::kPRow, NK = KT / 16;
    float* Qs = smem;
    const int group = threadIdx.x >> 7;
    float* KVs = Qs + AttnSmem<D>::kQ + group * (AttnSmem<D>::kKV + AttnSmem<D>::kP);
    float* Ps = KVs + AttnSmem<D>::kKV;        // [32 queries][KT keys], row stride PR
    const int n = u / p.heads, h = u % p.heads;
    const int tid = threadIdx.x & 127, tk = tid & 15, tq = tid >> 4;
    const int r0 = qtile * 32;
    const float sc = p.scale * 1.4426950408889634f;  // logits in base-2 units
    const int S = p.c + p.b;
    const int last_row = min(r0 + 31, p.b - 1);
    const int ncols = p.c + last_row + 1;      // columns any query of this block can see

    for (int x = threadIdx.x; x < 32 * (D / 4); x += 256) {
        const int r = x / (D / 4), q4 = x % (D / 4);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r0 + r < p.b) v = load4(unit_base<T>(p.q, n, h) + (int64_t)(r0 + r) * p.q.st + 4 * q4);
        *reinterpret_cast<float4*>(Qs + r * RS + 4 * q4) = make_float4(v.x * sc, v.y * sc, v.z * sc, v.w * sc);
    }
    auto stage = [&](const CatView& x, int j0) {
        for (int e = tid; e < KT * (D / 4); e += 128) {
            const int r = e / (D / 4), q4 = e % (D / 4);
            const int j = j0 + r;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (j < S) v = load4(cat_row<T>(x, n, h, j) + 4 * q4);
            *reinterpret_cast<float4*>(KVs + r * RS + 4 * q4) = v;
        }
    };
    __syncthreads();
    float m[4], l[4];
    f32x4 o[4][NC];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        m[a] = -INFINITY;
        l[a] = 0.f;
#pragma unroll
        for (int c = 0; c < NC; ++c) o[a][c] = f32x4{0ull, 0ull};
    }
#pragma unroll 1
    for (int j0 = group * KT; j0 < ncols; j0 += 2 * KT) {
        group_sync(1 + group);
        stage(p.xk, j0);
        group_sync(1 + group);
        f32x2 s2[4][NK];                       // sums over the even and over the odd channels
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < NK; ++b) s2[a][b] = 0ull;
#pragma unroll 2
        for (int d4 = 0; d4 < D / 4; ++d4) {
            f32x4 q[4], kk[NK];
#pragma unroll
            for (int a = 0; a < 4; ++a) q[a] = load_pairs(Qs + (4 * tq + a) * RS + 4 * d4);
#pragma unroll
            for (int b = 0; b < NK; ++b) kk[b] = load_pairs(KVs + (tk + 16 * b) * RS + 4 * d4);
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < NK; ++b) { fma2(q[a].lo, kk[b].lo, s2[a][b]); fma2(q[a].hi, kk[b].hi, s2[a][b]); }
        }
        float s[4][NK];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < NK; ++b) { const float2 f = unpair(s2[a][b]); s[a][b] = f.x + f.y; }
        // softmax of this tile: running maximum and sum per query
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int vis = p.c + r0 + 4 * tq + a + 1;           // columns this query sees
            float tmax = -INFINITY;
#pragma unroll
            for (int b = 0; b < NK; ++b) {
                if (j0 + tk + 16 * b >= min(vis, S)) s[a][b] = -INFINITY;
                tmax = fmaxf(tmax, s[a][b]);
            }
#pragma unroll
            for (int of = 8; of; of >>= 1) tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, of));
            // (the second group's first tile may hold no key a query sees: its maximum stays -inf, its terms come out as zeros)
            const float mnew = fmaxf(m[a], tmax), base = mnew == -INFINITY ? 0.f : mnew;
            const float corr = exp2f(m[a] - base);
            float sum = 0.f;
#pragma unroll
            for (int b = 0; b < NK; ++b) {
                const float e = exp2f(s[a][b] - base);
                sum += e;
                Ps[(4 * tq + a) * PR + tk + 16 * b] = e;
            }
            l[a] = fmaf(l[a], corr, sum);
            m[a] = mnew;
#pragma unroll
            for (int c = 0; c < NC; ++c) { mul2(pair(corr, corr), o[a][c].lo); mul2(pair(corr, corr), o[a][c].hi); }
        }
        group_sync(1 + group);
        stage(p.xv, j0);
        group_sync(1 + group);
#pragma unroll 2
        for (int k4 = 0; k4 < KT / 4; ++k4) {
            float4 pr[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) pr[a] = *reinterpret_cast<const float4*>(Ps + (4 * tq + a) * PR + 4 * k4);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const f32x4 v = load_pairs(KVs + (4 * k4 + e) * RS + 64 * c + 4 * tk);
#pragma unroll
                    for (int a = 0; a < 4; ++a) {
                        const float w = e == 0 ? pr[a].x : e == 1 ? pr[a].y : e == 2 ? pr[a].z : pr[a].w;
                        fma4(pair(w, w), v, o[a][c]);
                    }
                }
            }
        }
    }
    // the second group's (maximum, sum, output) of every query through shared memory
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int of = 8; of; of >>= 1) l[a] += __shfl_xor_sync(0xffffffffu, l[a], of);
    group_sync(1 + group);
    float* rec = Qs + AttnSmem<D>::kQ + AttnSmem<D>::kKV + AttnSmem<D>::kP;      // the second group's own buffers: [32][D], [32][2]
    if (group == 1) {
#pragma unroll
        for (int a = 0; a < 4; ++a) {
#pragma unroll
            for (int c = 0; c < NC; ++c) *reinterpret_cast<float4*>(rec + (4 * tq + a) * RS + 64 * c + 4 * tk) = to_float4(o[a][c]);
            if (tk == 0) {
                rec[32 * RS + 2 * (4 * tq + a)] = m[a];
                rec[32 * RS + 2 * (4 * tq + a) + 1] = l[a];
            }
        }
    }
    __syncthreads();
    if (group == 1) return;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const int r = r0 + 4 * tq + a;
        if (r >= p.b) continue;
        const float m1 = rec[32 * RS + 2 * (4 * tq + a)], l1 = rec[32 * RS + 2 * (4 * tq + a) + 1];
        const float mt = fmaxf(m[a], m1);                        // (m[a] is finite: every query sees key 0)
        const float w0 = exp2f(m[a] - mt), w1 = exp2f(m1 - mt), lt = l[a] * w0 + l1 * w1;
        const float inv0 = w0 / lt, inv1 = w1 / lt;
        T* orow = unit_base_mut<T>(p.o, n, h) + (int64_t)r * p.o.st;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const float4 v = to_float4(o[a][c]), w = *reinterpret_cast<const float4*>(rec + (4 * tq + a) * RS + 64 * c + 4 * tk);
            store4(orow + 64 * c + 4 * tk, make_float4(v.x * inv0 + w.x * inv1, v.y * inv0 + w.y * inv1, v.z * inv0 + w.z * inv1, v.w * inv0 + w.w * inv1));
        }
        if (p.lse && tk == 0) p.lse[(int64_t)u * p.lse_stride + r] = (mt + log2f(lt)) * 0.6931471805599453f;
    }
}

// ------------------------------------------------------------------ one launch: attention and convolution of a step
// Step 3 (Eq. 1 with the old cache) and the convolution of Step 4 read the same inputs and do not depend on each other.
// Blocks 0 .. n_attn-1: attention, the query tiles with the most keys first; then the convolution, two tiles per block.
struct StepParams {
    AttnParams a;
    CompressParams c;
    int n_attn, n_conv;
};
template <typename T, int D, int OT>
__global__ void __launch_bounds__(256, 2) step_kernel(const __grid_constant__ StepParams P) {
    extern __shared__ __align__(16) float smem[];
    if ((int)blockIdx.x < P.n_attn) start_next();         // (the blends take their places once the convolution's blocks are gone)
    wait_for_previous();
    if ((int)blockIdx.x < P.n_attn) {
        const int qtiles = (P.a.b + 31) / 32;
        attention_body<T, D>(P.a, smem, qtiles - 1 - (int)blockIdx.x / P.a.units, blockIdx.x % P.a.units);
    } else {
        const int group = threadIdx.x >> 7, tile = 2 * (blockIdx.x - P.n_attn) + group;
        if (tile < P.n_conv) conv_body<T, OT>(P.c, smem + group * (WindowConv<T, OT>::smem_bytes(P.c.k) / 4), tile, threadIdx.x & 127, group);
    }
}

// ------------------------------------------------------------------ bias, ReLU
// One warp per (unit, slot) row: the finished logits in the first partial sum's place.
__global__ void __launch_bounds__(256) relu_kernel(CompressParams p) {
    start_and_wait();
    const int row = blockIdx.x * 8 + threadIdx.x / 32;
    if (row >= p.units * p.M) return;
    const LogitRow R(p, row);
    float* r = p.R + (int64_t)row * p.Sr;
    for (int j = threadIdx.x % 32; j < p.S; j += 32) r[j] = R.at(j);
}

// ------------------------------------------------------------------ Eq. 4, Eq. 5
// new cache = R [X_K | X_V] / s (the division commutes with the sum), s the row sums of R + eps (a protected slot's row is a
// unit row and its denominator exactly 1, so it keeps its entry bit for bit). A block takes 16 slots x 64 of the 2 D channels; its
// four groups of 64 threads take every fourth tile of 16 positions (4 slots x 4 channels per thread) and meet in shared
// memory at the end. With `to_cache` 0 (the output cache IS the input cache: other blocks still read it) the unnormalised
// blends go to p.UK, p.UV and finalize_cache_kernel writes the cache.
template <typename T, int D>
__global__ void __launch_bounds__(256) blend_kernel(CompressParams p, int to_cache) {
    __shared__ __align__(16) float Xs[4][16][64];
    __shared__ __align__(16) float Rs[4][16][16];      // [group][position][slot]
    wait_for_previous();
    const int u = blockIdx.z, n = u / p.heads, h = u % p.heads;
    const int i0 = blockIdx.x * 16, cb = blockIdx.y * 64;
    const bool is_v = cb >= D;
    const CatView& x = is_v ? p.xv : p.xk;
    const int ch0 = is_v ? cb - D : cb;
    const int tid = threadIdx.x, g = tid >> 6, t = tid & 63, tc = t & 15, ts = t >> 4;
    __shared__ float row_sum[16][16];                  // [slot][group, position quad]
    float4 acc[4];
    float part = 0.f;                                  // this thread's share of its slot's row sum
#pragma unroll
    for (int a = 0; a < 4; ++a) acc[a] = make_float4(0.f, 0.f, 0.f, 0.f);
    const int rounds = (p.S + 63) / 64;
    const LogitRow row(p, u * p.M + min(i0 + (t >> 2), p.M - 1));
    float4 xr[4], rr;
    auto fetch = [&](int round) {
        const int p0 = (round * 4 + g) * 16;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int j = p0 + ts + 4 * e;
            xr[e] = j < p.S ? load4(cat_row<T>(x, n, h, j) + ch0 + 4 * tc) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        const int j = p0 + 4 * (t & 3);
        rr = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i0 + (t >> 2) < p.M && j < p.S) {
            if ((p.Sr & 3) == 0) rr = row.at4(j);
            else rr = make_float4(row.at(j), j + 1 < p.S ? row.at(j + 1) : 0.f, j + 2 < p.S ? row.at(j + 2) : 0.f, j + 3 < p.S ? row.at(j + 3) : 0.f);
            part += rr.x + rr.y + rr.z + rr.w;
        }
    };
    fetch(0);
#pragma unroll 1
    for (int round = 0; round < rounds; ++round) {
        __syncthreads();
#pragma unroll
        for (int e = 0; e < 4; ++e) *reinterpret_cast<float4*>(&Xs[g][ts + 4 * e][4 * tc]) = xr[e];
        const int q = 4 * (t & 3), sl = t >> 2;
        Rs[g][q][sl] = rr.x; Rs[g][q + 1][sl] = rr.y; Rs[g][q + 2][sl] = rr.z; Rs[g][q + 3][sl] = rr.w;
        __syncthreads();
        if (round + 1 < rounds) fetch(round + 1);
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const float4 v = *reinterpret_cast<const float4*>(&Xs[g][j][4 * tc]);
            const float4 w = *reinterpret_cast<const float4*>(&Rs[g][j][4 * ts]);
            axpy4(w.x, v, acc[0]); axpy4(w.y, v, acc[1]); axpy4(w.z, v, acc[2]); axpy4(w.w, v, acc[3]);
        }
    }
    __syncthreads();
#pragma unroll
    for (int a = 0; a < 4; ++a) *reinterpret_cast<float4*>(&Xs[g][4 * ts + a][4 * tc]) = acc[a];
    row_sum[t >> 2][4 * g + (t & 3)] = part;
    __syncthreads();
    const int sl = tid >> 4, i = i0 + sl;              // one slot, four channels per thread
    if (i >= p.M) return;
    float4 v = *reinterpret_cast<const float4*>(&Xs[0][sl][4 * tc]);
#pragma unroll
    for (int e = 1; e < 4; ++e) {
        const float4 w = *reinterpret_cast<const float4*>(&Xs[e][sl][4 * tc]);
        v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
    }
    float s = 0.f;                                     // the sixteen shares in pairs (rounding errors of a tree, not of a chain)
    {
        float t[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) t[e] = (row_sum[sl][4 * e] + row_sum[sl][4 * e + 1]) + (row_sum[sl][4 * e + 2] + row_sum[sl][4 * e + 3]);
        s = (t[0] + t[1]) + (t[2] + t[3]) + p.eps;
    }
    if (i < p.prot) s = 1.f;
    if (blockIdx.y == 0 && tc == 0) p.s[(int64_t)u * p.M + i] = s;
    if (to_cache) {
        const float inv = 1.f / s;
        const View& out = is_v ? p.v_out : p.k_out;
        store4(unit_base_mut<T>(out, n, h) + (int64_t)i * out.st + ch0 + 4 * tc, make_float4(v.x * inv, v.y * inv, v.z * inv, v.w * inv));
    } else {
        *reinterpret_cast<float4*>((is_v ? p.UV : p.UK) + ((int64_t)u * p.M + i) * D + ch0 + 4 * tc) = v;
    }
}

// new cache = U / s (Eq. 7 applied after the blend).
template <typename T>
__global__ void finalize_cache_kernel(CompressParams p) {
    start_and_wait();
    const int u = blockIdx.y, n = u / p.heads, h = u % p.heads;
    const int per_row = p.d / 4, total = p.M * per_row;
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < total; x += gridDim.x * blockDim.x) {
        const int i = x / per_row, ch = 4 * (x % per_row);
        const float inv = 1.f / p.s[(int64_t)u * p.M + i];
        const int64_t src = ((int64_t)u * p.M + i) * p.d + ch;
        const float4 a = *reinterpret_cast<const float4*>(p.UK + src), b = *reinterpret_cast<const float4*>(p.UV + src);
        store4(unit_base_mut<T>(p.k_out, n, h) + (int64_t)i * p.k_out.st + ch, make_float4(a.x * inv, a.y * inv, a.z * inv, a.w * inv));
        store4(unit_base_mut<T>(p.v_out, n, h) + (int64_t)i * p.v_out.st + ch, make_float4(b.x * inv, b.y * inv, b.z * inv, b.w * inv));
    }
}

__global__ void write_weights_kernel(const float* __restrict__ R, const float* __restrict__ s, float* __restrict__ W,
                                     int64_t rows, int S, int Sr) {
    const int64_t total = rows * S;
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < total; x += (int64_t)gridDim.x * blockDim.x)
        W[x] = R[(x / S) * Sr + x % S] / s[x / S];
}

template <typename F>
int checked(F&& launch) {
    launch();
    return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

template <typename T, int D, int OT>
int launch_step(const StepParams& P, int blocks, cudaStream_t st) {
    const size_t conv = 2 * WindowConv<T, OT>::smem_bytes(P.c.k), attn = sizeof(float) * AttnSmem<D>::kFloats;
    const size_t smem = P.n_attn == 0 ? conv : (P.n_attn == blocks ? attn : std::max(conv, attn));
    static bool done[64] = {};
    if (!smem_limit(step_kernel<T, D, OT>, 112 * 1024, done)) return -1;
    return launch_after(step_kernel<T, D, OT>, dim3(blocks), dim3(256), smem, st, P) ? 1 : -1;
}
template <typename T, int D>
int launch_step_tiles(const StepParams& P, int M, int blocks, cudaStream_t st) {
    switch (slot_tile(M)) {
        case 64: return launch_step<T, D, 64>(P, blocks, st);
        case 32: return launch_step<T, D, 32>(P, blocks, st);
        default: return launch_step<T, D, 16>(P, blocks, st);
    }
}

// Convolution, with the attention `a` in the same launch or without (a == nullptr).
template <typename T>
int convolution(const AttnParams* a, const CompressParams& p, cudaStream_t st) {
    StepParams P{};
    P.c = p;
    if (a) {
        P.a = *a;
        P.n_attn = (a->b + 31) / 32 * a->units;
    }
    P.n_conv = conv_tiles(p);
    const int blocks = P.n_attn + (P.n_conv + 1) / 2;
    prof_begin(p.prof, a ? 2 : 0, st);
    const int rc = p.d == 128 ? launch_step_tiles<T, 128>(P, p.M, blocks, st) : launch_step_tiles<T, 64>(P, p.M, blocks, st);
    prof_end(p.prof, st);
    return rc;
}

template <typename T>
int blends(const CompressParams& p, cudaStream_t st) {
    const bool in_place = p.k_out.ptr == p.xk.cache.ptr || p.v_out.ptr == p.xv.cache.ptr;
    dim3 grid((p.M + 15) / 16, 2 * p.d / 64, p.units);
    if (!(p.d == 128 ? launch_after(blend_kernel<T, 128>, grid, dim3(256), 0, st, p, in_place ? 0 : 1)
                     : launch_after(blend_kernel<T, 64>, grid, dim3(256), 0, st, p, in_place ? 0 : 1)))
        return -1;
    if (!in_place) return 1;
    return launch_after(finalize_cache_kernel<T>, dim3((p.M * p.d / 4 + 255) / 256, p.units), dim3(256), 0, st, p) ? 2 : -1;
}

template <typename T>
int compress_typed(const AttnParams* a, CompressParams p, cudaStream_t st) {
    p.splits = conv_splits(p);
    const int n = convolution<T>(a, p, st);
    const int m = n < 0 ? -1 : blends<T>(p, st);
    if (m < 0) return -1;
    if (!p.W_out) return n + m;
    if (!launch_after(relu_kernel, dim3((p.units * p.M + 7) / 8), dim3(256), 0, st, p)) return -1;
    const int w = simt_write_weights(p.R, p.s, p.W_out, (int64_t)p.units * p.M, p.S, p.Sr, st);
    return w < 0 ? -1 : n + m + 1 + w;
}

template <typename T>
int attention_typed(const AttnParams& p, cudaStream_t st) {
    StepParams P{};
    P.a = p;
    P.n_attn = (p.b + 31) / 32 * p.units;
    prof_begin(p.prof, 1, st);
    const int rc = p.d == 128 ? launch_step<T, 128, 64>(P, P.n_attn, st) : launch_step<T, 64, 64>(P, P.n_attn, st);
    prof_end(p.prof, st);
    return rc;
}

template <typename T>
int pack_typed(const T* G, T* forward, T* reverse, int sets, int M, int C, int k, cudaStream_t st) {
    int n = 0;
    if (forward) {
        if (checked([&] { pack_forward_kernel<T><<<dim3((C * k + 31) / 32, (M + 31) / 32, sets), dim3(32, 8), 0, st>>>(G, forward, M, C * k); }) < 0) return -1;
        ++n;
    }
    if (reverse) {
        static bool done[64] = {};
        if (!smem_limit(pack_reverse_kernel<T>, 256 * 63 * (int)sizeof(T), done)) return -1;
        if (checked([&] { pack_reverse_kernel<T><<<sets * M, 256, (size_t)C * k * sizeof(T), st>>>(G, reverse, C, k); }) < 0) return -1;
        ++n;
    }
    return n;
}

}  // namespace

// ------------------------------------------------------------------ host launchers
int simt_pack_weights(int dtype, const void* G, void* forward, void* reverse, int sets, int M, int c_in, int k, cudaStream_t st) {
    if (dtype == LOCOCO_F32) return pack_typed((const float*)G, (float*)forward, (float*)reverse, sets, M, c_in, k, st);
    return pack_typed((const __nv_bfloat16*)G, (__nv_bfloat16*)forward, (__nv_bfloat16*)reverse, sets, M, c_in, k, st);
}

int simt_convert_bias(int dtype, const void* bias, float* out, int n, cudaStream_t st) {
    const int blocks = (n + 255) / 256;
    if (dtype == LOCOCO_F32) return checked([&] { to_f32_kernel<float><<<blocks, 256, 0, st>>>((const float*)bias, out, n); });
    return checked([&] { to_f32_kernel<__nv_bfloat16><<<blocks, 256, 0, st>>>((const __nv_bfloat16*)bias, out, n); });
}

int simt_fill(int dtype, const FillParams& p, cudaStream_t st) {
    const int vec = dtype == LOCOCO_F32 ? 4 : 8;
    const int total = p.b * (p.d / vec);
    dim3 grid((total + 255) / 256, p.units);
    return (dtype == LOCOCO_F32 ? launch_after(fill_kernel<float>, grid, dim3(256), 0, st, p)
                                : launch_after(fill_kernel<__nv_bfloat16>, grid, dim3(256), 0, st, p)) ? 1 : -1;
}

size_t simt_R_floats(int units, int M, int Smax, int c_in) {
    // one set of logits, and as many partial ones as conv_splits asks for (splits * tiles <= six tiles of 4096 per SM)
    const size_t one = (size_t)units * M * ((Smax + 3) / 4 * 4);
    return std::min(one * std::max(1, c_in / 32), std::max(one, (size_t)6 * kSMs * 4096));
}

int simt_write_weights(const float* R, const float* s, float* W, int64_t rows, int S, int Sr, cudaStream_t st) {
    const int64_t total = rows * S;
    const int blocks = (int)((total + 255) / 256 < 8192 ? (total + 255) / 256 : 8192);
    return checked([&] { write_weights_kernel<<<blocks, 256, 0, st>>>(R, s, W, rows, S, Sr); });
}

int simt_compress(int dtype, const CompressParams& p, cudaStream_t st) {
    return dtype == LOCOCO_F32 ? compress_typed<float>(nullptr, p, st) : compress_typed<__nv_bfloat16>(nullptr, p, st);
}

int simt_chunk_step(int dtype, const AttnParams& a, const CompressParams& p, cudaStream_t st) {
    return dtype == LOCOCO_F32 ? compress_typed<float>(&a, p, st) : compress_typed<__nv_bfloat16>(&a, p, st);
}

int simt_attention(int dtype, const AttnParams& p, cudaStream_t st) {
    return dtype == LOCOCO_F32 ? attention_typed<float>(p, st) : attention_typed<__nv_bfloat16>(p, st);
}

}  // namespace lococo
