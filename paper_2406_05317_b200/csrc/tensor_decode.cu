// The generation stage (Section 3.3: chunks of ONE token on a full cache) on the tensor cores: attention of the one query
// and the cache update of a step in one kernel, bf16, d = 128, M = 128 slots, c_in = d.
//
// S = M + 1 = 129 positions are one tile of 144 columns per unit; a step is the convolution's 21 weight tiles of 32 KB
// against it, and everything else is latency. What the kernel does about either:
//  - more units than SMs: two CTAs per SM, one unit each, in half an SM's shared memory and TMEM (decode_shared_kernel): while one
//    waits for rows, exchanges or stores, the other's MMAs (72 cycles each at N = 144) have the tensor pipe. (One CTA of two units per SM,
//    a weight tile for both, halves the weights' traffic but puts its latencies one after the other. Per step of a graph of 100, k = 21: 150 units 27.1 -> 24.8 us,
//    296 28.9 -> 26.9, 300 51.4 -> 39.2, 512 52.7 -> 47.3 (a step that is waited for 53.3 -> 50.9), 1536 153 -> 131; k = 5: 150 18.7 -> 16.6, 512 37.0 -> 30.4. Bound now, by count: shared memory,
//    whose 128 bytes per cycle an MMA's operands and the arriving weights take for about 100 of its cycles);
//  - few units: a unit is shared by a cluster of 2 or 4 CTAs. Each takes its share of the taps, with its weight tiles
//    requested before the kernel waits for anything; the partial logits meet through distributed shared memory (a CTA
//    finishes 72, or 40 / 32, of the columns), R goes to all CTAs of the cluster, and each blends its own part of the
//    256 key and value channels: no blend is summed across CTAs. One CTA per unit took 13 us from its key tile to the
//    last store, 8.4 us of it MMAs;
//  - the query's attention is done by warps that have nothing to do while the convolution runs, straight from the cache
//    rows in L2. All reads of a unit's cache thus belong to its own CTA or cluster, and the new rows go IN PLACE: no second
//    cache, no copy back (12 us per step at 512 units).
// The key tile comes in by the tensor copy engine: rows -pad .. 127 of the cache (rows before 0 arrive as zeros) and 16
// rows of the chunk (one valid, the others zeros), side by side as 64-channel halves of 128-byte swizzled rows; a tap is a
// row offset. Rows that only columns beyond S read hold whatever is there.
#include <algorithm>
#include <atomic>

#include "handle.h"
#include "simt.cuh"
#include "tc_common.cuh"
#include "tensor_maps.cuh"

namespace lococo {
namespace {

using namespace tc;

constexpr int kSlots = 128, kD = 128, kThreads = 384;
constexpr int kCols = 144;                        // S = 129, rounded up to the MMA's step
constexpr uint32_t kStage = 32768;                // one tap: 128 slots x 128 channels
constexpr uint32_t kRBytes = kCols / 8 * 2048u;   // R: [position group][slot][8 positions], bf16
constexpr uint32_t kVHalf = kCols * 128u;         // 144 rows x 64 channels
constexpr int kMaxSmem = 232448 - 128;
constexpr int kRec = 4 + kD;                      // attention record of a warp: maximum, sum, -, -, 128 outputs

struct alignas(64) DecodeParams {
    CUtensorMap k_cache, k_chunk, v_cache, v_chunk, k_out, v_out;
    View q, o, kc, vc, kn, vn;
    const __nv_bfloat16* gimage;                  // [sets][tap][16][128][8]
    const float* bias;
    float* lse;
    int64_t lse_stride;
    float eps, scale;
    int heads, units, k, prot, weights_per_head;
    int* status;
};

// columns [col_begin(r), col_begin(r + 1)) of the logits are finished by CTA r of the cluster; multiples of 8
template <int CS>
__host__ __device__ constexpr int col_begin(int r) { return CS == 1 ? r * kCols : (CS == 2 ? 72 * r : (r < 3 ? 40 * r : 112 + 32 * (r - 3))); }

template <int CS>
struct Layout {
    // bytes from a 1024-byte boundary: [X: weight ring; later R and the value tiles, at last the output boxes][key tiles][sums][barriers]
    // [attention records][clusters: the other CTAs' partial logits]
    uint32_t rows_k, half_k, stages, x, zk, sums, bars, rec, part, total;
    __host__ __device__ explicit Layout(int k) {
        const uint32_t pad = (k - 1) / 2;
        rows_k = (uint32_t)kSlots + 1 + k - 1 > pad + kCols ? (uint32_t)kSlots + k : pad + kCols;
        half_k = rows_k * 128u;
        const uint32_t v = CS == 4 ? kVHalf : 2 * kVHalf, after = kRBytes + v;
        const uint32_t records = 8u * kRec * 4u, parts = (uint32_t)(CS - 1) * (CS == 2 ? 72u : 40u) * kSlots * 4u;
        const uint32_t fixed = 2 * half_k + 3 * CS * kSlots * 4u + 256u + records + parts + 1024u;
        stages = 6;
        while (stages > 3 && stages * kStage + fixed > (uint32_t)kMaxSmem) --stages;
        x = stages * kStage > after ? stages * kStage : after;
        zk = x;
        sums = zk + 2 * half_k;
        bars = sums + 3 * CS * kSlots * 4u;
        rec = bars + 256u;
        part = bars + 256u + records;
        total = part + parts + 1024u;
    }
};

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&v)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]) : "r"(taddr) : "memory");
}

// Eq. 1 for the one query of unit u, by W warps (this is warp w of them; named barrier `bar` of 32 W threads): a warp takes
// every W-th group of eight keys, a lane four channels; the warps' (maximum, sum, output) meet in `rec`. Rows are read around
// L1: the previous step wrote them.
template <int W>
__device__ __forceinline__ void attend(const DecodeParams& P, int u, int w, float* rec, int bar) {
    const int lane = threadIdx.x & 31, n = u / P.heads, h = u % P.heads;
    auto f4 = [](uint2 x, float (&o)[4]) {
        const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&x.x));
        const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&x.y));
        o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y;
    };
    float q[4];
    f4(__ldcg(reinterpret_cast<const uint2*>(unit_base<__nv_bfloat16>(P.q, n, h)) + lane), q);
    const __nv_bfloat16* kc = unit_base<__nv_bfloat16>(P.kc, n, h) + 4 * lane;
    const __nv_bfloat16* vc = unit_base<__nv_bfloat16>(P.vc, n, h) + 4 * lane;
    const float sc2 = P.scale * 1.4426950408889634f;
    float m = -INFINITY, l = 0.f, o[4] = {0.f, 0.f, 0.f, 0.f};
    // groups of eight keys 0 .. 15 are the cache's; the seventeenth is the query's own key
#pragma unroll 1
    for (int g = w; g < 17; g += W) {
        uint2 kr[8], vr[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const bool own = g == 16;
            const int j = 8 * g + e;
            const __nv_bfloat16* kp = own ? unit_base<__nv_bfloat16>(P.kn, n, h) + 4 * lane : kc + (int64_t)j * P.kc.st;
            const __nv_bfloat16* vp = own ? unit_base<__nv_bfloat16>(P.vn, n, h) + 4 * lane : vc + (int64_t)j * P.vc.st;
            kr[e] = __ldcg(reinterpret_cast<const uint2*>(kp));
            vr[e] = __ldcg(reinterpret_cast<const uint2*>(vp));
        }
        float s[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            float k[4];
            f4(kr[e], k);
            s[e] = fmaf(q[0], k[0], fmaf(q[1], k[1], fmaf(q[2], k[2], q[3] * k[3])));
        }
#pragma unroll
        for (int of = 16; of; of >>= 1)
#pragma unroll
            for (int e = 0; e < 8; ++e) s[e] += __shfl_xor_sync(0xffffffffu, s[e], of);
        float mt = m;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            s[e] = g == 16 && e > 0 ? -INFINITY : s[e] * sc2;
            mt = fmaxf(mt, s[e]);
        }
        const float f = exp2f(m - mt);
        l *= f;
#pragma unroll
        for (int c = 0; c < 4; ++c) o[c] *= f;
        m = mt;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float p = exp2f(s[e] - m);
            float v[4];
            f4(vr[e], v);
            l += p;
#pragma unroll
            for (int c = 0; c < 4; ++c) o[c] = fmaf(p, v[c], o[c]);
        }
    }
    float* mine = rec + w * kRec;
    if (lane == 0) { mine[0] = m; mine[1] = l; }
    *reinterpret_cast<float4*>(mine + 4 + 4 * lane) = make_float4(o[0], o[1], o[2], o[3]);
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(32 * W) : "memory");
    if (w == 0) {
        float ma = -INFINITY;
#pragma unroll
        for (int e = 0; e < W; ++e) ma = fmaxf(ma, rec[e * kRec]);
        float la = 0.f, r[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int e = 0; e < W; ++e) {
            const float f = exp2f(rec[e * kRec] - ma);        // (a warp without keys has maximum -inf: factor 0)
            la += rec[e * kRec + 1] * f;
            const float4 t = *reinterpret_cast<const float4*>(rec + e * kRec + 4 + 4 * lane);
            r[0] = fmaf(t.x, f, r[0]); r[1] = fmaf(t.y, f, r[1]); r[2] = fmaf(t.z, f, r[2]); r[3] = fmaf(t.w, f, r[3]);
        }
        const float inv = 1.f / la;
        reinterpret_cast<uint2*>(unit_base_mut<__nv_bfloat16>(P.o, n, h))[lane] = make_uint2(pack_bf16(r[0] * inv, r[1] * inv), pack_bf16(r[2] * inv, r[3] * inv));
        if (P.lse && lane == 0) P.lse[(int64_t)u * P.lse_stride] = (ma + log2f(la)) * 0.6931471805599453f;
    }
}

// Eight logits of columns 8 g ..: bias, ReLU, the unit row of a protected slot (Section 5.2), zeros from S = 129 on; bf16 into `out`,
// returns their sum as rounded. plain: no protected slots, no columns past the last.
__device__ __forceinline__ float finish8(const DecodeParams& P, const float (&f)[8], float bias, int g, int slot, bool plain, uint4& out) {
    const bool keep = slot < P.prot;
    uint32_t pk[4];
    float sum = 0.f;
#pragma unroll
    for (int e = 0; e < 8; e += 2) {
        __nv_bfloat162 pr;
        if (plain) {
            // round first, then clamp: rounding is monotonic and keeps zero
            pr = __hmax2(__floats2bfloat162_rn(f[e] + bias, f[e + 1] + bias), __floats2bfloat162_rn(0.f, 0.f));
        } else {
            const int j = 8 * g + e;
            float a = fmaxf(f[e] + bias, 0.f), b = fmaxf(f[e + 1] + bias, 0.f);
            if (keep) { a = j == slot ? 1.f : 0.f; b = j + 1 == slot ? 1.f : 0.f; }
            if (j > kSlots) a = 0.f;
            if (j + 1 > kSlots) b = 0.f;
            pr = __floats2bfloat162_rn(a, b);
        }
        pk[e >> 1] = *reinterpret_cast<const uint32_t*>(&pr);
        sum += __low2float(pr) + __high2float(pr);
    }
    out = make_uint4(pk[0], pk[1], pk[2], pk[3]);
    return sum;
}
// The 48 columns of warp group eg, read out in one go, into R; returns their sum.
__device__ __forceinline__ float read_out(const DecodeParams& P, uint32_t lane_addr, uint8_t* r, int eg, int slot, float bias) {
    float sum = 0.f;
    uint32_t v[3][16];
#pragma unroll
    for (int i = 0; i < 3; ++i) tmem_ld16(lane_addr + 48 * eg + 16 * i, v[i]);
    tmem_ld_wait();
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const bool plain = P.prot == 0 && 48 * eg + 16 * i + 16 <= kSlots;
#pragma unroll
        for (int y = 0; y < 2; ++y) {
            const int g = 6 * eg + 2 * i + y;
            float f[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) f[e] = __uint_as_float(v[i][8 * y + e]);
            uint4 r4;
            sum += plain ? finish8(P, f, bias, g, slot, true, r4) : finish8(P, f, bias, g, slot, false, r4);
            *reinterpret_cast<uint4*>(r + g * 2048u + slot * 16u) = r4;
        }
    }
    return sum;
}
// 32 columns of the new rows, from column c0 on, into their swizzled box of 128 slots x 64 channels.
__device__ __forceinline__ void put_rows(uint8_t* boxes, int c0, int slot, const uint32_t (&a)[32], float inv) {
    uint8_t* row = boxes + (c0 >> 6) * 16384 + slot * 128;
#pragma unroll
    for (int e = 0; e < 32; e += 8)
        *reinterpret_cast<uint4*>(row + (((((c0 & 63) + e) >> 3) ^ (slot & 7)) << 4)) =
            make_uint4(pack_bf16(__uint_as_float(a[e]) * inv, __uint_as_float(a[e + 1]) * inv), pack_bf16(__uint_as_float(a[e + 2]) * inv, __uint_as_float(a[e + 3]) * inv),
                       pack_bf16(__uint_as_float(a[e + 4]) * inv, __uint_as_float(a[e + 5]) * inv), pack_bf16(__uint_as_float(a[e + 6]) * inv, __uint_as_float(a[e + 7]) * inv));
}

// Grid: units clusters of CS CTAs. Thread 128 issues the MMAs, thread 160 feeds the weight ring, thread 192 drives the
// key and value tiles; warps 0-3 and 8-11 attend while the convolution runs; all twelve warps share the read-outs: warp w owns
// TMEM lanes (slots) 32 * (w % 4) ..., and every third group of columns.
template <int CS>
__global__ void __launch_bounds__(kThreads, 1) decode_kernel(const __grid_constant__ DecodeParams P) {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    __shared__ uint32_t tmem_slot;
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const Layout<CS> L(P.k);
    const int tid = threadIdx.x, warp = tid >> 5, eg = warp >> 2, slot = (warp & 3) * 32 + (tid & 31);
    const int rank = CS == 1 ? 0 : (int)cluster_rank();
    const int pad = (P.k - 1) / 2, NS = L.stages;
    const int u = blockIdx.x / CS, n = u / P.heads, h = u % P.heads;
    const uint32_t ring = smem_u32(smem), zk = ring + L.zk, vt = ring + kRBytes;
    float* sums = reinterpret_cast<float*>(smem + L.sums);               // [CTA of the cluster][3 groups][128 slots]
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L.bars);
    volatile int* failed = reinterpret_cast<volatile int*>(bars + 18);
    const uint32_t bar_full = smem_u32(bars), bar_empty = bar_full + 8 * 6, bar_acc = bar_empty + 8 * 6, bar_blend = bar_acc + 8, bar_k = bar_blend + 8, bar_v = bar_k + 8;
    if (warp == 4) {
        if ((tid & 31) < 16) mbar_init(bar_full + 8 * (tid & 31), 1);
        if (tid == 128) *failed = 0;
        fence_barrier_init();
    }
    if (warp == 0) {
        tmem_alloc(smem_u32(&tmem_slot), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&tmem_slot);
    if (CS > 1) cluster_arrive();         // (waited for before the first access to another CTA's shared memory)
    const __nv_bfloat16* gimg = P.gimage + (int64_t)(P.weights_per_head ? h : 0) * P.k * (kStage / 2);
    const int taps = (P.k - rank + CS - 1) / CS;                          // every CS-th tap, from tap `rank` on
    auto load_stage = [&](int it) {
        const uint32_t s = it % NS;
        if (it >= NS) mbar_wait(bar_empty + 8 * s, ((it / NS) - 1) & 1, P.status, failed, 51);
        mbar_expect_tx(bar_full + 8 * s, kStage);
        bulk_load(ring + s * kStage, gimg + (int64_t)(rank + CS * it) * (kStage / 2), kStage, bar_full + 8 * s);
    };
    // The weights were packed by an earlier call, whose kernels a later one waited for before it let this one start (the
    // signal below comes after the wait), so their first tiles may be asked for ahead of everything.
    if (warp == 5 && elect_one())
        for (int i = 0; i < min(NS, taps); ++i) load_stage(i);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    // ---- key tiles: cache rows -pad .. 127, then the chunk's row and 15 rows of zeros
    if (tid == 192) {
        mbar_expect_tx(bar_k, 2u * (kSlots + pad + 16) * 128u);
        for (int half = 0; half < 2; ++half) {
            const uint32_t dst = zk + half * L.half_k;
            tma_load_4d(dst, &P.k_cache, 64 * half, -pad, h, n, bar_k);
            tma_load_4d(dst + (kSlots + pad) * 128, &P.k_chunk, 64 * half, 0, h, n, bar_k);
        }
    }
    // ---- Eq. 6: this CTA's taps
    const uint32_t idesc_conv = instr_desc_bf16(kCols, false, false);
    if (warp == 5 && elect_one()) {
        for (int it = NS; it < taps; ++it) load_stage(it);
    } else if (warp == 4 && elect_one()) {
        const uint64_t a0 = smem_desc(ring, 2048, 128), b0 = smem_desc_sw128(zk, 16, 1024);
        const uint32_t half = L.half_k >> 4;
        mbar_wait(bar_k, 0, P.status, failed, 52);
        uint32_t st = 0, ph = 0;
        for (int it = 0; it < taps; ++it) {
            mbar_wait(bar_full + 8 * st, ph, P.status, failed, 53);
            tc_fence_after();
            const uint64_t ad = a0 + st * (kStage >> 4);
            const uint64_t bd = b0 + (uint32_t)(rank + CS * it) * 8u;         // tap t = row offset t
            umma_ss_k4(tmem, ad, bd, 256u, 2u, idesc_conv, it != 0);
            umma_ss_k4(tmem, ad + 1024u, bd + half, 256u, 2u, idesc_conv, 1);
            umma_commit(bar_empty + 8 * st);
            if (++st == (uint32_t)NS) { st = 0; ph ^= 1; }
        }
        umma_commit(bar_acc);
    }
    // ---- Eq. 1 meanwhile
    {
        float* rec = reinterpret_cast<float*>(smem + L.rec);
        if (rank == CS - 1 && (warp < 4 || warp >= 8)) attend<8>(P, u, warp < 4 ? warp : warp - 4, rec, 1);
    }
    __syncthreads();                      // the cache has been read by the attention
    mbar_wait(bar_acc, 0, P.status, failed, 54);
    tc_fence_after();
    // ---- value tiles, over the drained ring, while the accumulators are read out
    if (tid == 192) {
        const bool mine = CS == 1 || (CS == 2 ? rank == 1 : rank >= 2);
        if (mine) {
            const int halves = CS == 4 ? 1 : 2;
            mbar_expect_tx(bar_v, (uint32_t)halves * kVHalf);
            for (int e = 0; e < halves; ++e) {
                const int half = CS == 4 ? rank - 2 : e;
                tma_load_4d(vt + e * kVHalf, &P.v_cache, 64 * half, 0, h, n, bar_v);
                tma_load_4d(vt + e * kVHalf + kSlots * 128, &P.v_chunk, 64 * half, 0, h, n, bar_v);
            }
        }
    }
    const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t part = ring + L.part;                                  // partial logits of the other CTAs: [source][4 columns][slot][4]
    constexpr int kPartCols = CS == 2 ? 72 : 40;
    if constexpr (CS > 1) {
        // this CTA's partial logits of the columns that the others finish, to their shared memory
        cluster_wait();
        const int own0 = col_begin<CS>(rank) / 8, own1 = col_begin<CS>(rank + 1) / 8;
#pragma unroll 2
        for (int g = eg; g < kCols / 8; g += 3) {
            if (g >= own0 && g < own1) continue;
            int r = 0;
            while (8 * g >= col_begin<CS>(r + 1)) ++r;
            uint32_t v[8];
            tmem_ld8(lane_addr + 8 * g, v);
            tmem_ld_wait();
            if (taps == 0)                                                // (k < CS: a CTA without taps)
#pragma unroll
                for (int e = 0; e < 8; ++e) v[e] = 0u;
            const int src = rank < r ? rank : rank - 1;                   // sources of CTA r, without itself, in order
            const uint32_t dst = remote(part + ((uint32_t)((src * kPartCols + 8 * g - col_begin<CS>(r)) / 4) * kSlots + slot) * 16u, r);
            st_remote(dst, make_uint4(v[0], v[1], v[2], v[3]));
            st_remote(dst + kSlots * 16u, make_uint4(v[4], v[5], v[6], v[7]));
        }
        cluster_sync();
    }
    // ---- bias, ReLU, row sums (Eq. 7), bf16 -> A operand of the blends (in every CTA of the cluster)
    {
        {
            const float bias = P.bias ? P.bias[(P.weights_per_head ? h * kSlots : 0) + slot] : 0.f;
            if constexpr (CS == 1) {
                sums[eg * kSlots + slot] = read_out(P, lane_addr, smem, eg, slot, bias);
            } else {
                const float4* part_ptr = reinterpret_cast<const float4*>(smem + L.part) + slot;
                float sum = 0.f;
                const int g0 = col_begin<CS>(rank) / 8, g1 = col_begin<CS>(rank + 1) / 8;
#pragma unroll 2
                for (int g = g0 + eg; g < g1; g += 3) {
                    uint32_t v[8];
                    tmem_ld8(lane_addr + 8 * g, v);
                    // summed in pairs, in the order of the CTAs, this one's share in its place
                    float t[CS][8];
#pragma unroll
                    for (int s = 0; s < CS; ++s) {
                        if (s == rank) continue;
                        const float4* src = part_ptr + (int64_t)(((s < rank ? s : s - 1) * kPartCols + 8 * (g - g0)) / 4) * kSlots;
                        const float4 a = src[0], b = src[kSlots];
                        t[s][0] = a.x; t[s][1] = a.y; t[s][2] = a.z; t[s][3] = a.w;
                        t[s][4] = b.x; t[s][5] = b.y; t[s][6] = b.z; t[s][7] = b.w;
                    }
                    tmem_ld_wait();
#pragma unroll
                    for (int s = 0; s < CS; ++s)
                        if (s == rank)
#pragma unroll
                            for (int e = 0; e < 8; ++e) t[s][e] = taps > 0 ? __uint_as_float(v[e]) : 0.f;
                    float f[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) f[e] = CS == 4 ? (t[0][e] + t[1][e]) + (t[CS - 2][e] + t[CS - 1][e]) : t[0][e] + t[1][e];
                    uint4 r4;
                    sum += finish8(P, f, bias, g, slot, false, r4);
#pragma unroll
                    for (int r = 0; r < CS; ++r) st_remote(remote(ring + g * 2048u + slot * 16u, r), r4);
                }
                const uint32_t idx = (rank * 3 + eg) * kSlots + slot;
#pragma unroll
                for (int r = 0; r < CS; ++r) st_remote(remote(smem_u32(sums + idx), r), sum);
            }
        }
        asm volatile("fence.proxy.async;" ::: "memory");                  // generic writes (the other CTAs' shared memory too) before the MMAs' reads
    }
    tc_fence_before();
    if (CS > 1) cluster_sync(); else __syncthreads();
    // ---- Eq. 4, Eq. 5 (unnormalised): this CTA's channels of [K | V]
    constexpr int kN = CS == 4 ? 64 : 128;                                // columns per product
    if (warp == 4 && elect_one()) {
        asm volatile("fence.proxy.async;" ::: "memory");
        tc_fence_after();
        const uint32_t idesc = instr_desc_bf16(kN, false, true);
        auto blend = [&](uint32_t d, uint32_t b_addr, uint32_t block) {
            uint64_t ad = smem_desc(ring, 2048, 128), bd = smem_desc_sw128(b_addr, block, 1024);
#pragma unroll 1
            for (int kk = 0; kk < kCols / 16; ++kk) umma_ss(d, ad + kk * 256u, bd + kk * 128u, idesc, kk != 0);    // 16 positions: 16 rows of 128 bytes
        };
        if constexpr (CS == 1) {
            blend(tmem, zk + pad * 128, L.half_k);
            mbar_wait(bar_v, 0, P.status, failed, 55);
            tc_fence_after();
            blend(tmem + 128, vt, kVHalf);
        } else {
            const bool values = CS == 2 ? rank == 1 : rank >= 2;
            if (values) {
                mbar_wait(bar_v, 0, P.status, failed, 55);
                tc_fence_after();
                blend(tmem, vt, kVHalf);
            } else {
                blend(tmem, zk + (CS == 4 ? rank * L.half_k : 0u) + pad * 128, L.half_k);
            }
        }
        umma_commit(bar_blend);
    }
    mbar_wait(bar_blend, 0, P.status, failed, 56);
    tc_fence_after();
    // ---- Eq. 7: divide by the row sum; the rows leave in place as swizzled boxes of 128 slots x 64 channels. (The boxes take
    // R's and the values' place, which the blends have read.)
    constexpr int kBoxes = CS == 1 ? 4 : (CS == 2 ? 2 : 1);               // [K | V][64-channel halves], or this CTA's part of them
    {
        float tot = 0.f;
#pragma unroll
        for (int e = 0; e < 3 * CS; ++e) tot += sums[e * kSlots + slot];
        const float inv = slot < P.prot ? 1.f : 1.f / (tot + P.eps);      // a protected slot's row is e_i: denominator exactly 1
        // 32 columns per piece, every third piece, all of a thread's pieces requested before the first is used
        constexpr int kPieces = (2 * kBoxes + 2) / 3;
        uint32_t a[kPieces][32];
#pragma unroll
        for (int i = 0; i < kPieces; ++i)
            if (32 * (eg + 3 * i) < 64 * kBoxes) tmem_ld32(lane_addr + 32 * (eg + 3 * i), a[i]);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < kPieces; ++i)
            if (32 * (eg + 3 * i) < 64 * kBoxes) put_rows(smem, 32 * (eg + 3 * i), slot, a[i], inv);
    }
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    if (tid == 0) {
        for (int y = 0; y < kBoxes; ++y) {
            const int piece = rank * kBoxes + y;                          // of [K 0-63 | K 64-127 | V 0-63 | V 64-127]
            tma_store_4d(piece < 2 ? &P.k_out : &P.v_out, ring + y * 16384, 64 * (piece & 1), 0, h, n);
        }
        bulk_stores_read();
    }
    if (warp == 0) {
        __syncwarp();
        tmem_dealloc(tmem, 512);
    }
}

// The same step by half an SM: one CTA per unit, two CTAs per SM. What makes it fit: four ring stages of 16 KB (half a tap), 256 TMEM
// columns (the blends take the logits' columns once these are read out), and the values' second half in the place of the key
// tile once the keys are blended. Shared memory: [ring; later R and the values' first half, at last the output boxes][key tile; later the
// values' second half][sums][records][barriers]. The arithmetic, and the bits, are those of decode_kernel<1>.
struct SharedLayout {
    static constexpr uint32_t kPiece = kStage / 2, kStages = 4, kZk = kStages * kPiece, kRecords = 4u * kRec * 4u;
    uint32_t half_k, sums, rec, bars, total;
    __host__ __device__ constexpr explicit SharedLayout(int k) : half_k(0), sums(0), rec(0), bars(0), total(0) {
        const uint32_t pad = (k - 1) / 2;
        half_k = (pad + kCols) * 128u;            // (pad + 144 rows: at least the 128 + k that hold something)
        sums = kZk + 2 * half_k;
        rec = sums + 3 * kSlots * 4u;
        bars = rec + kRecords;
        total = bars + 256u + 1024u;
    }
};
constexpr int kHalfSm = 112 * 1024;               // dynamic shared memory that leaves room for a second CTA
constexpr int kMaxTaps = 27;
static_assert(SharedLayout(kMaxTaps).total <= kHalfSm, "two CTAs per SM");
__global__ void __launch_bounds__(kThreads, 2) decode_shared_kernel(const __grid_constant__ DecodeParams P) {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    __shared__ uint32_t tmem_slot;
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const SharedLayout L(P.k);
    constexpr uint32_t kPiece = SharedLayout::kPiece, NS = SharedLayout::kStages;
    const int tid = threadIdx.x, warp = tid >> 5, eg = warp >> 2, slot = (warp & 3) * 32 + (tid & 31);
    const int pad = (P.k - 1) / 2, u = blockIdx.x, n = u / P.heads, h = u % P.heads, pieces = 2 * P.k;
    const uint32_t ring = smem_u32(smem), zk = ring + SharedLayout::kZk, v0 = ring + kRBytes;
    float* sums = reinterpret_cast<float*>(smem + L.sums);               // [3 groups][128 slots]
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L.bars);
    volatile int* failed = reinterpret_cast<volatile int*>(bars + 16);
    const uint32_t bar_full = smem_u32(bars), bar_empty = bar_full + 8 * NS, bar_acc = bar_empty + 8 * NS, bar_keys = bar_acc + 8, bar_blend = bar_keys + 8, bar_k = bar_blend + 8, bar_v = bar_k + 8;
    if (warp == 4) {
        if ((tid & 31) < 16) mbar_init(bar_full + 8 * (tid & 31), 1);
        if (tid == 128) *failed = 0;
        fence_barrier_init();
    }
    if (warp == 0) {
        tmem_alloc(smem_u32(&tmem_slot), 256);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&tmem_slot);
    const __nv_bfloat16* gimg = P.gimage + (int64_t)(P.weights_per_head ? h : 0) * P.k * (kStage / 2);
    auto load_piece = [&](int it) {
        const uint32_t s = it % NS;
        if (it >= (int)NS) mbar_wait(bar_empty + 8 * s, ((it / NS) - 1) & 1, P.status, failed, 51);
        mbar_expect_tx(bar_full + 8 * s, kPiece);
        bulk_load(ring + s * kPiece, gimg + (int64_t)it * (kPiece / 2), kPiece, bar_full + 8 * s);
    };
    if (warp == 5 && elect_one())                 // (before the wait: see decode_kernel)
        for (int i = 0; i < min((int)NS, pieces); ++i) load_piece(i);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (tid == 192) {
        mbar_expect_tx(bar_k, 2u * (kSlots + pad + 16) * 128u);
        for (int half = 0; half < 2; ++half) {
            const uint32_t dst = zk + half * L.half_k;
            tma_load_4d(dst, &P.k_cache, 64 * half, -pad, h, n, bar_k);
            tma_load_4d(dst + (kSlots + pad) * 128, &P.k_chunk, 64 * half, 0, h, n, bar_k);
        }
    }
    if (warp == 5 && elect_one()) {
        for (int it = NS; it < pieces; ++it) load_piece(it);
    } else if (warp == 4 && elect_one()) {
        const uint32_t idesc_conv = instr_desc_bf16(kCols, false, false);
        const uint64_t a0 = smem_desc(ring, 2048, 128), b0 = smem_desc_sw128(zk, 16, 1024);
        mbar_wait(bar_k, 0, P.status, failed, 52);
        uint32_t st = 0, ph = 0;
        for (int it = 0; it < pieces; ++it) {
            mbar_wait(bar_full + 8 * st, ph, P.status, failed, 53);
            tc_fence_after();
            umma_ss_k4(tmem, a0 + st * (kPiece >> 4), b0 + (uint32_t)(it & 1) * (L.half_k >> 4) + (uint32_t)(it >> 1) * 8u, 256u, 2u, idesc_conv, it != 0);
            umma_commit(bar_empty + 8 * st);
            if (++st == NS) { st = 0; ph ^= 1; }
        }
        umma_commit(bar_acc);
    }
    if (warp < 4) attend<4>(P, u, warp, reinterpret_cast<float*>(smem + L.rec), 1);
    __syncthreads();                              // the cache has been read by the attention
    mbar_wait(bar_acc, 0, P.status, failed, 54);
    tc_fence_after();
    auto load_values = [&](int half, uint32_t dst) {
        mbar_expect_tx(bar_v + 8 * half, kVHalf);
        tma_load_4d(dst, &P.v_cache, 64 * half, 0, h, n, bar_v + 8 * half);
        tma_load_4d(dst + kSlots * 128, &P.v_chunk, 64 * half, 0, h, n, bar_v + 8 * half);
    };
    if (tid == 192) load_values(0, v0);           // over the drained ring, behind R
    const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    sums[eg * kSlots + slot] = read_out(P, lane_addr, smem, eg, slot, P.bias ? P.bias[(P.weights_per_head ? h * kSlots : 0) + slot] : 0.f);
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    if (warp == 4 && elect_one()) {
        tc_fence_after();
        auto blend = [&](uint32_t d, uint32_t b_addr, uint32_t block, uint32_t idesc) {
            const uint64_t ad = smem_desc(ring, 2048, 128), bd = smem_desc_sw128(b_addr, block, 1024);
#pragma unroll 1
            for (int kk = 0; kk < kCols / 16; ++kk) umma_ss(d, ad + kk * 256u, bd + kk * 128u, idesc, kk != 0);
        };
        blend(tmem, zk + pad * 128, L.half_k, instr_desc_bf16(128, false, true));
        umma_commit(bar_keys);
        for (int half = 0; half < 2; ++half) {
            mbar_wait(bar_v + 8 * half, 0, P.status, failed, 55);
            tc_fence_after();
            blend(tmem + 128 + 64 * half, half ? zk : v0, kVHalf, instr_desc_bf16(64, false, true));
        }
        umma_commit(bar_blend);
    } else if (tid == 192) {
        mbar_wait(bar_keys, 0, P.status, failed, 57);
        load_values(1, zk);                       // (the keys' blend has read the tile)
    }
    mbar_wait(bar_blend, 0, P.status, failed, 56);
    tc_fence_after();
    const float inv = slot < P.prot ? 1.f : 1.f / (sums[slot] + sums[kSlots + slot] + sums[2 * kSlots + slot] + P.eps);
#pragma unroll 1
    for (int c0 = 32 * eg; c0 < 256; c0 += 96) {
        uint32_t a[32];
        tmem_ld32(lane_addr + c0, a);
        tmem_ld_wait();
        put_rows(smem, c0, slot, a, inv);
    }
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    if (tid == 0) {
        for (int y = 0; y < 4; ++y) tma_store_4d(y < 2 ? &P.k_out : &P.v_out, ring + y * 16384, 64 * (y & 1), 0, h, n);
        bulk_stores_read();
    }
    if (warp == 0) {
        __syncwarp();
        tmem_dealloc(tmem, 256);
    }
}

// (a single token's row stride is never used, and a caller's may be one the encoder refuses)
bool rows_map(CUtensorMap* map, View v, int tokens, int heads, int batch, int box_rows) {
    if (tokens == 1) v.st = kD;
    return make_rows_map(map, v, tokens, heads, batch, box_rows, kD);
}

// Clusters of CS CTAs that the current device runs at the same time, one CTA per SM. (A cluster lies within one group of SMs, and
// the groups' sizes differ from device to device: of 148 SMs, 33 clusters of four on the B200 that was measured, 74 of two.)
template <int CS>
int resident_clusters() {
    static std::atomic<int> known[64];
    static bool done[64] = {};
    int dev = -1;
    if (!simt::smem_limit(decode_kernel<CS>, kMaxSmem, done) || cudaGetDevice(&dev) != cudaSuccess) return 0;      // (dev: below 64)
    int n = known[dev].load(std::memory_order_relaxed);
    if (n == 0) {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(CS);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = kMaxSmem;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = CS;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&n, decode_kernel<CS>, &cfg) != cudaSuccess) {
            cudaGetLastError();
            n = 0;
        }
        known[dev].store(n, std::memory_order_relaxed);
    }
    return n;
}

template <int CS>
int launch_decode(const DecodeParams& P, int clusters, bool overlap, cudaStream_t st) {
    static bool done[64] = {};
    // one CTA per SM, or (CS = 0) two: a CTA always finds its TMEM columns free
    const int smem = CS == 0 ? kHalfSm : kMaxSmem;
    void (*const kernel)(DecodeParams) = [] {
        if constexpr (CS == 0) return decode_shared_kernel;
        else return decode_kernel<CS>;
    }();
    if (!simt::smem_limit(kernel, smem, done)) return -1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(clusters * std::max(CS, 1));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int n = 0;
    if (CS > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = CS;
        attr[n].val.clusterDim.y = attr[n].val.clusterDim.z = 1;
        ++n;
    }
    if (overlap) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    if (cudaLaunchKernelEx(&cfg, kernel, P) == cudaSuccess) return 1;
    cudaGetLastError();
    return -1;
}

}  // namespace

// Chunks of one token on a full cache of one slot block. (Whether the views can be read by the copy engine shows when the
// maps are made: tensor_decode_step returns 0 and the caller takes the general step.)
bool tensor_decode_supported(const lococo_handle* h, const AttnParams& a, const CompressParams& p) {
    return h->use_tensor && !h->persistent_loop && p.d == kD && p.M == kSlots && p.c_in == kD && p.xk.c == kSlots && a.b == 1 &&
           p.W_out == nullptr && p.k <= kMaxTaps;
}

int tensor_decode_step(lococo_handle* h, const AttnParams& a, const CompressParams& p, cudaStream_t st) {
    DecodeParams P{};
    const int heads = p.heads, batch = p.units / p.heads, pad = (p.k - 1) / 2;
    if (!rows_map(&P.k_cache, p.xk.cache, kSlots, heads, batch, kSlots + pad) || !rows_map(&P.v_cache, p.xv.cache, kSlots, heads, batch, kSlots) ||
        !rows_map(&P.k_chunk, p.xk.chunk, 1, heads, batch, 16) || !rows_map(&P.v_chunk, p.xv.chunk, 1, heads, batch, 16) ||
        !rows_map(&P.k_out, p.k_out, kSlots, heads, batch, kSlots) || !rows_map(&P.v_out, p.v_out, kSlots, heads, batch, kSlots))
        return 0;
    P.q = a.q; P.o = a.o; P.kc = p.xk.cache; P.vc = p.xv.cache; P.kn = p.xk.chunk; P.vn = p.xv.chunk;
    P.gimage = reinterpret_cast<const __nv_bfloat16*>(h->ws + h->off_gimage);
    P.bias = p.bias;
    P.lse = a.lse; P.lse_stride = a.lse_stride;
    P.eps = p.eps; P.scale = a.scale;
    P.heads = heads; P.units = p.units; P.k = p.k; P.prot = p.prot; P.weights_per_head = p.weights_per_head;
    P.status = reinterpret_cast<int*>(h->ws + h->off_status);
    // Half an SM per unit once there are more units than SMs (at 148 and below, an SM each has the deeper ring: 148 units 14.5 us, 150 as
    // halves 24.8), a unit per CTA down to half the SMs, and below that clusters of 2 or 4 CTAs per unit, as many as run at the
    // same time: a second round costs a whole step (36 units
    // as clusters of four 21.5 us per step, of two 10.7; k = 21). Per step, k = 5 / 21, in a graph of 100 steps: clusters of four
    // 11.2 / 11.5 us at 33 units, of two 10.2 / 10.7 at 36 and 10.9 / 11.8 at 74, a CTA per unit 10.0 / 14.0 at 75 and
    // 10.4 / 14.5 at 148.
    const bool overlap = h->weights_settled(st);
    prof_begin(p.prof, 2, st);
    int r;
    if (p.units > kSMs) {
        r = launch_decode<0>(P, p.units, overlap, st);
    } else if (p.units <= 37 && p.units <= resident_clusters<4>()) {
        r = launch_decode<4>(P, p.units, overlap, st);
    } else if (p.units <= 74 && p.units <= resident_clusters<2>()) {
        r = launch_decode<2>(P, p.units, overlap, st);
    } else {
        r = launch_decode<1>(P, p.units, overlap, st);
    }
    prof_end(p.prof, st);
    return r;
}

}  // namespace lococo
