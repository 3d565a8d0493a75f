// Shared by the CUDA-core kernels, forward and backward: vector access to rows of float or bf16, launches that overlap the
// previous kernel's tail, and the register-tiled convolution both directions use.
#pragma once
#include <algorithm>
#include <atomic>

#include "common.cuh"

namespace lococo {
namespace simt {

__device__ __forceinline__ float4 load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
    const uint2 v = *reinterpret_cast<const uint2*>(p);
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v.y));
    return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void store4(float* p, const float4& v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void store4(__nv_bfloat16* p, const float4& v) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
    *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
}
template <typename T>
__device__ __forceinline__ void load8(const T* p, float (&v)[8]) {
    const float4 a = load4(p), b = load4(p + 4);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ float dot4(const float4& a, const float4& b, float acc) {
    acc = fmaf(a.x, b.x, acc); acc = fmaf(a.y, b.y, acc);
    acc = fmaf(a.z, b.z, acc); acc = fmaf(a.w, b.w, acc);
    return acc;
}
__device__ __forceinline__ void axpy4(float s, const float4& x, float4& y) {
    y.x = fmaf(s, x.x, y.x); y.y = fmaf(s, x.y, y.y); y.z = fmaf(s, x.z, y.z); y.w = fmaf(s, x.w, y.w);
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(valid ? 16u : 0u) : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src, bool valid) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(valid ? 4u : 0u) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// The kernels of a call are launched as programmatic dependents: a kernel's launch overlaps the tail of the one before it,
// and every kernel waits here, before it touches anything, until the one before is complete and its results are visible.
__device__ __forceinline__ void start_and_wait() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
// Kernels with long blocks let the next launch in only when their blocks end. Blocks that wait are placed where room is first, two on an SM that
// is done early while others get none, and stay there: that costs more than a launch that is not hidden. Triggered at the start of
// blends, convolutions and the backward launches -> at their end: 12 heads of 128, 5 chunks of 200, M = 128, k = 21 759 -> 715 us, 3 heads 464 -> 341;
// k = 5 and 8 heads, 4 of 512 496 -> 449; a training step of 8 heads, 4 of 300, k = 21 3446 -> 3126. Worst of 76 sizes: 16 heads, k = 13 892 -> 900.
__device__ __forceinline__ void start_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// (`overlap` false: in plain stream order.)
template <typename... Params, typename... Args>
inline bool launch_maybe_after(bool overlap, void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, const Args&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlap ? 1 : 0;
    if (cudaLaunchKernelEx(&cfg, kernel, args...) == cudaSuccess) return true;
    cudaGetLastError();
    return false;
}
template <typename... Params, typename... Args>
inline bool launch_after(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, const Args&... args) {
    return launch_maybe_after(true, kernel, grid, block, smem, st, args...);
}
// The dynamic shared-memory limit of a kernel is a per-device attribute: it is set on the first launch on each device.
template <typename Kernel>
inline bool smem_limit(Kernel kernel, int bytes, bool (&done)[64]) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    if (!done[dev]) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return false;
        done[dev] = true;
    }
    return true;
}

// A kernel launched as clusters of up to 16 CTAs: its per-device attributes, and how many clusters of each size a device runs at
// the same time (a cluster lies within one group of SMs).
constexpr int kMaxCluster = 16;
inline int next_cluster(int ctas) { return ctas < 8 ? 2 * ctas : ctas + 1; }      // the sizes in use: 1, 2, 4, 8, 9 .. 16
struct ClusterKernel {
    bool ready[64] = {};
    std::atomic<bool> counted[64] = {};
    std::atomic<int> resident[64][kMaxCluster + 1] = {};
};
// The current device, with the kernel's attributes set there; or -1
template <typename Kernel>
inline int cluster_device(ClusterKernel& k, Kernel kernel, int max_smem) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return -1;
    if (!k.ready[dev]) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem) != cudaSuccess ||
            cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return -1;
        k.ready[dev] = true;
    }
    return dev;
}
inline cudaLaunchAttribute cluster_of(int ctas) {
    cudaLaunchAttribute a;
    a.id = cudaLaunchAttributeClusterDimension;
    a.val.clusterDim.x = ctas;
    a.val.clusterDim.y = a.val.clusterDim.z = 1;
    return a;
}
// Clusters of every size (index: CTAs) that the current device runs at once (0: none, or it cannot be told), or nullptr. Asked of the runtime once per
// device, for all sizes: plans are made in every call, and 24 such questions per call cost a one-chunk call 10 us of host time.
template <typename Kernel>
inline const std::atomic<int>* resident_clusters(ClusterKernel& k, Kernel kernel, int max_smem, int threads) {
    const int dev = cluster_device(k, kernel, max_smem);
    if (dev < 0) {
        cudaGetLastError();
        return nullptr;
    }
    if (k.counted[dev].load(std::memory_order_acquire)) return k.resident[dev];
    for (int ctas = 1; ctas <= kMaxCluster; ctas = next_cluster(ctas)) {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(ctas);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = max_smem;
        cudaLaunchAttribute attr = cluster_of(ctas);
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
            cudaGetLastError();
            n = 0;
        }
        k.resident[dev][ctas].store(n, std::memory_order_relaxed);      // (threads that come here together store the same)
    }
    k.counted[dev].store(true, std::memory_order_release);
    return k.resident[dev];
}
template <typename... Params, typename... Args>
inline bool launch_clusters(ClusterKernel& k, void (*kernel)(Params...), int max_smem, int ctas, int clusters, int threads, size_t smem, cudaStream_t st, const Args&... args) {
    if (cluster_device(k, kernel, max_smem) < 0) return false;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(clusters * ctas);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1] = cluster_of(ctas);
    cfg.attrs = attr;
    cfg.numAttrs = ctas > 1 ? 2 : 1;
    if (cudaLaunchKernelEx(&cfg, kernel, args...) == cudaSuccess) return true;
    cudaGetLastError();
    return false;
}

// Two fp32 FMAs per instruction (each rounded as an FMA of its own): the kernels here are bound by instruction issue, and a
// float4 from shared memory is two such operands as it lies.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pair(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 unpair(f32x2 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ void fma2(f32x2 a, f32x2 b, f32x2& acc) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b)); }
__device__ __forceinline__ void add2(f32x2 a, f32x2& acc) { asm("add.rn.f32x2 %0, %1, %0;" : "+l"(acc) : "l"(a)); }
__device__ __forceinline__ void mul2(f32x2 a, f32x2& acc) { asm("mul.rn.f32x2 %0, %1, %0;" : "+l"(acc) : "l"(a)); }
struct f32x4 { f32x2 lo, hi; };                  // a float4 as two operands
__device__ __forceinline__ f32x4 load_pairs(const float* p) {
    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
    return f32x4{v.x, v.y};
}
__device__ __forceinline__ void fma4(f32x2 a, const f32x4& x, f32x4& y) { fma2(a, x.lo, y.lo); fma2(a, x.hi, y.hi); }
__device__ __forceinline__ float4 to_float4(const f32x4& v) {
    const float2 a = unpair(v.lo), b = unpair(v.hi);
    return make_float4(a.x, a.y, b.x, b.y);
}

// Sums of v[0..N-1] over the L lanes of a group (powers of two); lane l of the group is left with max(1, N / L) results in
// v[0..], from index l * N / L on (L > N: every L / N lanes hold the same one).
template <int N, int L>
__device__ __forceinline__ void reduce_lanes(float (&v)[N], int lane) {
    int n = N;
#pragma unroll
    for (int m = L / 2; m > 0; m >>= 1) {
        if (n == 1) {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], m);
            continue;
        }
        n >>= 1;
        const bool up = lane & m;
#pragma unroll
        for (int e = 0; e < N / 2; ++e) {
            if (e >= n) break;
            const float send = up ? v[e] : v[e + n], keep = up ? v[e + n] : v[e];
            v[e] = keep + __shfl_xor_sync(0xffffffffu, send, m);
        }
    }
}

// Barrier of a group of 128 threads of a block (group g of a block of several, or the whole block: g = 0).
__device__ __forceinline__ void group_sync(int g) { asm volatile("bar.sync %0, 128;" ::"r"(g) : "memory"); }

// Accumulators of a WindowConv thread: eight outputs (as pairs) x four positions.
struct ConvAcc {
    f32x2 v[4][4];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int y = 0; y < 4; ++y) v[x][y] = 0ull;
    }
    __device__ __forceinline__ float get(int x, int y) const { const float2 f = unpair(v[x >> 1][y]); return (x & 1) ? f.y : f.x; }
    __device__ __forceinline__ void add(const ConvAcc& o) {
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int y = 0; y < 4; ++y) { const float2 a = unpair(v[x][y]), b = unpair(o.v[x][y]); v[x][y] = pair(a.x + b.x, a.y + b.y); }
    }
};

// A 1-D convolution of many channels in fp32, one tile of OT outputs x PT positions per group of 128 threads (`tid` within the
// group, `bar` its barrier):
//   acc[o][p] += sum over c in [8 c_begin, 8 c_end), t in [0, k) of W[c][t][o] * X[c][x0 + p + t]      (W: n_in x k x n_out)
// Bound: FMA issue. A thread owns 8 outputs x 4 consecutive positions; the window of 4 + 3 inputs that four taps need sits
// in registers and serves 128 FMAs (two per instruction), so that ten vector loads from shared memory feed them (a scheme that reloaded every
// input for every tap, 8 loads for 16 FMAs, ran at a tenth of the FMA rate). Inputs are staged eight channels at a time,
// transposed to [channel][position]; weights come in pieces of eight channels x eight taps. Both are double-buffered: the
// weight copies are asynchronous and the next inputs wait in registers while a piece is computed.
// `in.load8(c, x, v)` delivers X[c .. c + 7][x], zeros outside the data.
template <typename T, int OT>
struct WindowConv {
    static constexpr int TI = OT / 8, TJ = 128 / TI, PT = 4 * TJ;
    static constexpr int kWFloats = 8 * 8 * OT;                   // one piece of weights: [8 channels][8 taps][OT]
    static constexpr int kRounds = (PT + 62 + 127) / 128;         // rows of an input stage per thread
    __host__ __device__ static size_t smem_bytes(int k) { return sizeof(float) * (2 * kWFloats + 2 * 8 * (size_t)(PT + (k + 2) / 4 * 4 + 4)); }
    // thread's outputs: two groups of four consecutive ones, half a tile apart
    __device__ static __forceinline__ int out_index(int ti, int x) { return x < 4 ? 4 * ti + x : OT / 2 + 4 * ti + x - 4; }

    // kSums: `total` takes sums of sixteen channels at a time (a long contraction's rounding errors grow with the longest chain of additions).
    template <bool kSums = false, typename Input>
    __device__ static __forceinline__ void run(const T* w, int n_in, int n_out, int k, int o0, int x0, int c_begin, int c_end, const Input& in,
                                               float* smem, ConvAcc& acc, int tid, int bar, ConvAcc* total = nullptr) {
        const int ti = tid % TI, tj = tid / TI;
        const int rows = PT + k - 1, ZW = PT + (k + 2) / 4 * 4 + 4;
        float* Ws = smem;                       // [2][8][8][OT]
        float* Zs = smem + 2 * kWFloats;        // [2][8][ZW]
        const int tap_pieces = (k + 7) / 8;
        const int steps = (c_end - c_begin) * tap_pieces;
        const bool vec = (n_out & 3) == 0;
        // (a thread copies the same four outputs of the same channel for every kTapStep-th tap: no division by a variable. With one per
        // copied vector, and the pieces' numbers divided out in every step: 2048 tokens of 8 heads, M = 128, B = 512, k = 21 653 us, now 605;
        // 12 heads, k = 17 861 / 780; k = 9, whose second piece is a single tap, 499 / 510.)
        constexpr int kTapStep = 128 / (8 * (OT / 4));
        const int w_o = 4 * (tid % (OT / 4)), w_c = tid / (OT / 4) % 8, w_t = tid / (8 * (OT / 4));
        auto load_weights = [&](int step) {
            const int chunk = step / tap_pieces, c = 8 * (c_begin + chunk) + w_c, t0 = 8 * (step - chunk * tap_pieces), nt = min(8, k - t0);
            const T* src = w + ((int64_t)c * k + t0 + w_t) * n_out + o0 + w_o;
            float* d = Ws + (step & 1) * kWFloats + (w_c * 8 + w_t) * OT + w_o;
            const bool in_range = c < n_in;
            const bool live = in_range && o0 + w_o < n_out;
#pragma unroll 1
            for (int t = w_t; t < nt; t += kTapStep, src += kTapStep * n_out, d += kTapStep * OT) {
                if (sizeof(T) == 4 && vec) {
                    cp_async16(d, live ? src : w, live);
                } else {
#pragma unroll
                    for (int e = 0; e < 4; ++e) d[e] = in_range && o0 + w_o + e < n_out ? to_f32(src[e]) : 0.f;
                }
            }
            cp_async_commit();
        };
        float next[kRounds][8];
        auto fetch_inputs = [&](int chunk) {
#pragma unroll
            for (int r = 0; r < kRounds; ++r)
                if (tid + 128 * r < rows) in.load8(8 * chunk, x0 + tid + 128 * r, next[r]);
        };
        auto put_inputs = [&](int chunk) {
            float* dst = Zs + (chunk & 1) * 8 * ZW;
#pragma unroll
            for (int r = 0; r < kRounds; ++r)
                if (tid + 128 * r < rows) {
#pragma unroll
                    for (int c = 0; c < 8; ++c) dst[c * ZW + tid + 128 * r] = next[r][c];
                }
        };
        if (steps <= 0) return;
        load_weights(0);
        fetch_inputs(c_begin);
        put_inputs(c_begin);
        int chunk = c_begin, piece = -1;
#pragma unroll 1
        for (int step = 0; step < steps; ++step) {
            if (++piece == tap_pieces) { piece = 0; ++chunk; }
            cp_async_wait<0>();
            group_sync(bar);                    // this step's weights and inputs are there; the buffers of the step before are free
            if (step + 1 < steps) load_weights(step + 1);
            const bool fetch = piece == tap_pieces - 1 && step + 1 < steps;
            if (fetch) fetch_inputs(chunk + 1);
            const float* wp = Ws + (step & 1) * kWFloats + 4 * ti;
            const float* zp = Zs + (chunk & 1) * 8 * ZW + 4 * tj + 8 * piece;
            const int nt = min(8, k - 8 * piece);
            // four taps from a window of seven inputs
            auto taps = [&](const f32x2 (&z)[8], const float* wt, int count) {
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    if (t >= count) break;
                    const f32x4 a = load_pairs(wt + t * OT), b = load_pairs(wt + t * OT + OT / 2);
#pragma unroll
                    for (int y = 0; y < 4; ++y) {
                        fma2(a.lo, z[t + y], acc.v[0][y]);
                        fma2(a.hi, z[t + y], acc.v[1][y]);
                        fma2(b.lo, z[t + y], acc.v[2][y]);
                        fma2(b.hi, z[t + y], acc.v[3][y]);
                    }
                }
            };
            auto window = [&](f32x2 (&z)[8], const float* src, int at) {
                const float4 v = *reinterpret_cast<const float4*>(src);
                z[at] = pair(v.x, v.x); z[at + 1] = pair(v.y, v.y); z[at + 2] = pair(v.z, v.z); z[at + 3] = pair(v.w, v.w);
            };
            if (nt == 8) {
#pragma unroll 2
                for (int c = 0; c < 8; ++c) {
                    f32x2 z[8];
                    window(z, zp + c * ZW, 0);
                    window(z, zp + c * ZW + 4, 4);
                    taps(z, wp + c * 8 * OT, 4);
#pragma unroll
                    for (int e = 0; e < 4; ++e) z[e] = z[e + 4];
                    window(z, zp + c * ZW + 8, 4);
                    taps(z, wp + (c * 8 + 4) * OT, 4);
                }
            } else {
#pragma unroll 1
                for (int t4 = 0; t4 < nt; t4 += 4) {
#pragma unroll 2
                    for (int c = 0; c < 8; ++c) {
                        f32x2 z[8];
                        window(z, zp + c * ZW + t4, 0);
                        window(z, zp + c * ZW + t4 + 4, 4);
                        taps(z, wp + (c * 8 + t4) * OT, nt - t4);
                    }
                }
            }
            if (kSums && piece == tap_pieces - 1 && (((chunk - c_begin) & 1) || step + 1 == steps)) {
                total->add(acc);
                acc.clear();
            }
            if (fetch) put_inputs(chunk + 1);   // (the buffer this chunk's predecessor used: its readers passed the barrier above)
        }
    }
};

// ------------------------------------------------------------------ Eq. 6 (forward, and the backward pass's recompute)
// The forward convolution: contraction over the channels of [cache; chunk] rows.
template <typename T>
struct ForwardInput {
    const CompressParams& p;
    int n, h;
    // eight consecutive channels of row j, zeros outside [0, S)
    __device__ __forceinline__ void load8(int ch0, int j, float (&v)[8]) const {
        if (j < 0 || j >= p.S) {
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = 0.f;
            return;
        }
        const T* row = ch0 < p.d ? cat_row<T>(p.xk, n, h, j) + ch0 : cat_row<T>(p.xv, n, h, j) + ch0 - p.d;
        simt::load8<T>(row, v);
    }
};

template <typename T, int OT>
__device__ __forceinline__ void conv_body(const CompressParams& p, float* smem, int block, int tid, int group) {
    constexpr int PT = WindowConv<T, OT>::PT;
    const int pos_tiles = (p.S + PT - 1) / PT, slot_tiles = (p.M + OT - 1) / OT;
    const int jt = block % pos_tiles; block /= pos_tiles;
    const int it = block % slot_tiles; block /= slot_tiles;
    const int splits = p.splits, split = block % splits, u = block / splits;
    const int n = u / p.heads, h = u % p.heads, pad = (p.k - 1) / 2;
    const int j0 = jt * PT, i0 = it * OT;
    const T* w = reinterpret_cast<const T*>(p.g_packed) + (p.weights_per_head ? (int64_t)h * p.k * p.M * p.c_in : 0);
    const int chunks = p.c_in / 8, c_begin = chunks * split / splits, c_end = chunks * (split + 1) / splits;
    ConvAcc acc;
    const ForwardInput<T> in{p, n, h};
    acc.clear();
    WindowConv<T, OT>::run(w, p.c_in, p.M, p.k, i0, j0 - pad, c_begin, c_end, in, smem, acc, tid, 1 + group);
    float* P = p.R + ((int64_t)split * p.units + u) * p.M * p.Sr;
    const int ti = tid % (OT / 8), tj = tid / (OT / 8);
    const int j = j0 + 4 * tj;
    if (j >= p.S) return;
#pragma unroll
    for (int x = 0; x < 8; ++x) {
        const int i = i0 + WindowConv<T, OT>::out_index(ti, x);
        if (i >= p.M) continue;
        float* row = P + (int64_t)i * p.Sr + j;
        if ((p.Sr & 3) == 0) {
            *reinterpret_cast<float4*>(row) = make_float4(acc.get(x, 0), acc.get(x, 1), acc.get(x, 2), acc.get(x, 3));
        } else {
#pragma unroll
            for (int y = 0; y < 4; ++y)
                if (j + y < p.S) row[y] = acc.get(x, y);
        }
    }
}

// Slots per block of the convolution: 64, or (small caches) as few as hold them.
inline int slot_tile(int M) { return M > 32 ? 64 : (M > 16 ? 32 : 16); }

// Blocks that share one tile's channels. A tile is 4096 outputs by 128 threads, and an SM holds four such blocks: while the
// tiles are fewer than a round and a half of that, the channels are split, so that a call of few
// units leaves no SM idle and its last round is short; a split keeps at least four chunks of eight channels, and R has to
// have the room for its partial sums.
inline int conv_splits(const CompressParams& p) {
    const int OT = slot_tile(p.M), PT = 4096 / OT;
    const int64_t tiles = (int64_t)((p.S + PT - 1) / PT) * ((p.M + OT - 1) / OT) * p.units;
    const int64_t want = 6 * kSMs / tiles;
    return (int)std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(want, p.R_sets), p.c_in / 32));
}

inline int conv_tiles(const CompressParams& p) {
    const int OT = slot_tile(p.M), PT = 4096 / OT;
    return (p.S + PT - 1) / PT * ((p.M + OT - 1) / OT) * p.units * p.splits;
}


// Row `row` of the logits (a warp): the partial convolutions added in their order, bias and ReLU applied, protected slots'
// unit rows put in; zero from S on. at(j): four consecutive logits (Sr a multiple of 4), or (one = true) a single one.
struct LogitRow {
    const float* r;
    int64_t step;          // floats between partial sums
    int splits, S, i;
    float bias;
    bool keep;
    __device__ __forceinline__ LogitRow(const CompressParams& p, int row) {
        i = row % p.M;
        const int u = row / p.M;
        r = p.R + (int64_t)row * p.Sr;
        step = (int64_t)p.units * p.M * p.Sr;
        splits = p.splits; S = p.S;
        bias = p.bias ? p.bias[(p.weights_per_head ? (u % p.heads) * p.M : 0) + i] : 0.f;
        keep = i < p.prot;
    }
    __device__ __forceinline__ float finish(float v, int j) const { return j >= S ? 0.f : (keep ? (j == i ? 1.f : 0.f) : fmaxf(v + bias, 0.f)); }
    __device__ __forceinline__ float4 at4(int j) const {
        float4 v = *reinterpret_cast<const float4*>(r + j);
        for (int s = 1; s < splits; ++s) {
            const float4 t = *reinterpret_cast<const float4*>(r + s * step + j);
            v.x += t.x; v.y += t.y; v.z += t.z; v.w += t.w;
        }
        return make_float4(finish(v.x, j), finish(v.y, j + 1), finish(v.z, j + 2), finish(v.w, j + 3));
    }
    __device__ __forceinline__ float at(int j) const {
        float v = r[j];
        for (int s = 1; s < splits; ++s) v += r[s * step + j];
        return finish(v, j);
    }
};

}  // namespace simt
}  // namespace lococo
