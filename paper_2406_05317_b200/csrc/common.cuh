// Internal declarations shared by the LoCoCo CUDA translation units.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "lococo.h"

namespace lococo {

// SMs of a B200. A constant, because workspaces are sized and plans are made by it on the host, also where no device is in sight; no
// kernel needs the device to have as many.
constexpr int kSMs = 148;

// Device-side view of a lococo_tensor (strides in elements).
struct View {
    char* ptr;
    int64_t sb, sh, st;
};

// One (sequence, head) unit's [cache; chunk] concatenation, cache first (Eq. 3).
struct CatView {
    View cache, chunk;
    int c;  // valid cache rows
    int b;  // chunk rows
};

template <typename T>
__device__ __forceinline__ const T* unit_base(const View& v, int n, int h) {
    return reinterpret_cast<const T*>(v.ptr) + n * v.sb + h * v.sh;
}
template <typename T>
__device__ __forceinline__ T* unit_base_mut(const View& v, int n, int h) {
    return reinterpret_cast<T*>(v.ptr) + n * v.sb + h * v.sh;
}
// Row j of the concatenation for unit (n, h).
template <typename T>
__device__ __forceinline__ const T* cat_row(const CatView& x, int n, int h, int j) {
    return j < x.c ? unit_base<T>(x.cache, n, h) + (int64_t)j * x.cache.st
                   : unit_base<T>(x.chunk, n, h) + (int64_t)(j - x.c) * x.chunk.st;
}

__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 x) { return __bfloat162float(x); }
template <typename T> __device__ __forceinline__ T from_f32(float x);
template <> __device__ __forceinline__ float from_f32<float>(float x) { return x; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float x) { return __float2bfloat16_rn(x); }

// Thread-block clusters: this CTA's rank, the cluster's barrier, another CTA's shared memory.
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ uint32_t remote(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_remote(uint32_t addr, float v) { asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory"); }
__device__ __forceinline__ void st_remote(uint32_t addr, const uint4& v) {
    asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// Parameters of one compress step (Algorithm 2, Steps 4-5) for all units.
struct CompressParams {
    CatView xk, xv;       // keys and values, [cache; chunk]
    View k_out, v_out;    // new cache
    int heads, units, d, M, k, c_in, S;
    int Sr;                // row stride of R (CUDA-core path): S, or S rounded up to a multiple of 4 where there is room
    int R_sets;            // sets of [units][M][Sr] logits that R has room for (partial sums of a split convolution)
    int splits;            // partial sums in use
    int weights_per_head;
    const void* g_packed;  // CUDA-core path: [heads|1][c_in][k][M], storage dtype
    const float* bias;     // [heads|1][M] or nullptr
    float eps;
    float* R;              // [units][M][Sr] ReLU'd logits
    float* s;              // [units][M] denominators of Eq. 7
    float* UK;             // [units][M][d] unnormalised blends
    float* UV;
    float* W_out;          // optional [units][M][S]
    void* R16;             // the backward's recompute (tensor-core path): R^T in bf16, [units][R16_unit / R16_stride][R16_stride]
    int R16_stride;        // slots per row, multiple of 16
    int64_t R16_unit;
    int64_t R16_term;      // elements from R's values to their remainders (where they are kept)
    int prot = 0;          // protected slots (Section 5.2): rows i < prot of Eq. 7's matrix are the unit rows e_i
    void* prof;            // host only: Profiler* or nullptr
};

// Parameters of one chunk attention (Algorithm 2, Step 3) for all units.
struct AttnParams {
    View q, o;
    CatView xk, xv;
    int heads, units, d, b, c;
    float scale;
    float* lse;        // optional [units][lse_stride]
    int64_t lse_stride;
    void* prof;        // host only: Profiler* or nullptr
};

struct FillParams {
    View src_k, src_v, dst_k, dst_v;  // src rows 0..b-1 -> dst rows c..c+b-1
    int heads, units, d, c, b;
    int late = 0;          // 1: the next launch is let in when the blocks end, not when they start
};

// CUDA-core kernels (simt_forward.cu). Each returns the number of kernels launched, or -1.
// Weight images: `forward` [sets][c_in][k][M], `reverse` [sets][M][k][c_in] with the taps reversed (either may be null).
int simt_pack_weights(int dtype, const void* G, void* forward, void* reverse, int sets, int M, int c_in, int k, cudaStream_t st);
int simt_fill(int dtype, const FillParams& p, cudaStream_t st);
int simt_compress(int dtype, const CompressParams& p, cudaStream_t st);
int simt_attention(int dtype, const AttnParams& p, cudaStream_t st);
// Attention with the old cache and the cache update of one compress step.
int simt_chunk_step(int dtype, const AttnParams& a, const CompressParams& p, cudaStream_t st);
int simt_write_weights(const float* R, const float* s, float* W, int64_t rows, int S, int Sr, cudaStream_t st);
// Floats of R at the largest S (all partial sums included).
size_t simt_R_floats(int units, int M, int Smax, int c_in);
// Brackets the launches between them with an event pair when p is a live Profiler*.
void prof_begin(void* p, int kind, cudaStream_t st);
void prof_end(void* p, cudaStream_t st);

int simt_convert_bias(int dtype, const void* bias, float* out, int n, cudaStream_t st);

}  // namespace lococo
