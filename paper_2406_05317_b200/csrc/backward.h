// Shared by the CUDA-core and the tensor-core backward kernels.
#pragma once
#include "common.cuh"

struct lococo_handle;

namespace lococo {

// One reversed step of Algorithm 2 for all units.
struct BwdStep {
    CatView xk, xv;            // [saved cache; chunk]
    View q, o, d_o;            // this chunk's queries, outputs, output gradients
    View dq, dk, dv;           // this chunk's gradients (outputs)
    int heads, units, d, M, k, c_in, c, b, S;
    int weights_per_head;
    const void* g_reverse;     // [sets][M][k][c_in], taps reversed
    float scale;
    const float* lse;          // this chunk's log-sum-exp, [units][lse_stride]
    int64_t lse_stride;
    float *R, *s;              // CUDA-core path: recomputed ReLU'd logits [units][M][Sr]; denominators [units][M]
    int Sr;                    // S rounded up to a multiple of 4
    float* dA;                 // CUDA-core path: [units][M][Sr]: dw, then dA in place
    const float* delta;        // [units][delta_stride]: <dO_r, O_r>, first query of this chunk
    int64_t delta_stride;
    float *gK, *gV;            // [units][M], rows g_st floats apart: gradient w.r.t. the cache (after the step in, before the step out)
    int g_st;
    float *dG, *dbias;         // [sets][M][c_in][k], [sets][M]
};

// Tensor-core versions (bf16, tensor_backward.cu). The scratch is carved from the caller's backward scratch; every function
// returns the number of launches or -1. prepare before the first step of a call, finish after its last.
bool tensor_backward_supported(const lococo_handle* h);
size_t tensor_backward_scratch_bytes(const lococo_handle* h, int B);
int tensor_backward_prepare(lococo_handle* h, int B, char* scratch, cudaStream_t st);
int tensor_backward_step(lococo_handle* h, const BwdStep& p, const CompressParams& fwd, int B, char* scratch, cudaStream_t st);
int tensor_backward_finish(lococo_handle* h, int B, char* scratch, float* dG, cudaStream_t st);

// Several reversed steps at once (fp32 storage, CUDA cores): chunks n0 .. n0 + count - 1 of a call. Arrays that hold something of every
// chunk of the group are indexed by n - n0.
struct BwdGroup {
    BwdStep first;             // views of the call's first token and first snapshot; delta and lse of the first token
    int L, B, c0, n0, count;   // tokens of the call, chunk length, cache length before the call
    int64_t snap_step;         // floats between snapshots
    int S, Sr;                 // of a whole chunk on a full cache: the stride of positions in all arrays here
    int splits;                // partial sums of the recomputed convolution
    int ctas;                  // CTAs per unit for the chain
    const void* g_packed;      // as in CompressParams
    const float* bias;
    float eps;
    int prot;
    View gk_final, gv_final;   // gradient w.r.t. the cache after the call (null pointers: zero), read by the group with the last chunk
    float *gK, *gV;            // [units][M][d]: gradient w.r.t. the cache before the group
    float* attn;               // [count][units][S][2 d]: the attention's share of dX
    float* R;                  // [count][splits][units][M][Sr]: partial logits, then (first of the splits) R
    float *s, *inner;          // [count][units][M]: denominators of Eq. 7; <dw, w>
    float* g;                  // [count + 1][units][M][2 d]: gradient w.r.t. the cache before chunk n0 + i
    float* dA;                 // [count][units][M][Sr]
    float* last;               // [units][M][2 d]: the cache after the call's last chunk
};
// Chunks of a group (0: one step at a time is the way) where there is room for `room` floats, and the floats of scratch that a group takes; both
// depend on the sizes alone.
int simt_group_chunks(const lococo_handle* h, int L, int B, size_t room, size_t* floats);
// Lays the arrays of G out in the `floats` at `scratch` (what simt_group_chunks said, or less chunks' worth of it), and says how many they take.
size_t simt_group_layout(BwdGroup& G, float* scratch, size_t floats);
int simt_group_clusters(const BwdGroup& G);        // CTAs per unit for the chain (0: clusters that this device would not run, or one after another)
bool simt_group_possible(const lococo_handle* h, int B);      // ... that a device whose SMs form any clusters could run: where not, no scratch is set aside
int simt_backward_group(const BwdGroup& G, cudaStream_t st);
int simt_backward_chain(const BwdGroup& G, cudaStream_t st);      // (simt_chain.cu: the part of a group that is a chain)

// CUDA-core versions (simt_backward.cu). `parts`: simt_backward_parts_floats of scratch.
size_t simt_backward_parts_floats(int units, int M, int B, int d);
// dX = `attn` + the gradient of a filled cache, handed on as in every step (fill steps of either path).
int simt_backward_fill_split(int dtype, const BwdStep& p, const float* attn, cudaStream_t st);
int simt_backward_step(int dtype, const BwdStep& p, const CompressParams& fwd, float* parts, cudaStream_t st);

}  // namespace lococo
