// Host-side state behind a lococo_handle, and the hooks of the tensor-core path.
#pragma once

#include <vector>

#include "common.cuh"

namespace lococo {
// Optional CUDA-event timing of individual kernel classes, on the launching stream.
enum ProfKind { PROF_CONV = 0, PROF_ATTENTION = 1, PROF_STEP = 2, PROF_SEQUENCE = 3, PROF_KINDS = 4 };
struct Profiler {
    struct Rec { cudaEvent_t a, b; int kind; };
    bool on = false;
    std::vector<Rec> recs;  // event pairs, reused across profile runs
    size_t used = 0;
    void begin(int kind, cudaStream_t st);
    void end(cudaStream_t st);
    void release();
};
}  // namespace lococo

struct lococo_handle {
    lococo_config cfg{};
    int prot = 0;   // protected slots (Section 5.2)
    int units = 0;          // batch * heads
    size_t elt = 0;         // bytes per stored element
    float scale = 0.f;      // softmax scale in effect
    bool use_tensor = false;
    // true once a kernel of this library has been launched in the current call: only then may the next one be
    // launched as a programmatic dependent (its early, pre-wait reads must not race with a foreign kernel)
    bool chain_open = false;
    // A generation-stage or short-chunk kernel may ask for its weight tiles before it waits for the kernel before it, once another such
    // kernel has come after the packing of the weights: for calls that run, whether one has run; and the capture, if any, in which one
    // has been recorded (that says nothing about what runs, and nothing about other captures).
    bool decode_open = false;
    unsigned long long decode_capture = 0;
    bool weights_settled(cudaStream_t st) {
        cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
        unsigned long long id = 0;
        if (cudaStreamGetCaptureInfo(st, &status, &id) != cudaSuccess || status != cudaStreamCaptureStatusActive) {
            cudaGetLastError();      // (the legacy default stream while another one is captured)
            const bool settled = decode_open;
            decode_open = true;
            return settled;
        }
        const bool settled = decode_open || decode_capture == id;
        decode_capture = id;
        return settled;
    }
    void weights_packed() { decode_open = false; decode_capture = 0; }
    bool persistent_loop = false;   // consecutive compress steps as one persistent launch (LOCOCO_PATH_TENSOR_PERSISTENT)
    bool weights_set = false;
    bool has_bias = false;
    char* ws = nullptr;     // caller-owned device workspace
    size_t ws_need = 0;
    size_t R_floats = 0;    // logits the workspace's R has room for
    size_t off_status = 0, off_gpack = 0, off_greverse = 0, off_bias = 0, off_s = 0, off_UK = 0, off_UV = 0, off_R = 0;
    size_t off_gimage = 0, off_part = 0, off_steps = 0, off_sync = 0;  // tensor-core path
    size_t off_alt_k = 0, off_alt_v = 0;   // second cache (the chunk loop alternates between the caller's and this one)
    size_t off_stream = 0;                 // queue and versions of tensor_stream.cu
    size_t off_merge = 0;                  // per (unit, slot block): partial sets stored in the current step
    // persistent chunk loop: step descriptors staged in pinned host memory (a small ring, one slot per call)
    static constexpr int kSeqSlots = 4;
    unsigned char* seq_host = nullptr;
    cudaEvent_t seq_event[kSeqSlots] = {};
    int seq_slot = 0, seq_count = 0;
    // what a backward step does beside its chain (tensor_backward.cu), and where the two meet (created on first use)
    cudaStream_t side = nullptr;
    cudaEvent_t side_ev[5] = {};
    // lococo_process_sequence_host: copy streams and per-chunk events (created on first use)
    cudaStream_t host_in = nullptr, host_out = nullptr;
    cudaEvent_t* host_ev = nullptr;
    int host_ev_n = 0;
    int seq_items = 0, seq_per_unit = 0;   // items queued so far: all units, one unit
    int coop_grid = 0;      // 0: not probed yet, -1: persistent kernel unavailable, > 0: CTAs that fit the device
    int64_t launches = 0;
    // CUDA graph of the chunk loop for the most recent argument set of lococo_process_sequence
    struct LoopGraph {
        unsigned char key[256] = {};   // the call's arguments, byte for byte
        size_t key_len = 0;
        int seen = 0;                  // identical calls so far (the graph is captured on the second)
        cudaGraphExec_t exec = nullptr;
        int64_t launches = 0;          // kernels inside the graph
        int c_out = 0;                 // cache length after the loop
        bool disabled = false;         // a graph call failed once: stay eager
    } loop_graph;
    lococo::Profiler prof;
};

namespace lococo {

// Where the weights of the blends, the probabilities of the attention and what the backward pass makes of them enter the tensor
// cores as two bf16 terms each, value and remainder: head dimension 64, and cache sizes that are no multiple of 128.
__host__ __device__ constexpr bool split_terms(int d, bool whole_blocks) { return d != 128 || !whole_blocks; }

// Tensor-core (tcgen05) path, tensor_forward.cu.
bool tensor_config_supported(const lococo_config* c);
void tensor_layout_workspace(lococo_handle* h, size_t* off);
int tensor_pack_weights(lococo_handle* h, const void* G, cudaStream_t st);
bool tensor_compress_supported(const lococo_handle* h, const CompressParams& p);
int tensor_compress(lococo_handle* h, const CompressParams& p, cudaStream_t st);
// The backward pass's recompute of a compress step: R^T (bf16, one or two terms) and the denominators of Eq. 7, and what the gradient needs of
// the cache gradient g = [gK | gV] (fp32, [units][M][d] each): dot = <g, new cache> per slot (= <dw, w> of Eq. 7 reversed),
// and g and g / s as two bf16 terms each (value and remainder), rows [gK | gV].
struct RecomputeOut {
    void* r_t;            // [terms][units][Sp][Mp]
    int Mp, Sp;
    const float *gK, *gV;
    void *g, *g_lo, *gs, *gs_lo;
    float* dot;           // [units][M]
};
int tensor_recompute(lococo_handle* h, const CompressParams& p, const RecomputeOut& out, cudaStream_t st);
bool tensor_step_direct(lococo_handle* h, const CompressParams& p);
bool tensor_attention_supported(const lococo_handle* h, const AttnParams& p);
int tensor_attention(lococo_handle* h, const AttnParams& p, cudaStream_t st);
// A step of one token on a full cache of 128 slots, in place (tensor_decode.cu); 0: the copy engine cannot read these views.
bool tensor_decode_supported(const lococo_handle* h, const AttnParams& a, const CompressParams& p);
int tensor_decode_step(lococo_handle* h, const AttnParams& a, const CompressParams& p, cudaStream_t st);
// `steps` consecutive steps of 1 to 64 tokens each on a full cache of 128 slots, attention and cache update of a unit in one CTA,
// in place (a single step may also write another cache), one launch (tensor_stream.cu); 0: the copy engine cannot read these
// views. The workspace words it synchronises on are zero between launches.
bool tensor_stream_supported(const lococo_handle* h, const AttnParams& a, const CompressParams& p);
int tensor_stream_steps(lococo_handle* h, const AttnParams& a, const CompressParams& p, int steps, cudaStream_t st);
size_t tensor_stream_sync_bytes(const lococo_handle* h);
int tensor_chunk_step(lococo_handle* h, const AttnParams& a, const CompressParams& p, cudaStream_t st);
// Persistent chunk loop: queue consecutive compress steps, then run them all in one launch of one CTA per SM.
bool tensor_sequence_add(lococo_handle* h, const AttnParams& a, const CompressParams& p, cudaStream_t st);
int tensor_sequence_launch(lococo_handle* h, cudaStream_t st, void* prof);
void tensor_sequence_release(lococo_handle* h);

// The whole chunk loop of a small fp32 problem in one launch (simt_loop.cu): how, where that is the faster way.
struct LoopPlan {
    int ctas, chain_warps, tile;      // CTAs per unit (0: not this way), warps that update the cache, convolution tile
};
LoopPlan simt_loop_plan(const lococo_handle* h, int L, int B, int c0);
int simt_loop(lococo_handle* h, const LoopPlan& plan, View q, View k, View v, int L, int B, View o, View kc, View vc, int c0, char* saved, size_t snap_step,
              size_t snap_all, cudaStream_t st);

}  // namespace lococo
