// Backward pass of Algorithm 2: gradients of
//   loss = <dO, O> + <dK_cache_final, K_cache_final> + <dV_cache_final, V_cache_final>
// w.r.t. Q, K, V and the conv weights (Section 3.2.1: the conv parameters are trained end to
// end), by reversing the chunk loop. Per step, with X = [cache before the step; chunk]:
//   cache update  fill:      dX[0:S]  = g                       (g = gradient w.r.t. the cache after the step)
//                 compress:  R, s recomputed from the saved cache (Eq. 6, ReLU, Eq. 7)
//                            dw  = g_K X_K^T + g_V X_V^T         (through Eq. 4, Eq. 5)
//                            dX += w^T g                          (the blend's own inputs)
//                            dA  = [A>0] (dw - <dw, w>_row) / s   (through Eq. 7 and the ReLU)
//                            dG += dA (*) Z,  dZ += dA (*) G      (through Eq. 6; dZ lands in dX)
//   attention     textbook softmax-attention gradient from dO, O and the saved log-sum-exp (Eq. 1)
//   split         first c rows of dX are the gradient w.r.t. the previous cache, the rest is dK_n, dV_n
// The contractions run on the tensor cores (tensor_backward.cu) or on the CUDA cores (simt_backward.cu).
#include <algorithm>

#include "backward.h"
#include "handle.h"
#include "simt.cuh"

namespace lococo {

namespace {

// delta[u][r] = <dO_r, O_r> for all queries of the call: a row is shared by d / 8 lanes, eight channels each.
template <typename T>
__global__ void __launch_bounds__(256) bwd_delta_kernel(View o, View d_o, float* delta, int heads, int L, int d) {
    const int u = blockIdx.y, n = u / heads, h = u % heads, lanes = d / 8;
    const int row = (blockIdx.x * 256 + threadIdx.x) / lanes, ch = 8 * (threadIdx.x % lanes);
    float acc = 0.f;
    if (row < L) {
        float a[8], b[8];
        simt::load8(unit_base<T>(o, n, h) + (int64_t)row * o.st + ch, a);
        simt::load8(unit_base<T>(d_o, n, h) + (int64_t)row * d_o.st + ch, b);
#pragma unroll
        for (int e = 0; e < 8; ++e) acc = fmaf(a[e], b[e], acc);
    }
    for (int of = lanes / 2; of > 0; of >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, of);
    if (row < L && ch == 0) delta[(int64_t)u * L + row] = acc;
}

// g = gradient of the loss w.r.t. the final cache (zero where the caller passes none).
template <typename T>
__global__ void bwd_init_g_kernel(View gk_in, View gv_in, float* gK, float* gV, int heads, int M, int d) {
    const int u = blockIdx.y, n = u / heads, h = u % heads;
    const int total = M * d;
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < total; x += gridDim.x * blockDim.x) {
        const int row = x / d, ch = x % d;
        gK[(int64_t)u * total + x] = gk_in.ptr ? to_f32((unit_base<T>(gk_in, n, h) + (int64_t)row * gk_in.st)[ch]) : 0.f;
        gV[(int64_t)u * total + x] = gv_in.ptr ? to_f32((unit_base<T>(gv_in, n, h) + (int64_t)row * gv_in.st)[ch]) : 0.f;
    }
}

// The gradient w.r.t. the cache the loop started from, out of the fp32 accumulators (all M rows; rows beyond the
// initial fill count hold zeros).
template <typename T>
__global__ void bwd_store_g_kernel(const float* gK, const float* gV, View gk_out, View gv_out, int heads, int M, int d) {
    const int u = blockIdx.y, n = u / heads, h = u % heads;
    const int total = M * d;
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < total; x += gridDim.x * blockDim.x) {
        const int row = x / d, ch = x % d;
        if (gk_out.ptr) unit_base_mut<T>(gk_out, n, h)[(int64_t)row * gk_out.st + ch] = from_f32<T>(gK[(int64_t)u * total + x]);
        if (gv_out.ptr) unit_base_mut<T>(gv_out, n, h)[(int64_t)row * gv_out.st + ch] = from_f32<T>(gV[(int64_t)u * total + x]);
    }
}

bool launched() { return cudaGetLastError() == cudaSuccess; }

template <typename T>
int deltas(View o, View d_o, float* delta, int heads, int units, int L, int d, cudaStream_t st) {
    const int rows = 256 / (d / 8);
    bwd_delta_kernel<T><<<dim3((L + rows - 1) / rows, units), 256, 0, st>>>(o, d_o, delta, heads, L, d);
    return launched() ? 1 : -1;
}

template <typename T>
int init_g(View gk, View gv, float* gK, float* gV, int heads, int units, int M, int d, cudaStream_t st) {
    bwd_init_g_kernel<T><<<dim3((M * d + 255) / 256, units), 256, 0, st>>>(gk, gv, gK, gV, heads, M, d);
    return launched() ? 1 : -1;
}

template <typename T>
int store_g(const float* gK, const float* gV, View gk, View gv, int heads, int units, int M, int d, cudaStream_t st) {
    bwd_store_g_kernel<T><<<dim3((M * d + 255) / 256, units), 256, 0, st>>>(gK, gV, gk, gv, heads, M, d);
    return launched() ? 1 : -1;
}

}  // namespace
}  // namespace lococo

using namespace lococo;

namespace {

size_t align256(size_t x) { return (x + 255) / 256 * 256; }

bool bview_ok(const lococo_tensor& t, size_t elt) {
    if (!t.ptr || (reinterpret_cast<uintptr_t>(t.ptr) & 15u)) return false;
    if ((t.stride_batch * (int64_t)elt) % 16 || (t.stride_head * (int64_t)elt) % 16 || (t.stride_token * (int64_t)elt) % 16)
        return false;
    return t.stride_token > 0;
}

View bdev(const lococo_tensor& t, int64_t tokens, size_t elt) {
    View v{static_cast<char*>(t.ptr), t.stride_batch, t.stride_head, t.stride_token};
    if (v.ptr) v.ptr += tokens * t.stride_token * (int64_t)elt;
    return v;
}

struct Scratch {
    size_t gK, gV, parts, dA, delta, tensor, group;
    size_t least, total;       // what some way of doing the call fits in; what the fastest takes
    size_t group_floats;       // room of the groups
    int group_chunks;          // chunks that one go of the CUDA cores can take (0: a step at a time)
};

// `bytes`: of the caller's scratch. With less than `total` groups are of fewer chunks, or there are none.
Scratch scratch_layout(const lococo_handle* h, int L, int B, size_t bytes) {
    const lococo_config& c = h->cfg;
    const size_t units = h->units, Smax = (size_t)c.M + B;
    Scratch s{};
    size_t off = 0;
    auto take = [&](size_t bytes) { const size_t o = off; off = align256(off + bytes); return o; };
    s.gK = take(units * c.M * c.head_dim * sizeof(float));
    s.gV = take(units * c.M * c.head_dim * sizeof(float));
    s.delta = take(units * (size_t)L * sizeof(float));
    if (tensor_backward_supported(h)) {
        s.tensor = take(tensor_backward_scratch_bytes(h, B));
    } else {
        s.parts = take(simt_backward_parts_floats(h->units, c.M, B, c.head_dim) * sizeof(float));
        s.dA = take(units * c.M * ((Smax + 3) / 4 * 4) * sizeof(float));
        // (in the place of what single steps need: a call takes the one way or the other)
        s.least = off;
        s.group = s.parts;
        s.group_chunks = simt_group_chunks(h, L, B, bytes < s.group ? 0 : (bytes - s.group) / sizeof(float), &s.group_floats);
        off = std::max(off, s.group + align256(s.group_floats * sizeof(float)));
    }
    s.total = off;
    if (s.least == 0) s.least = off;
    return s;
}

}  // namespace

extern "C" {

lococo_status lococo_backward_scratch_bytes(const lococo_handle* h, int32_t L, int32_t B, size_t* out) {
    if (!h || !out || L < 1 || B < 1 || B > h->cfg.max_chunk) return LOCOCO_ERR_INVALID_ARG;
    *out = scratch_layout(h, L, B, SIZE_MAX).total;
    return LOCOCO_OK;
}

lococo_status lococo_process_sequence_backward(lococo_handle* h, lococo_tensor Q, lococo_tensor K, lococo_tensor V,
                                               lococo_tensor O, int32_t L, int32_t B, int32_t cache_len_in, const void* saved,
                                               lococo_tensor dO, lococo_tensor dKc_final, lococo_tensor dVc_final,
                                               lococo_tensor dQ, lococo_tensor dK, lococo_tensor dV, float* dG, float* dbias,
                                               lococo_tensor dKc_in, lococo_tensor dVc_in, void* scratch,
                                               size_t scratch_bytes, void* stream) {
    if (!h) return LOCOCO_ERR_INVALID_ARG;
    if (!h->ws || !h->weights_set) return LOCOCO_ERR_WORKSPACE;
    const lococo_config& cfg = h->cfg;
    if (L < 1 || B < 1 || B > cfg.max_chunk || !saved || !dG || !scratch) return LOCOCO_ERR_INVALID_ARG;
    if (cache_len_in < 0 || cache_len_in > cfg.M) return LOCOCO_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(saved) & 255u) || (reinterpret_cast<uintptr_t>(scratch) & 255u) ||
        (reinterpret_cast<uintptr_t>(dG) & 15u))
        return LOCOCO_ERR_INVALID_ARG;
    const size_t e = h->elt;
    if (!bview_ok(Q, e) || !bview_ok(K, e) || !bview_ok(V, e) || !bview_ok(O, e) || !bview_ok(dO, e) || !bview_ok(dQ, e) ||
        !bview_ok(dK, e) || !bview_ok(dV, e))
        return LOCOCO_ERR_INVALID_ARG;
    if ((dKc_final.ptr && !bview_ok(dKc_final, e)) || (dVc_final.ptr && !bview_ok(dVc_final, e))) return LOCOCO_ERR_INVALID_ARG;
    if ((dKc_in.ptr && !bview_ok(dKc_in, e)) || (dVc_in.ptr && !bview_ok(dVc_in, e))) return LOCOCO_ERR_INVALID_ARG;
    if (dbias && !h->has_bias) return LOCOCO_ERR_INVALID_ARG;
    const Scratch sl = scratch_layout(h, L, B, scratch_bytes);
    if (scratch_bytes < sl.least) return LOCOCO_ERR_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    char* sc = static_cast<char*>(scratch);
    float* gK = reinterpret_cast<float*>(sc + sl.gK);
    float* gV = reinterpret_cast<float*>(sc + sl.gV);

    const int n_chunks = (L + B - 1) / B;
    const size_t snap_step = (size_t)h->units * cfg.M * cfg.head_dim * e;
    const size_t snap_all = align256((size_t)n_chunks * snap_step);
    const char* sv = static_cast<const char*>(saved);
    const float* lse_all = reinterpret_cast<const float*>(sv + 2 * snap_all);

    float* delta = reinterpret_cast<float*>(sc + sl.delta);

    // the CUDA cores take several chunks at a time where those of one would not fill the chip
    BwdGroup G{};
    if (sl.group_chunks) {
        const lococo_tensor snap{const_cast<char*>(sv), (int64_t)cfg.heads * cfg.M * cfg.head_dim, (int64_t)cfg.M * cfg.head_dim, (int64_t)cfg.head_dim};
        lococo_tensor snapV = snap;
        snapV.ptr = const_cast<char*>(sv) + snap_all;
        BwdStep& p = G.first;
        p.xk = CatView{bdev(snap, 0, e), bdev(K, 0, e), 0, 0};
        p.xv = CatView{bdev(snapV, 0, e), bdev(V, 0, e), 0, 0};
        p.q = bdev(Q, 0, e); p.o = bdev(O, 0, e); p.d_o = bdev(dO, 0, e);
        p.dq = bdev(dQ, 0, e); p.dk = bdev(dK, 0, e); p.dv = bdev(dV, 0, e);
        p.heads = cfg.heads; p.units = h->units; p.d = cfg.head_dim; p.M = cfg.M; p.k = cfg.k; p.c_in = cfg.c_in;
        p.weights_per_head = cfg.weights_per_head;
        p.g_reverse = h->ws + h->off_greverse;
        p.scale = h->scale;
        p.lse = lse_all; p.lse_stride = L;
        p.delta = delta; p.delta_stride = L;
        p.dG = dG; p.dbias = dbias;
        G.L = L; G.B = std::min(B, L); G.c0 = cache_len_in;
        G.snap_step = (int64_t)(snap_step / e);
        G.S = cfg.M + G.B; G.Sr = (G.S + 3) / 4 * 4;
        p.Sr = G.Sr;
        G.g_packed = h->ws + h->off_gpack;
        G.bias = h->has_bias ? reinterpret_cast<const float*>(h->ws + h->off_bias) : nullptr;
        G.eps = cfg.norm_eps; G.prot = h->prot;
        G.gk_final = bdev(dKc_final, 0, e); G.gv_final = bdev(dVc_final, 0, e);
        G.gK = gK; G.gV = gV;
    }
    // (A group's last launch writes dK and dV while it reads K and V for dG; single steps are done with a chunk's rows when they write
    // its gradients. A caller who wants them in place gets the latter.)
    auto in_place = [&](const lococo_tensor& t) { return t.ptr == K.ptr || t.ptr == V.ptr; };
    // (Groups take the chain through the cache apart, and with fewer than two compress steps there is none. us, in a group / a step at a time: one
    // fill step and one compress step, 127 units, d = 128, M = 14, B = 8 221 / 172, 4 units, M = 6, B = 4 60 / 50; three fill steps before it, 144
    // units, d = 64 108 / 82; two compress steps, 3 units, d = 64, M = 8, B = 51 81 / 118, 42 units, d = 128, M = 20, B = 121 218 / 209.)
    const int fills = cache_len_in + L <= cfg.M ? n_chunks : (cfg.M - cache_len_in) / B;
    if (sl.group_chunks && n_chunks - fills >= 2 && !in_place(dK) && !in_place(dV)) G.ctas = simt_group_clusters(G);
    const bool grouped = G.ctas > 0;
    // groups n0, n0 + group_chunks, ... from the last chunk back; the one that is left at the front may be shorter
    auto group_before = [&](int n) {
        G.count = std::min(n, sl.group_chunks);
        G.n0 = n - G.count;
        return simt_group_layout(G, reinterpret_cast<float*>(sc + sl.group), sl.group_floats) <= sl.group_floats;
    };
    for (int n = n_chunks; grouped && n > 0; n -= G.count)
        if (!group_before(n)) return LOCOCO_ERR_WORKSPACE;
    char* tb = tensor_backward_supported(h) ? sc + sl.tensor : nullptr;
    if (tb) {
        const int r = tensor_backward_prepare(h, B, tb, st);
        if (r < 0) return LOCOCO_ERR_CUDA;
        h->launches += r;
    }
    int launched_n = 0;
    if (!grouped) {      // (a group's chain reads the caller's tensors)
        launched_n = cfg.dtype == LOCOCO_F32
                         ? init_g<float>(bdev(dKc_final, 0, e), bdev(dVc_final, 0, e), gK, gV, cfg.heads, h->units, cfg.M, cfg.head_dim, st)
                         : init_g<__nv_bfloat16>(bdev(dKc_final, 0, e), bdev(dVc_final, 0, e), gK, gV, cfg.heads, h->units, cfg.M,
                                                 cfg.head_dim, st);
        if (launched_n < 0) return LOCOCO_ERR_CUDA;
        h->launches += launched_n;
    }
    launched_n = cfg.dtype == LOCOCO_F32 ? deltas<float>(bdev(O, 0, e), bdev(dO, 0, e), delta, cfg.heads, h->units, L, cfg.head_dim, st)
                                         : deltas<__nv_bfloat16>(bdev(O, 0, e), bdev(dO, 0, e), delta, cfg.heads, h->units, L, cfg.head_dim, st);
    if (launched_n < 0) return LOCOCO_ERR_CUDA;
    h->launches += launched_n;

    // cache fill count before every step of the forward
    int c_before[4096];
    if (n_chunks > 4096) return LOCOCO_ERR_UNSUPPORTED_SHAPE;
    for (int n = 0, c = cache_len_in; n < n_chunks; ++n) {
        const int b = std::min(B, L - n * B);
        c_before[n] = c;
        c = c + b <= cfg.M ? c + b : cfg.M;
    }
    for (int n = n_chunks; grouped && n > 0; n -= G.count) {
        group_before(n);
        const int r = simt_backward_group(G, st);
        if (r < 0) return LOCOCO_ERR_CUDA;
        h->launches += r;
    }
    for (int n = grouped ? -1 : n_chunks - 1; n >= 0; --n) {
        const int t0 = n * B, b = std::min(B, L - t0), c = c_before[n];
        lococo_tensor snapK{const_cast<char*>(sv) + (size_t)n * snap_step, (int64_t)cfg.heads * cfg.M * cfg.head_dim,
                            (int64_t)cfg.M * cfg.head_dim, (int64_t)cfg.head_dim};
        lococo_tensor snapV = snapK;
        snapV.ptr = const_cast<char*>(sv) + snap_all + (size_t)n * snap_step;
        BwdStep p{};
        p.xk = CatView{bdev(snapK, 0, e), bdev(K, t0, e), c, b};
        p.xv = CatView{bdev(snapV, 0, e), bdev(V, t0, e), c, b};
        p.q = bdev(Q, t0, e); p.o = bdev(O, t0, e); p.d_o = bdev(dO, t0, e);
        p.dq = bdev(dQ, t0, e); p.dk = bdev(dK, t0, e); p.dv = bdev(dV, t0, e);
        p.heads = cfg.heads; p.units = h->units; p.d = cfg.head_dim; p.M = cfg.M; p.k = cfg.k; p.c_in = cfg.c_in;
        p.c = c; p.b = b; p.S = c + b;
        p.weights_per_head = cfg.weights_per_head;
        p.g_reverse = h->ws + h->off_greverse;
        p.scale = h->scale;
        p.lse = lse_all + t0; p.lse_stride = L;
        p.R = reinterpret_cast<float*>(h->ws + h->off_R);
        p.s = reinterpret_cast<float*>(h->ws + h->off_s);
        p.dA = reinterpret_cast<float*>(sc + sl.dA);
        p.Sr = (p.S + 3) / 4 * 4;
        p.delta = delta + t0; p.delta_stride = L;
        p.gK = gK; p.gV = gV; p.g_st = cfg.head_dim;
        p.dG = dG; p.dbias = dbias;
        CompressParams f{};
        f.xk = p.xk; f.xv = p.xv;
        f.heads = cfg.heads; f.units = h->units; f.d = cfg.head_dim; f.M = cfg.M; f.k = cfg.k; f.c_in = cfg.c_in;
        f.S = p.S; f.weights_per_head = cfg.weights_per_head; f.g_packed = h->ws + h->off_gpack;
        f.Sr = p.Sr;
        f.R_sets = (int)std::min<size_t>(64, h->R_floats / ((size_t)f.units * f.M * f.Sr));
        f.bias = h->has_bias ? reinterpret_cast<const float*>(h->ws + h->off_bias) : nullptr;
        f.eps = cfg.norm_eps; f.prot = h->prot; f.R = p.R; f.s = p.s;
        const int r = tb ? tensor_backward_step(h, p, f, B, tb, st)
                         : simt_backward_step(cfg.dtype, p, f, reinterpret_cast<float*>(sc + sl.parts), st);
        if (r < 0) return LOCOCO_ERR_CUDA;
        h->launches += r;
    }
    if (tb) {
        const int r = tensor_backward_finish(h, B, tb, dG, st);
        if (r < 0) return LOCOCO_ERR_CUDA;
        h->launches += r;
    }
    // what the accumulators hold now is the gradient w.r.t. the cache the forward started from
    if (dKc_in.ptr || dVc_in.ptr) {
        const int r = cfg.dtype == LOCOCO_F32
                          ? store_g<float>(gK, gV, bdev(dKc_in, 0, e), bdev(dVc_in, 0, e), cfg.heads, h->units, cfg.M, cfg.head_dim, st)
                          : store_g<__nv_bfloat16>(gK, gV, bdev(dKc_in, 0, e), bdev(dVc_in, 0, e), cfg.heads, h->units, cfg.M,
                                                   cfg.head_dim, st);
        if (r < 0) return LOCOCO_ERR_CUDA;
        h->launches += r;
    }
    return LOCOCO_OK;
}

}  // extern "C"
