// Shared declarations of the CUDA side: views of the caller's buffers, small device helpers.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "cachefocus.h"
#include "cachefocus_debug.h"

namespace cf {

constexpr int kTile = CF_TILE_TOKENS;
constexpr int kMaxDocs = CF_MAX_DOCS_PER_REQUEST;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

struct GeomView {
    int n_q_heads, n_kv_heads, head_dim, dtype, rope_layout, pos_range;
    double rope_theta;
};

struct BatchView {
    int n_requests, n_docs_total, q_len, prefix_len, tail_reserve, n_reuse;
    long long total_tokens, token_stride;
    const int* req_doc_begin;
    const int* doc_offsets;
    const int* doc_src_start;
};

// Typed pointers into a plan buffer (see cf_plan_layout).
struct PlanView {
    int* status;
    int* kept;
    int* kept_count;
    int* dst_start;
    int* group;
    int* n_reuse;
    int* query_start;
    int* n_tiles;
    int* tile_begin;
    int* doc_tile_begin;
    int* doc_tile_count;
    int* tile_doc;
    int* tile_row0;
    int* tile_len;
    float2* trig;
    int max_tiles;
};

// First tile slot of request b: an upper bound of the tiles all earlier requests can own
// (a document of len tokens owns ceil(len/kTile) <= 1 + len/kTile tiles).
__host__ __device__ inline int tile_base(int doc_begin, int row_begin) {
    return doc_begin + row_begin / kTile;
}

// Division of 0 <= n < 2^31 by a divisor the host knows: three dependent instructions instead of the thirty of a division whose
// divisor comes out of a register (and over a hundred in 64 bits), on the way to the first load of kernels that run for 3 us.
// Multiplication by the reciprocal and a shift (Granlund and Montgomery, Division by Invariant Integers using Multiplication, 1994).
struct Divisor {
    unsigned d, mul, shift;
    Divisor() = default;
    explicit Divisor(int by) : d((unsigned)by), mul(0), shift(0) {
        while (shift < 31 && (1u << shift) < d) ++shift;
        mul = (unsigned)((((1ull << shift) - d) << 32) / d) + 1u;
    }
#ifdef __CUDACC__
    __device__ __forceinline__ int quotient(int n) const { return (int)((__umulhi((unsigned)n, mul) + (unsigned)n) >> shift); }
    __device__ __forceinline__ int remainder(int n) const { return n - quotient(n) * (int)d; }
#endif
};

GeomView make_geom_view(const cf_geom* g);
BatchView make_batch_view(const cf_batch* b);
PlanView make_plan_view(const cf_geom* g, const cf_batch* b, void* plan);
int validate(const cf_geom* g, const cf_batch* b);
int sm_count();
// Index of the current device for per-device caches (attributes such as the dynamic shared memory
// limit of a kernel and the SM count belong to a device, not to the process); -1 if unknown.
constexpr int kMaxDevices = 64;
int current_device();
// One flag per device: true once the calling site has configured its kernel on that device.
struct PerDeviceOnce {
    bool done[kMaxDevices] = {};
};
// Sets the dynamic shared memory limit of `kernel` once per device; CF_OK or CF_ERR_CUDA.
template <typename K>
int configure_smem_once(PerDeviceOnce& once, K kernel, int bytes) {
    const int dev = current_device();
    if (dev >= 0 && once.done[dev]) return CF_OK;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess)
        return CF_ERR_CUDA;
    if (dev >= 0) once.done[dev] = true;
    return CF_OK;
}
// Launches a kernel that may be scheduled while earlier kernels of the stream still run (programmatic stream
// serialisation).  Kernels call chain_next() before their own chain_wait(), so a kernel may be resident while any number of
// its predecessors are running or waiting themselves: until chain_wait() it touches no global memory at all, whoever wrote
// it (its own parameters and shared memory are all it may use), and every kernel launched this way executes chain_wait()
// before it ends, so that a chain stays ordered.  Takes the launch latency (1 to 1.5 us) out of chains of kernels that run
// for a few microseconds each.
template <typename... P, typename... A>
int launch_chained_clusters(void (*kernel)(P...), dim3 grid, int threads, size_t smem, unsigned cluster, cudaStream_t stream, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;       // clusters along x
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...) == cudaSuccess ? CF_OK : CF_ERR_CUDA;
}
template <typename... P, typename... A>
int launch_chained(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t stream, A... args) {
    return launch_chained_clusters(kernel, grid, threads, smem, 1, stream, args...);
}
int choose_splits(const cf_geom* g, const cf_batch* b, int n_layers);
int tiles_per_request_bound(const cf_batch* b);

// Partial results of the attention kernels, one slice per split, merged by the combine kernel.
// All logits are in base-2 units: t = (q.k) * softmax_scale * log2(e).
// A call covers n_layers layers; (layer, request) pairs are numbered lb = layer * B + request.
struct AttnWorkspace {
    float* part_o;     // [L*B][n_splits][Hq*Lq][D] sum_t 2^(t - m) v_t, not normalised (unset if m = -inf)
    float* part_m;     // [L*B][n_splits][Hq*Lq]    reference maximum m (-inf if the part is empty)
    float* part_l;     // [L*B][n_splits][Hq*Lq]    sum_t 2^(t - m)
    uint16_t* part_low; // [slots][D]               tensor-core path: low halves of part_o's numbers, of rows that have them
    float* tile_lse2;  // [L][max_tiles][Hq*Lq]     log2 of sum over the tile's tokens of 2^t
    float* row_lse2;   // [L*B][Hq*Lq]              log2 of the full softmax denominator
    int* marks;        // [shares][8]               tensor-core path: what a share leaves for the merge (ShareHead, cf_attn_line.cuh)
    int n_splits;
    int n_layers;
    int max_tiles;     // tile slots per layer in tile_lse2
    int rg_rows;       // query rows of a row tile of the tensor-core kernel, whose parts are numbered by share (cf_attn_tc.cu)
    // Key blocks besides the documents (the query-self block, a shared prefix cache) of a call that has some.
    // self_mode 1 (CUDA-core path): the blocks are one more part, (self_m, self_l, self_o) like (part_m, part_l,
    // part_o).  On the tensor-core path they are further key tiles, and part_ld holds every part's sum over the
    // documents' keys alone.
    float* self_o;     // [L*B][Hq*Lq][D]
    float* self_m;     // [L*B][Hq*Lq]
    float* self_l;     // [L*B][Hq*Lq]
    float* part_ld;    // like part_l, the documents' keys only (tensor-core path with further key blocks)
    int self_mode;
};
// low_halves = false: without part_low (the size that a limit stands on).
// part_layers > 0: the partial results (and the further key blocks' buffers) are sized for that many layers only, the
// per-tile and per-row log-sum-exps for n_layers (calls that fill one layer slot at a time and score the slots later).
size_t attn_workspace_layout(const cf_geom* g, const cf_batch* b, int n_splits, int n_layers, bool with_self,
                             AttnWorkspace* ws, void* base, int part_layers = 0, bool low_halves = true);

// Where the layers of a call sit (element strides between consecutive layers).
struct LayerSpan {
    int n_layers;
    long long q_stride, kv_stride, out_stride;
};

// ---- launchers (each returns a CF_* code) -------------------------------------------------
int launch_plan(const GeomView& gv, const BatchView& bv, const PlanView& pv, int mode,
                const int* order, const int* kept_count, int query_start, const float* score_accum,
                int keep, const int* keep_per_request, int strategy, float* clear_scores, cudaStream_t stream);
int launch_merge_attn(const cf_geom* g, long long n_rows, int q_len, const void* out_a, const float* lse_a,
                      const void* out_b, const float* lse_b, void* out, float* lse, cudaStream_t stream);
int launch_wait_probe(const PlanView& pv, long long limit_cycles, cudaStream_t stream);
int launch_reposition(const cf_geom* g, const cf_batch* b, const PlanView& pv, int n_layers,
                      long long layer_stride, const void* k_in, void* k_out, cudaStream_t stream);
int launch_assemble(const cf_geom* g, const cf_batch* b, const PlanView& pv, int n_layers, long long layer_stride,
                    long long self_stride, int out_rows, const void* k_in, const void* v_in, const void* k_self,
                    const void* v_self, void* k_out, void* v_out, int* final_rows, cudaStream_t stream);
int launch_attn_simt(const cf_geom* g, const cf_batch* b, const PlanView& pv, const LayerSpan& span,
                     const void* q, const void* k, const void* v, float scale_log2,
                     const AttnWorkspace& ws, cudaStream_t stream);
int launch_attn_tc(const cf_geom* g, const cf_batch* b, const PlanView& pv, const LayerSpan& span,
                   const void* q, const void* k, const void* v, const void* k_self, const void* v_self,
                   long long self_stride, const void* k_prefix, const void* v_prefix, long long prefix_stride,
                   int prefix_len, float scale_log2, const AttnWorkspace& ws, void* out, float* lse, cudaStream_t stream);
int attn_tc_row_tile(const cf_geom* g, const cf_batch* b);
size_t attn_tc_part_rows();
bool attn_tc_supported(const cf_geom* g, const cf_batch* b);
// One query row per head over the final caches of a decoding step (doc_offsets: of the decode plan).
bool decode_attn_supported(const cf_geom* g);
size_t decode_attn_workspace_bytes(const cf_geom* g, int n_requests, int n_layers);
int launch_decode_attn(const cf_geom* g, int n_requests, int cache_rows, int n_layers, const int* doc_offsets, const LayerSpan& span,
                       const void* q, const void* k, const void* v, float scale_log2, void* out, float* lse,
                       void* workspace, cudaStream_t stream);
int launch_combine(const cf_geom* g, const cf_batch* b, const PlanView& pv, const LayerSpan& span,
                   const AttnWorkspace& ws, void* out, float* lse, cudaStream_t stream);
int launch_self_block(const cf_geom* g, const cf_batch* b, const LayerSpan& span, long long self_stride,
                      const void* q, const void* k_self, const void* v_self, const void* k_prefix, const void* v_prefix,
                      long long prefix_stride, int prefix_len, float scale_log2, const AttnWorkspace& ws,
                      cudaStream_t stream);
// Shared body of the attention entry points (k_self = v_self = null: cached documents only).
int run_attn_layers(const cf_geom* geom, const cf_batch* batch, const void* plan, const LayerSpan& span,
                    const void* q, const void* k_cache, const void* v_cache, const void* k_self,
                    const void* v_self, long long self_stride, float softmax_scale,
                    void* out, float* lse, float* doc_scores, float* score_accum, void* workspace,
                    size_t workspace_bytes, cudaStream_t stream, const void* k_prefix = nullptr,
                    const void* v_prefix = nullptr, long long prefix_stride = 0, int prefix_len = 0, int slot = -1,
                    int n_slots = 0, int decode_cache_rows = 0);
// Document scores of the layers held in a workspace: doc_scores[l] = s^l (optional), S += s^l in layer order.
int launch_scores(const cf_geom* g, const cf_batch* b, const PlanView& pv, const AttnWorkspace& ws, float* doc_scores,
                  float* score_accum, cudaStream_t stream);

// Arguments of the cache-construction attention kernels (cf_document_prefill_attn).
struct DocAttnArgs {
    int n_docs, n_layers, max_doc_len, prefix_len, n_q_heads, n_kv_heads;
    long long total_tokens, token_stride, q_layer_stride, kv_layer_stride, prefix_layer_stride, out_layer_stride;
    const int* doc_offsets;
    float scale_log2;
};
int launch_docattn_simt(const cf_geom* g, const DocAttnArgs& a, const void* q, const void* k, const void* v,
                        const void* kp, const void* vp, void* out, float* lse, cudaStream_t stream);
bool docattn_tc_supported(const cf_geom* g, const cf_doc_batch* docs);
int launch_docattn_tc(const cf_geom* g, const DocAttnArgs& a, const void* q, const void* k, const void* v,
                      const void* kp, const void* vp, void* out, float* lse, int* status, cudaStream_t stream);
int attn_path();

// ---- device helpers -----------------------------------------------------------------------
// Every earlier kernel of the stream is complete and its writes are visible (returns at once for an ordinary launch).
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// The successor in the stream may be scheduled on what this grid leaves free.
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ float to_float(float x) { return x; }
__device__ __forceinline__ float to_float(__nv_bfloat16 x) { return __bfloat162float(x); }
template <typename T> __device__ __forceinline__ T from_float(float x);
template <> __device__ __forceinline__ float from_float<float>(float x) { return x; }
template <> __device__ __forceinline__ __nv_bfloat16 from_float<__nv_bfloat16>(float x) {
    return __float2bfloat16_rn(x);
}

// Eq. 2 on one slice (a, b) with (c, s) = cos, sin of the delta angle; fp32, fused multiply-adds.
__device__ __forceinline__ void rotate_pair(float a, float b, float c, float s, float& ya, float& yb) {
    ya = fmaf(a, c, -(b * s));
    yb = fmaf(a, s, b * c);
}

}  // namespace cf
