// Attention of one new token over the final caches (Algorithm 2, Phase 3), bf16 storage, head_dim 128.
//
// One query row per head streams the whole cache once: 2 to 14 flops per byte, so the pass is bound by HBM, and for the
// short caches that are left after pruning by latency.  Keys and values go from global memory straight to registers in
// the fragment order of mma.sync (no shared-memory staging, no tensor maps, no tensor memory to allocate); the matrix
// instruction is there because seven query heads per kv head would otherwise cost more CUDA-core issue slots than the
// stream leaves.  A warp takes 16 keys at a time:
//   S = Q K^T  m16n8k16, rows = query heads of the kv head; the contraction index is permuted so that a lane's 16-byte
//              load of a key row is two k-steps of its B fragment (the query fragment uses the same permutation)
//   O^T += V^T P^T  m16n8k16, rows = dims: a lane's 16-byte loads of value rows 2t, 2t+1, 2t+8, 2t+9 are paired by byte
//              permutes into A fragments, and S's accumulators are P^T's B fragments without moving a register
// The loads of the next keys are issued as soon as S has consumed the current ones, those of the next values behind PV:
// a warp always has 4 to 8 KB in flight, twelve warps per SM twice what the bandwidth-delay product asks for.
// The rows of a (layer, request, kv head) are split over the CTAs of a cluster, which merge through distributed shared
// memory: one launch per call, no workspace traffic.  Longer caches and larger batches are cut differently: all steps of
// all units on one line, one equal share per resident CTA, so that neither requests of unequal length nor a unit count
// that is no multiple of the SMs leaves a last wave; units cut between shares meet in a merge kernel.
// Measured (us per layer, the tensor-core kernel of the query-time path before it and this one): 1 request x 1011 rows,
// 12/2 heads 11.9 -> 5.4; 8 x 2764, 32/32 heads 87 -> 45.4 (5.9 TB/s); 4 x 16000, 28/4 heads 32.5 -> 24.5, eight layers
// per call 20.9 -> 16.9 (6.6 TB/s); 8 x 21600, 32/32 heads 359 -> 322 (6.7 TB/s).
#include <algorithm>

#include "cf_common.cuh"

namespace cf {

namespace {

constexpr int kDecThreads = 128;                   // four warps per CTA, three CTAs per SM
constexpr int kDecWarps = kDecThreads / 32;
constexpr int kDecDim = 128;
constexpr int kStepKeys = 16;
constexpr int kMaxCluster = 8;
constexpr float kDecRescale = 8.0f;                // log2 units: the reference maximum moves only beyond this

struct DecodeArgs {
    const __nv_bfloat16 *q, *k, *v;
    __nv_bfloat16* out;
    float* lse;
    const int* doc_offsets;                        // of the decode plan: request b uses rows [2b] .. [2b + 1) of the store
    long long q_stride, kv_stride, out_stride;     // elements between layers
    int n_requests, cache_rows, n_q_heads, n_kv_heads, row_tiles, group;   // group: query heads of a kv head
    Divisor by_requests, by_row_tiles;
    float scale_log2;
    float *part_o, *part_m, *part_l;               // parts of units that lie in several shares of the line
    int2* unit_parts;                              // [units] first share of a unit and the parts it was cut into (0: not cut)
};

__device__ __forceinline__ uint4 load_row(const __nv_bfloat16* p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ void mma16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ float exp2_fast(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&h);
}
__device__ __forceinline__ uint32_t word(const uint4& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// A float of CTA `rank`'s copy of the shared variable at `addr`.
__device__ __forceinline__ float peer_float(uint32_t addr, uint32_t rank) {
    float v;
    asm volatile("{\n.reg .b32 a;\nmapa.shared::cluster.u32 a, %1, %2;\nld.shared::cluster.f32 %0, [a];\n}" : "=f"(v) : "r"(addr), "r"(rank));
    return v;
}
__device__ __forceinline__ float2 peer_float2(uint32_t addr, uint32_t rank) {
    float2 v;
    asm volatile("{\n.reg .b32 a;\nmapa.shared::cluster.u32 a, %2, %3;\nld.shared::cluster.v2.f32 {%0, %1}, [a];\n}" : "=f"(v.x), "=f"(v.y) : "r"(addr), "r"(rank));
    return v;
}

// A run of 16-key steps of one unit (layer, request, kv head, tile of query heads).
struct Segment {
    int lb, head0, n_heads, kvh, used, s_begin, s_end, steps;
    int unit;                                      // its number: (layer * B + request) * tiles + kv head and tile
};

// Where the steps of all units lie on one line (order: layer, request, kv head and tile, step), which is cut into equal shares.
struct Line {
    const int* pref;                               // [n_requests + 1] prefix sums of the requests' steps
    int n_requests, tiles;                         // tiles = kv heads * tiles of query heads
    int per_layer;
    int n_shares, each, rest;                      // equal shares: the first `rest` of them hold one step more
    __device__ __forceinline__ int cut(int c) const { return c * each + min(c, rest); }
    __device__ __forceinline__ int share_of(int x) const {
        const int y = x - rest * (each + 1);
        return y < 0 ? x / (each + 1) : rest + y / each;
    }
};

constexpr int kMinSteps = 12;                      // three steps per warp
constexpr int kMaxStreamRequests = 256;

// Prefix sums of the requests' steps into shared memory; every thread of the block calls it.
__device__ __forceinline__ Line make_line(const DecodeArgs& a, int* s_pref, int n_layers, int max_shares) {
    if (threadIdx.x < 32) {
        int carry = 0;
        for (int b0 = 0; b0 < a.n_requests; b0 += 32) {
            const int b = b0 + threadIdx.x;
            int n = b < a.n_requests ? (a.doc_offsets[2 * b + 1] - a.doc_offsets[2 * b] + kStepKeys - 1) / kStepKeys : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int up = __shfl_up_sync(0xffffffffu, n, o);
                if ((int)threadIdx.x >= o) n += up;
            }
            if (b < a.n_requests) s_pref[b + 1] = carry + n;
            carry += __shfl_sync(0xffffffffu, n, 31);
        }
        if (threadIdx.x == 0) s_pref[0] = 0;
    }
    __syncthreads();
    Line line;
    line.pref = s_pref;
    line.n_requests = a.n_requests;
    line.tiles = a.n_kv_heads * a.row_tiles;
    line.per_layer = s_pref[a.n_requests] * line.tiles;
    const int total = line.per_layer * n_layers;
    line.n_shares = max(1, min(max_shares, total / kMinSteps));
    line.each = total / line.n_shares;
    line.rest = total - line.each * line.n_shares;
    return line;
}

// The unit at position x of the line, from that step on up to position `end` at most.
__device__ __forceinline__ Segment segment_at(const DecodeArgs& a, const Line& line, int x, int end, int kq) {
    Segment sg;
    const int layer = x / line.per_layer;
    int r = x - layer * line.per_layer;
    int lo = 0, hi = a.n_requests;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (line.pref[mid] * line.tiles <= r) lo = mid; else hi = mid;
    }
    r -= line.pref[lo] * line.tiles;
    sg.steps = line.pref[lo + 1] - line.pref[lo];
    const int kr = r / sg.steps;
    sg.s_begin = r - kr * sg.steps;
    sg.s_end = min(sg.steps, sg.s_begin + (end - x));
    sg.lb = layer * a.n_requests + lo;
    sg.unit = sg.lb * line.tiles + kr;
    sg.kvh = a.by_row_tiles.quotient(kr);
    const int row_tile = kr - sg.kvh * a.row_tiles, group = a.group;
    sg.head0 = sg.kvh * group + row_tile * kq;
    sg.n_heads = min(kq, group - row_tile * kq);
    sg.used = a.doc_offsets[2 * lo + 1] - a.doc_offsets[2 * lo];
    return sg;
}

// NQ: query heads per CTA in groups of eight (1: up to 8 heads per kv head, 2: up to 16; more heads take further CTAs).
// STREAM = false: a cluster per unit.  STREAM = true: CTA c takes share c of the line of all steps; a unit that lies in
// one share is finished there, a share leaves its part of a unit that began before it in slot 2c of the workspace and
// its part of one that goes on behind it in slot 2c + 1; the share a unit begins in notes into how many parts it was cut.
template <int NQ, bool STREAM>
__global__ void __launch_bounds__(kDecThreads, NQ == 1 ? 3 : 2)
decode_attn_kernel(DecodeArgs a, int n_layers) {
    constexpr int kQ = 8 * NQ, kPitch = kDecDim + 4;
    __shared__ __align__(16) float s_o[kDecWarps][kQ][kPitch];
    __shared__ float s_m[kDecWarps + 1][kQ], s_l[kDecWarps + 1][kQ];      // [kDecWarps]: the CTA's merged values
    __shared__ int s_pref[STREAM ? kMaxStreamRequests + 1 : 1];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int n_cta = STREAM ? 1 : (int)cluster_size(), rank = STREAM ? 0 : (int)cluster_rank();
    chain_next();
    chain_wait();
    Line line;
    Segment sg;
    int x_pos = 0, x_end = 0, used_from = 0, used_to = 0;
    if (STREAM) {
        line = make_line(a, s_pref, n_layers, (int)gridDim.x);
        if ((int)blockIdx.x >= line.n_shares) return;
        x_pos = line.cut(blockIdx.x);
        x_end = line.cut(blockIdx.x + 1);
        sg = segment_at(a, line, x_pos, x_end, kQ);
    } else {
        const int group = a.group;
        sg.kvh = a.by_row_tiles.quotient(blockIdx.y);
        const int row_tile = blockIdx.y - sg.kvh * a.row_tiles;
        sg.lb = blockIdx.z;
        sg.head0 = sg.kvh * group + row_tile * kQ;
        sg.n_heads = min(kQ, group - row_tile * kQ);
        const int b = a.by_requests.remainder(sg.lb);
        used_from = a.doc_offsets[2 * b];
        used_to = a.doc_offsets[2 * b + 1];
        // The warps of the cluster take the steps in turn: a warp's first one is known before the rows in use are, and its loads
        // travel with theirs.  Rows of the slot that are not in use are masked, their values replaced by zeros.  (Equal runs of steps,
        // cut once the rows were known, by divisions out of registers: with the append a layer of 1011 rows, 12/2 heads, took 7.6 us,
        // this way 6.6, of which 0.3 are the append's, which loads its first piece together with the number of rows.  Slots with 20 rows
        // in use or fewer pay 0.3 to 0.6 us for steps that are loaded and not needed.)
        sg.s_begin = rank * kDecWarps;
        sg.s_end = sg.s_begin + 1 + kDecWarps;                      // (the first step of every warp; the rest below)
        sg.used = a.cache_rows;
    }
    const int stride = n_cta * kDecWarps;

    uint4 qf[NQ][4], kf[2][4], vf[4][2];
    const __nv_bfloat16 *k, *v;
    const size_t pitch = (size_t)a.n_kv_heads * kDecDim;
    auto load_k = [&](int s) {                                      // rows past the end repeat the last one and are masked
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const __nv_bfloat16* p = k + (size_t)min(s * kStepKeys + j * 8 + g, sg.used - 1) * pitch;
#pragma unroll
            for (int c = 0; c < 4; ++c) kf[j][c] = load_row(p + c * 32);
        }
    };
    auto load_v = [&](int s) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const __nv_bfloat16* p = v + (size_t)min(s * kStepKeys + 2 * t + (j & 1) + (j >> 1) * 8, sg.used - 1) * pitch;
            vf[j][0] = load_row(p);
            vf[j][1] = load_row(p + 64);
        }
    };
    // query fragments (chunk c = dims 32c + 8t .. + 7) and the first keys and values of a segment
    auto start = [&]() {
        const int layer = a.by_requests.quotient(sg.lb), b = sg.lb - layer * a.n_requests;
        const __nv_bfloat16* q = a.q + (size_t)layer * a.q_stride + ((size_t)b * a.n_q_heads + sg.head0) * kDecDim + t * 8;
        const size_t base = (size_t)layer * a.kv_stride + ((size_t)b * a.cache_rows * a.n_kv_heads + sg.kvh) * kDecDim;
        k = a.k + base + t * 8;
        v = a.v + base + g * 8;
#pragma unroll
        for (int x = 0; x < NQ; ++x)
#pragma unroll
            for (int c = 0; c < 4; ++c)
                qf[x][c] = x * 8 + g < sg.n_heads ? load_row(q + (size_t)(x * 8 + g) * kDecDim + c * 32) : make_uint4(0u, 0u, 0u, 0u);
        if (sg.s_begin + warp < sg.s_end) {
            load_k(sg.s_begin + warp);
            load_v(sg.s_begin + warp);
        }
    };
    start();
    if (!STREAM) {
        sg.used = used_to - used_from;
        sg.steps = sg.s_end = (sg.used + kStepKeys - 1) / kStepKeys;
        const int valid = sg.used - (sg.s_begin + warp) * kStepKeys;
        if (valid < kStepKeys)
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (2 * t + (j & 1) + (j >> 1) * 8 >= valid) vf[j][0] = vf[j][1] = make_uint4(0u, 0u, 0u, 0u);
    }
    while (true) {
    float o[NQ][8][4], m[NQ], l[NQ];
#pragma unroll
    for (int x = 0; x < NQ; ++x) {
        m[x] = -INFINITY;
        l[x] = 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) o[x][i][e] = 0.f;
    }
    for (int s = sg.s_begin + warp; s < sg.s_end; s += stride) {
        const bool more = s + stride < sg.s_end;
        float sc[2][4];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            sc[j][0] = sc[j][1] = sc[j][2] = sc[j][3] = 0.f;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                mma16816(sc[j], qf[0][c].x, NQ > 1 ? qf[NQ - 1][c].x : 0u, qf[0][c].y, NQ > 1 ? qf[NQ - 1][c].y : 0u, kf[j][c].x, kf[j][c].y);
                mma16816(sc[j], qf[0][c].z, NQ > 1 ? qf[NQ - 1][c].z : 0u, qf[0][c].w, NQ > 1 ? qf[NQ - 1][c].w : 0u, kf[j][c].z, kf[j][c].w);
            }
        }
        if (more) load_k(s + stride);
        const int valid = sg.used - s * kStepKeys;                     // keys of this step that exist
        uint32_t p[NQ][2];
#pragma unroll
        for (int x = 0; x < NQ; ++x) {                              // query 8x + g; keys 2t, 2t+1, 2t+8, 2t+9
            float e[4] = {sc[0][2 * x] * a.scale_log2, sc[0][2 * x + 1] * a.scale_log2, sc[1][2 * x] * a.scale_log2, sc[1][2 * x + 1] * a.scale_log2};
            if (valid < kStepKeys) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (2 * t + (i & 1) + (i >> 1) * 8 >= valid) e[i] = -INFINITY;
            }
            float mx = fmaxf(fmaxf(e[0], e[1]), fmaxf(e[2], e[3]));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
            const bool move = mx > m[x] + kDecRescale;              // first step: m = -inf
            if (__any_sync(0xffffffffu, move)) {
                float alpha = 1.f;
                if (move) {
                    alpha = exp2_fast(m[x] - mx);
                    m[x] = mx;
                }
                l[x] *= alpha;
                // the accumulators' columns are queries 8x + 2t and 8x + 2t + 1
                const float a0 = __shfl_sync(0xffffffffu, alpha, 8 * t), a1 = __shfl_sync(0xffffffffu, alpha, 8 * t + 4);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    o[x][i][0] *= a0;
                    o[x][i][1] *= a1;
                    o[x][i][2] *= a0;
                    o[x][i][3] *= a1;
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) e[i] = exp2_fast(e[i] - m[x]);
            l[x] += (e[0] + e[1]) + (e[2] + e[3]);
            p[x][0] = pack2(e[0], e[1]);
            p[x][1] = pack2(e[2], e[3]);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int i = 0; i < 4; ++i) {                           // dims 64h + 8g + 2i and + 2i + 1
                const uint32_t a0 = __byte_perm(word(vf[0][h], i), word(vf[1][h], i), 0x5410), a1 = __byte_perm(word(vf[0][h], i), word(vf[1][h], i), 0x7632);
                const uint32_t a2 = __byte_perm(word(vf[2][h], i), word(vf[3][h], i), 0x5410), a3 = __byte_perm(word(vf[2][h], i), word(vf[3][h], i), 0x7632);
#pragma unroll
                for (int x = 0; x < NQ; ++x) mma16816(o[x][h * 4 + i], a0, a1, a2, a3, p[x][0], p[x][1]);
            }
        if (more) load_v(s + stride);
    }

    // the next segment's first loads travel under the merge of this one
    const Segment done = sg;
    bool more_segments = false;
    if (STREAM) {
        x_pos += sg.s_end - sg.s_begin;
        more_segments = x_pos < x_end;
        if (more_segments) {
            sg = segment_at(a, line, x_pos, x_end, kQ);
            start();
        }
    }
    // ---- merge: the four warps, then the CTAs of the cluster
#pragma unroll
    for (int x = 0; x < NQ; ++x) {
        l[x] += __shfl_xor_sync(0xffffffffu, l[x], 1);
        l[x] += __shfl_xor_sync(0xffffffffu, l[x], 2);
        if (t == 0) {
            s_m[warp][8 * x + g] = m[x];
            s_l[warp][8 * x + g] = l[x];
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int d = h * 64 + g * 8 + 2 * i;
                *reinterpret_cast<float2*>(&s_o[warp][8 * x + 2 * t][d]) = make_float2(o[x][h * 4 + i][0], o[x][h * 4 + i][2]);
                *reinterpret_cast<float2*>(&s_o[warp][8 * x + 2 * t + 1][d]) = make_float2(o[x][h * 4 + i][1], o[x][h * 4 + i][3]);
            }
    }
    __syncthreads();
    if (tid < kQ) {
        float mm = s_m[0][tid];
#pragma unroll
        for (int w = 1; w < kDecWarps; ++w) mm = fmaxf(mm, s_m[w][tid]);
        float ll = 0.f;
#pragma unroll
        for (int w = 0; w < kDecWarps; ++w) {
            const float f = s_m[w][tid] > -INFINITY ? exp2_fast(s_m[w][tid] - mm) : 0.f;
            ll = fmaf(s_l[w][tid], f, ll);
            s_m[w][tid] = f;                                        // the warp's weight from here on
        }
        s_m[kDecWarps][tid] = mm;
        s_l[kDecWarps][tid] = ll;
    }
    __syncthreads();
    if (!STREAM && n_cta > 1) {
        for (int idx = tid; idx < done.n_heads * (kDecDim / 2); idx += kDecThreads) {   // this CTA's result, in warp 0's rows
            const int r = idx >> 6, d = (idx & 63) * 2;
            float x = 0.f, y = 0.f;
#pragma unroll
            for (int w = 0; w < kDecWarps; ++w) {
                const float2 p = *reinterpret_cast<const float2*>(&s_o[w][r][d]);
                x = fmaf(p.x, s_m[w][r], x);
                y = fmaf(p.y, s_m[w][r], y);
            }
            *reinterpret_cast<float2*>(&s_o[0][r][d]) = make_float2(x, y);
        }
        cluster_sync();
    }
    const uint32_t addr_o = (uint32_t)__cvta_generic_to_shared(&s_o[0][0][0]);
    const uint32_t addr_m = (uint32_t)__cvta_generic_to_shared(&s_m[kDecWarps][0]), addr_l = (uint32_t)__cvta_generic_to_shared(&s_l[kDecWarps][0]);
    const int layer = a.by_requests.quotient(done.lb), b = done.lb - layer * a.n_requests;
    const bool whole = !STREAM || (done.s_begin == 0 && done.s_end == done.steps);
    if (STREAM && tid == 0 && done.s_begin == 0)                    // x_pos: the position behind this segment
        a.unit_parts[done.unit] = make_int2((int)blockIdx.x, whole ? 0 : line.share_of(x_pos - done.s_end + done.steps - 1) - (int)blockIdx.x + 1);
    // every CTA of the cluster writes its share of the (head, dim pair) items
    for (int idx = rank * kDecThreads + tid; idx < done.n_heads * (kDecDim / 2); idx += n_cta * kDecThreads) {
        const int r = idx >> 6, d = (idx & 63) * 2;
        float x = 0.f, y = 0.f, mm, ll;
        if (!STREAM && n_cta > 1) {
            float mr[kMaxCluster];
            mm = -INFINITY;
            ll = 0.f;
#pragma unroll
            for (int c = 0; c < kMaxCluster; ++c) {
                mr[c] = c < n_cta ? peer_float(addr_m + r * 4, c) : -INFINITY;
                mm = fmaxf(mm, mr[c]);
            }
#pragma unroll
            for (int c = 0; c < kMaxCluster; ++c)
                if (c < n_cta && mr[c] > -INFINITY) {
                    const float f = exp2_fast(mr[c] - mm);
                    const float2 p = peer_float2(addr_o + (r * kPitch + d) * 4, c);
                    ll = fmaf(peer_float(addr_l + r * 4, c), f, ll);
                    x = fmaf(p.x, f, x);
                    y = fmaf(p.y, f, y);
                }
        } else {
            mm = s_m[kDecWarps][r];
            ll = s_l[kDecWarps][r];
#pragma unroll
            for (int w = 0; w < kDecWarps; ++w) {
                const float2 p = *reinterpret_cast<const float2*>(&s_o[w][r][d]);
                x = fmaf(p.x, s_m[w][r], x);
                y = fmaf(p.y, s_m[w][r], y);
            }
        }
        if (!whole) {
            const size_t slot = ((size_t)2 * blockIdx.x + (done.s_begin == 0 ? 1 : 0)) * kQ + r;
            *reinterpret_cast<float2*>(a.part_o + slot * kDecDim + d) = make_float2(x, y);
            if (d == 0) {
                a.part_m[slot] = mm;
                a.part_l[slot] = ll;
            }
        } else {
            const float inv = ll > 0.f ? 1.f / ll : 0.f;
            *reinterpret_cast<uint32_t*>(a.out + (size_t)layer * a.out_stride + ((size_t)b * a.n_q_heads + done.head0 + r) * kDecDim + d) = pack2(x * inv, y * inv);
            if (d == 0 && a.lse) a.lse[(size_t)done.lb * a.n_q_heads + done.head0 + r] = (ll > 0.f ? mm + log2f(ll) : -INFINITY) * kLn2;
        }
    }
    if (!more_segments) break;
    __syncthreads();                                                // the shared results have been read
    }
    if (!STREAM && n_cta > 1) cluster_sync();                       // nobody leaves while its shared memory is being read
}

// Units cut over several shares: one block per (layer, request, head) merges the parts, its warps every fourth one.  How a
// unit was cut is read from what the attention kernel left.  Made again from the plan (dependent loads, a scan and a barrier
// behind the wait) it took a step of 32 layers of 8 x 2764 rows, 32/32 heads, from 1526 to 1588 us; this way 1574 to 1581.
__global__ void __launch_bounds__(kDecThreads)
decode_merge_kernel(DecodeArgs a, int kq) {
    __shared__ __align__(16) float s_w[4][kDecDim];
    __shared__ float s_ml[2][4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, row = blockIdx.x;            // (layer * B + request) * heads + head
    const int lb = row / a.n_q_heads, h = row - lb * a.n_q_heads, layer = lb / a.n_requests, b = lb - layer * a.n_requests;
    const int group = a.n_q_heads / a.n_kv_heads, kvh = h / group, in_group = h - kvh * group, row_tile = in_group / kq, r = in_group - row_tile * kq;
    chain_next();
    chain_wait();
    const int2 cut = a.unit_parts[(lb * a.n_kv_heads + kvh) * a.row_tiles + row_tile];
    if (cut.y == 0) return;                                         // finished by its one share
    const int c0 = cut.x, c1 = c0 + cut.y - 1;
    float mm = -INFINITY, ll = 0.f, acc[4] = {0.f, 0.f, 0.f, 0.f};
    for (int cb = c0 + warp; cb <= c1; cb += 16) {                  // four parts in flight
        float mp[4], lp[4];
        float4 p[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int c = cb + 4 * u;
            const size_t slot = ((size_t)2 * c + (c == c0 ? 1 : 0)) * kq + r;
            mp[u] = -INFINITY;
            if (c <= c1) {
                mp[u] = a.part_m[slot];
                lp[u] = a.part_l[slot];
                p[u] = *reinterpret_cast<const float4*>(a.part_o + slot * kDecDim + lane * 4);
            }
        }
        const float m_new = fmaxf(fmaxf(mm, fmaxf(mp[0], mp[1])), fmaxf(mp[2], mp[3]));
        if (m_new == -INFINITY) continue;
        const float keep = exp2_fast(mm - m_new);
        mm = m_new;
        ll *= keep;
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i] *= keep;
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (mp[u] > -INFINITY) {
                const float w = exp2_fast(mp[u] - m_new);
                ll = fmaf(lp[u], w, ll);
                acc[0] = fmaf(p[u].x, w, acc[0]);
                acc[1] = fmaf(p[u].y, w, acc[1]);
                acc[2] = fmaf(p[u].z, w, acc[2]);
                acc[3] = fmaf(p[u].w, w, acc[3]);
            }
    }
    *reinterpret_cast<float4*>(&s_w[warp][lane * 4]) = make_float4(acc[0], acc[1], acc[2], acc[3]);
    if (lane == 0) {
        s_ml[0][warp] = mm;
        s_ml[1][warp] = ll;
    }
    __syncthreads();
    const float m_all = fmaxf(fmaxf(s_ml[0][0], s_ml[0][1]), fmaxf(s_ml[0][2], s_ml[0][3]));
    float l_all = 0.f, x = 0.f;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        const float f = s_ml[0][w] > -INFINITY ? exp2_fast(s_ml[0][w] - m_all) : 0.f;
        l_all = fmaf(s_ml[1][w], f, l_all);
        x = fmaf(s_w[w][threadIdx.x], f, x);
    }
    const float inv = l_all > 0.f ? 1.f / l_all : 0.f;
    a.out[(size_t)layer * a.out_stride + ((size_t)b * a.n_q_heads + h) * kDecDim + threadIdx.x] = __float2bfloat16_rn(x * inv);
    if (threadIdx.x == 0 && a.lse) a.lse[row] = (l_all > 0.f ? m_all + log2f(l_all) : -INFINITY) * kLn2;
}

}  // namespace

bool decode_attn_supported(const cf_geom* g) { return g->dtype == CF_BF16 && g->head_dim == kDecDim; }

static int stream_shares(const cf_geom* g) { return (g->n_q_heads / g->n_kv_heads > 8 ? 2 : 3) * sm_count(); }   // one wave

// Units of a call: (layer, request, kv head, tile of query heads).
static long long decode_units(const cf_geom* g, int n_requests, int n_layers) {
    const int group = g->n_q_heads / g->n_kv_heads, kq = group > 8 ? 16 : 8;
    return (long long)n_layers * n_requests * g->n_kv_heads * ((group + kq - 1) / kq);
}

// Workspace of a call: two parts per share, and how every unit was cut.
size_t decode_attn_workspace_bytes(const cf_geom* g, int n_requests, int n_layers) {
    const int kq = g->n_q_heads / g->n_kv_heads > 8 ? 16 : 8;
    return (size_t)stream_shares(g) * 2 * kq * (kDecDim + 2) * sizeof(float) + (size_t)decode_units(g, n_requests, n_layers) * sizeof(int2);
}

int launch_decode_attn(const cf_geom* g, int n_requests, int cache_rows, int n_layers, const int* doc_offsets, const LayerSpan& span,
                       const void* q, const void* k, const void* v, float scale_log2, void* out, float* lse, void* workspace,
                       cudaStream_t stream) {
    const int group = g->n_q_heads / g->n_kv_heads;
    const bool wide = group > 8;
    const int kq = wide ? 16 : 8, row_tiles = (group + kq - 1) / kq;
    if ((long long)g->n_kv_heads * row_tiles > 65535 || (long long)n_requests * n_layers > 65535) return CF_ERR_INVALID_ARG;
    const int shares = stream_shares(g);
    float* part_o = static_cast<float*>(workspace);
    float* part_m = part_o + (size_t)shares * 2 * kq * kDecDim;
    float* part_l = part_m + (size_t)shares * 2 * kq;
    int2* unit_parts = reinterpret_cast<int2*>(part_l + (size_t)shares * 2 * kq);
    const DecodeArgs a = {static_cast<const __nv_bfloat16*>(q), static_cast<const __nv_bfloat16*>(k), static_cast<const __nv_bfloat16*>(v),
                          static_cast<__nv_bfloat16*>(out), lse, doc_offsets, span.q_stride, span.kv_stride, span.out_stride, n_requests,
                          cache_rows, g->n_q_heads, g->n_kv_heads, row_tiles, group, Divisor(n_requests), Divisor(row_tiles), scale_log2, part_o, part_m, part_l, unit_parts};
    const long long units = decode_units(g, n_requests, n_layers);
    // A cluster per unit where one wave of clusters leaves a warp a few steps, the stream of equal shares for everything longer;
    // the line is eight steps.  Measured (us per layer with the append, cold, cluster against stream, the steps of a warp in
    // brackets): 2 units, 1000 rows (2) 9.6 / 12.4, 2000 (4) 11.9 / 12.2, 3000 (6) 14.1 / 12.1; 8 units, 2000 (4) 12.4 / 13.2, 3000 (6)
    // 14.7 / 13.7; 16 units, 3000 (6) 14.0 / 15.2, 4000 (8) 17.5 / 17.0; 32 units, 3000 (6) 18.8 / 19.1, 4000 (8) 21.6 / 21.6; 256
    // units, 500 (8) 20.5 / 21.5, 750 (12) 24.0 / 23.6, 2000 (31) 48.5 / 44.7.  So the two meet at four steps for a few units and
    // at ten for many.  What the rule sees is the slot, not the rows in use, which are known on the device only: 1011 rows of 2
    // units took 8.1 us in a slot of 1075 rows and 10.1 in one of 20 000.  (Figures of the kernel before a warp's first step was loaded
    // early, which takes about 0.7 us off the cluster's side.)
    int cluster = 1;
    while (cluster < kMaxCluster && units * cluster * 2 <= shares) cluster *= 2;
    bool stream_k = cache_rows > kStepKeys * kDecWarps * cluster * 8;
    // the line fits 32-bit arithmetic and the prefix sums their shared memory
    if (n_requests > kMaxStreamRequests || units * (cache_rows / kStepKeys + 1) > 0x7fffffffLL) stream_k = false;
    if (stream_k) {
        const int rc = wide ? launch_chained(decode_attn_kernel<2, true>, dim3(shares), kDecThreads, 0, stream, a, n_layers)
                            : launch_chained(decode_attn_kernel<1, true>, dim3(shares), kDecThreads, 0, stream, a, n_layers);
        if (rc != CF_OK) return rc;
        return launch_chained(decode_merge_kernel, dim3((unsigned)(n_layers * n_requests * g->n_q_heads)), kDecThreads, 0, stream, a, kq);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)cluster, (unsigned)(g->n_kv_heads * row_tiles), (unsigned)(n_requests * n_layers));
    cfg.blockDim = dim3(kDecThreads);
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cluster;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    const cudaError_t rc = wide ? cudaLaunchKernelEx(&cfg, decode_attn_kernel<2, false>, a, n_layers) : cudaLaunchKernelEx(&cfg, decode_attn_kernel<1, false>, a, n_layers);
    return rc == cudaSuccess ? CF_OK : CF_ERR_CUDA;
}

}  // namespace cf
