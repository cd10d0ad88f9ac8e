// Fused re-position + query-prefill attention on the Blackwell tensor cores (bf16, head_dim 128).
//
// Eq. 5 fused into Eq. 1: key tiles are streamed from the un-repositioned store by TMA into 128B-swizzled shared memory,
// rotated there in place by their document's delta (fp32, one rounding: bit for bit what cf_reposition_keys writes) and
// handed to the tensor cores.
//
// Work: the key tiles (runs of at most kTile rows of one document, from the plan) of every (layer, request, kv head, tile of
// at most 128 query rows) laid on one line and cut into equal shares, one per SM: a CTA walks its share, which may end in the
// middle of a unit and hold several whole ones.  A unit inside one share is finished there; parts of others meet in the merge
// kernel.  With one CTA per (unit, range) as before, 256 units on 148 SMs left a quarter of the last wave idle and every
// wave paid set-up and epilogue again.
//   warps 0-7            two softmax warpgroups, alternate key tiles of the same rows (thread = query row = TMEM lane)
//   warps 8, 10, 11, 13-15   key rotation in shared memory
//   warp 9               key, value and rotation-table loads     warp 12  MMA issue
// The two single-warp roles issue a few dozen dependent instructions per tile and are what the CTA waits for when they have
// to share their scheduler (warp index mod 4) with too much arithmetic: each has one rotation warp beside it, the other two
// schedulers have two (all six on three schedulers: 8 x 15 documents, 32 heads 101 us, this way 90).  Tile descriptions are fetched a tile ahead, and what the other roles need to know about a tile they find in shared memory.
// Tensor memory: O (128 columns), the query tile (64: as the A operand of QK^T it costs no shared-memory reads, which this
// kernel has none to spare of), three S buffers of 96 columns; P (bf16) overwrites the S columns already consumed.  S(n + 3) is issued behind PV(n), so a softmax warpgroup that has finished a
// tile finds its next S waiting.
// Softmax: both warpgroups accumulate into one O under one reference per row, the maximum over the first 16 keys of the
// segment.  P and the sums keep their relative precision for logits up to 80 (log2 units) above it and 126 below, so that no
// tile has to look at its maximum before its exponentials.  (A reference 40 above that maximum, which centres the range, costs
// three bits of the exponents and the log-sum-exps: 1.3e-6 off instead of 1.1e-7 for a row of one key.)  A row that does leave
// the range is marked (NaN sum) and computed from scratch over the CTA's own share once the roles have left their loops.
// What bounds it (per 96-key tile and 128 rows, in SM cycles): tensor cores 768 (8 x 48 + 6 x 64), exponentials 768 on
// the shared MUFU, shared memory 1150 (copies 384, rotation 384, QK^T 192, PV 192), so these overlap only if nobody
// waits for a chain.
// Every wait on an mbarrier is bounded; when a wait expires the CTA raises CF_ERR_TIMEOUT in the plan's status word, all
// roles leave their loops, and the CTA frees its tensor memory and exits.  Each barrier has one kind of waiter, which waits
// for every phase in order.
#include <algorithm>
#include <cstddef>

#include "cf_row_group.cuh"
#include "cf_tc_util.cuh"

namespace cf {

namespace {

using namespace tc;

constexpr int kThreads = 512;
constexpr int kRotateWarps = 6;
constexpr int kRowTile = 128;
constexpr int kKvHalf = kTile * 128;               // one 64-column half of a key or value tile
constexpr int kKvBytes = 2 * kKvHalf;
constexpr int kBoxes = kTile / 16;                 // copy boxes are 16, 32, .. kTile rows high
constexpr int kKStages = 6, kVStages = 3;          // with the three S buffers of two warpgroups: everything repeats after six tiles
constexpr int kSBuffers = 3;
constexpr int kMetaRing = 16, kSegRing = 16;
constexpr int kPrefSlots = 48;
constexpr int kLoadWarp = 9, kMmaWarp = 12;
constexpr int kTrigBytes = kD / 2 * 8;
constexpr uint32_t kColO = 0, kColQ = 128, kColS = 192;
constexpr float kSumLimit = 0x1p80f;               // a larger tile sum leaves the range: 2^47 are left for the values and the other tiles
static_assert(kColS + kSBuffers * kTile <= 512, "tensor memory columns");
static_assert(kTile % 16 == 0 && kTile <= 96, "three S buffers");
static_assert(kKStages == 6 && kVStages == 3 && kSBuffers == 3, "rings of one period");

struct StoreMaps {
    CUtensorMap k[kBoxes], v[kBoxes];              // the stores, one map per box height
    CUtensorMap ks, vs;                            // keys and values of the query tokens themselves (whole tiles)
    CUtensorMap kp, vp;                            // keys and values of a shared prefix cache (whole tiles)
};

struct Barriers {
    unsigned long long k_full[kKStages], k_ready[kKStages], k_empty[kKStages], v_empty[kVStages];
    unsigned long long s_full[6], pv_ready[6];                          // [tile mod 6]; pv_ready: P is stored and V has landed
    unsigned long long segment[kSegRing];                               // the description of the segment is there
    unsigned long long q_ready, q_free, o_done, o_free;                 // one phase per segment
    unsigned long long ref_full[2], sum_full[2];                        // [segment parity]
    unsigned int tmem_base;
    volatile int abort_flag;
    volatile int marked;                           // a row of the share has to be computed from scratch
};

// Tile descriptions: flags beside the length, and which keys they are.
constexpr int kFirstOfSegment = 1 << 8, kLastOfSegment = 1 << 9;
constexpr int kKindPrefix = -1, kKindSelf = -2;    // tile index of a prefix tile; kKindSelf - n: n-th tile of the query tokens

// a / b for a >= 0, b > 0 from the reciprocal, exact after its correction: the few divisions on the way to a CTA's first
// copy are a serial chain, and the integer division of the language is three times as long.
__device__ __forceinline__ int quick_div(int a, int b) {
    int q = (int)__fdividef((float)a, (float)b);
    int r = a - q * b;
    while (r < 0) {
        --q;
        r += b;
    }
    while (r >= b) {
        ++q;
        r -= b;
    }
    return q;
}

// The line of all key tiles (order: layer, request, kv head and tile of query rows, key tile).  A request's tiles are its
// documents' (plan), then those of the prefix cache, then those of the query tokens.
struct Line {
    const int *pref, *begin;
    int stride, n_requests, row_tiles, tiles;      // tiles = kv heads * tiles of query rows
    int n_prefix, n_self, per_layer, n_shares, each, rest;
    __device__ __forceinline__ int cut(int c) const { return c * each + min(c, rest); }
    __device__ __forceinline__ int share_of(int x) const {
        const int y = x - rest * (each + 1);
        return y < 0 ? quick_div(x, each + 1) : rest + quick_div(y, each);
    }
};

struct Segment {
    int lb, layer, b, kvh, row0, rows_here;        // unit: query rows row0 .. of the kv head
    int t_begin, t_end, n_unit, n_doc, tile0;      // tiles of the unit this segment covers; documents' tiles; first in the plan
};

// A share has at least two tiles.  Measured, attention and merge of a call (us, a least of 1 / 2 / 3 / 4; larger calls do not
// notice): 25 documents of 160 tokens, 12/2 heads 16.9 / 16.9 / 19.4 / 21.2; 6 documents 14.0 / 14.0 / 14.5 / 14.8; 20 documents of
// 90, 32/8 heads 15.3 / 14.8; 3 of 180, 32/32 heads 13.8 / 12.8; units of three and five tiles, which two do not divide: 3 and 5 of
// 90, 32/8 heads 12.5 / 15.6 and 13.3 / 16.1.  Three and more cost parallelism, between one and two it is even.
constexpr int kMinShare = 2;

// What the line is made from: prefix sums of the requests' tiles (one entry per `stride` requests), and with one entry per
// request also the requests' first tiles in the plan.  Filled by the first warp.
struct Requests {
    int pref[kPrefSlots + 1], begin[kPrefSlots];
};

__device__ __forceinline__ void scan_requests(const BatchView& bv, const PlanView& pv, int extra, Requests& rq) {
    const int lane = threadIdx.x & 31, stride = (bv.n_requests + kPrefSlots - 1) / kPrefSlots;
    int carry = 0;
    for (int b0 = 0; b0 < bv.n_requests; b0 += 32) {
        const int b = b0 + lane;
        int n = 0, begin = 0;
        if (b < bv.n_requests) {
            n = pv.n_tiles[b] + extra;
            if (stride == 1) begin = pv.tile_begin[b];
        }
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int up = __shfl_up_sync(0xffffffffu, n, o);
            if (lane >= o) n += up;
        }
        if (b < bv.n_requests) {
            if (stride == 1) rq.begin[b] = begin;
            if ((b + 1) % stride == 0 || b == bv.n_requests - 1) rq.pref[(b + stride) / stride] = carry + n;
        }
        carry += __shfl_sync(0xffffffffu, n, 31);
    }
    if (lane == 0) rq.pref[0] = 0;
}

__device__ __forceinline__ Line make_line(const BatchView& bv, const AttnWorkspace& ws, const Requests& rq, int n_kv_heads, int row_tiles,
                                          int n_prefix, int n_self, int max_shares) {
    Line line;
    line.pref = rq.pref;
    line.begin = rq.begin;
    line.n_requests = bv.n_requests;
    line.stride = (bv.n_requests + kPrefSlots - 1) / kPrefSlots;
    line.n_prefix = n_prefix;
    line.n_self = n_self;
    line.row_tiles = row_tiles;
    line.tiles = n_kv_heads * line.row_tiles;
    line.per_layer = rq.pref[(bv.n_requests + line.stride - 1) / line.stride] * line.tiles;
    const int total = line.per_layer * ws.n_layers;
    line.n_shares = max(1, min(max_shares, total / kMinShare));
    line.each = quick_div(total, line.n_shares);
    line.rest = total - line.each * line.n_shares;
    return line;
}

__device__ __forceinline__ Segment segment_at(const BatchView& bv, const PlanView& pv, const AttnWorkspace& ws, const Line& line, int group,
                                              int x, int end) {
    Segment sg;
    sg.layer = quick_div(x, line.per_layer);
    int r = x - sg.layer * line.per_layer;
    int lo = 0, hi = (line.n_requests + line.stride - 1) / line.stride;     // the last slot that starts at or before r
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (line.pref[mid] * line.tiles <= r) lo = mid; else hi = mid;
    }
    const int extra = line.n_prefix + line.n_self;
    int b = lo, start = line.pref[lo], n;
    if (line.stride == 1) {
        n = line.pref[b + 1] - start;
        sg.tile0 = line.begin[b];
    } else {
        b = lo * line.stride;
        n = pv.n_tiles[b] + extra;
        while ((start + n) * line.tiles <= r) {
            start += n;
            n = pv.n_tiles[++b] + extra;
        }
        sg.tile0 = pv.tile_begin[b];
    }
    r -= start * line.tiles;
    const int unit = quick_div(r, n);
    sg.n_unit = n;
    sg.n_doc = n - extra;
    sg.t_begin = r - unit * n;
    sg.t_end = min(n, sg.t_begin + (end - x));
    sg.b = b;
    sg.lb = sg.layer * line.n_requests + b;
    sg.kvh = quick_div(unit, line.row_tiles);
    sg.row0 = (unit - sg.kvh * line.row_tiles) * ws.rg_rows;
    sg.rows_here = min(ws.rg_rows, group * bv.q_len - sg.row0);
    return sg;
}

// What a CTA leaves for the merge kernel: the unit that begins in its share and goes on behind it (n_parts = 0: none).
struct ShareHead {
    int n_parts, lb, layer, b, row_first, rows_here, unused[2];          // row_first: of the unit among the rows of a request
};
static_assert(sizeof(ShareHead) == 32, "two 16-byte loads");

struct Shared {
    Barriers bars;
    int4 meta[kMetaRing];                          // tiles in flight: length and flags, tile index or kind, first row, kv head and layer
    Segment segments[kSegRing];                    // of the share
    ShareHead head;
    Line line;
    float ref[2][kRowTile];                        // [segment parity][row]
    alignas(16) float2 trig[kKStages][kD / 2];     // cosines and sines of the documents of the key stages
    float sum[2][2][kRowTile], docs[2][2][kRowTile];   // [segment parity][warpgroup][row]
    Requests requests;
};
constexpr int kSmemBytes = (kKStages + kVStages) * kKvBytes + (int)sizeof(Shared) + 1024;
static_assert(kSmemBytes <= 227 * 1024, "shared memory of one CTA");

// Keys and values of a call outside the tensor maps, for rows that are computed from scratch.
struct RowSources {
    const __nv_bfloat16 *q, *k, *v, *ks, *vs, *kp, *vp;
    long long self_stride, prefix_stride;
    float scale_log2;
    int with_self, prefix_len;
};

// Everything a kernel of this file is told: one constant, so that the rarely taken paths can be handed its address.
struct Params {
    BatchView bv;
    PlanView pv;
    AttnWorkspace ws;
    LayerSpan span;
    RowSources src;
    int n_q_heads, n_kv_heads, row_tiles, n_prefix, n_self, max_shares;   // n_prefix, n_self: key tiles
    Divisor q_len, tiles_of_rows, kv_heads, requests, merge_slices;       // of the batch; merge_slices: of a unit's rows in merge blocks
    __nv_bfloat16* out;
    float* lse;
};

// What row_lse2 holds of a row whose unit was cut, until its parts are merged: the share the unit begins in and the number of its
// parts, as a negative quiet NaN (a denominator that is not a number is written as the positive one).
constexpr uint32_t kPartsOf = 0xffc00000u;
constexpr int kMaxCodedShares = 1 << 10;
__device__ __forceinline__ uint32_t parts_code(int share, int n_parts) { return kPartsOf | ((uint32_t)n_parts << 10) | (uint32_t)share; }
__device__ __forceinline__ bool is_parts_code(uint32_t w) { return (w & kPartsOf) == kPartsOf; }
__device__ __forceinline__ int first_share(uint32_t w) { return (int)(w & (kMaxCodedShares - 1)); }
__device__ __forceinline__ int part_count(uint32_t w) { return (int)((w ^ kPartsOf) >> 10); }
#define CF_PARAMS                                                                                                  \
    [[maybe_unused]] const BatchView& bv = p.bv;                                                                   \
    [[maybe_unused]] const PlanView& pv = p.pv;                                                                    \
    [[maybe_unused]] const AttnWorkspace& ws = p.ws;                                                               \
    [[maybe_unused]] const LayerSpan& span = p.span;                                                               \
    [[maybe_unused]] const RowSources& src = p.src;                                                                \
    [[maybe_unused]] const int n_q_heads = p.n_q_heads, n_kv_heads = p.n_kv_heads;                                 \
    [[maybe_unused]] __nv_bfloat16* const out_all = p.out;                                                         \
[[maybe_unused]] float* const lse = p.lse

// Shared memory of a CTA that computes rows of its share from scratch, over the rings of keys and values.
constexpr int kRowWarps = kThreads / 32;
struct RowTile {                   // where a key tile lies; row j of the query sees its keys up to j - first
    const __nv_bfloat16 *k, *v;
    const float2* trig;            // null: not a document's
    long long pitch;
    int len, first, index;
};
struct RowScratch {
    rows::Stage stage[kRowWarps];  // of every warp
    RowTile tile[kRowWarps][2];    // the current tile and the next one (registers are what the keys and sums need)
    rows::Queries q;
    alignas(16) float o[rows::kGroupRows][kD];
    float m[kRowWarps][rows::kGroupRows], l[kRowWarps][rows::kGroupRows], docs[kRowWarps][rows::kGroupRows];   // of every warp
    Segment sg;
    unsigned todo[kRowTile / 32];  // rows of the segment that are still to be computed
    int row[rows::kGroupRows];     // the group, as rows of the segment
    int n_rows;
    int x;                         // position of the share behind the segment
};
static_assert(sizeof(RowScratch) <= (kKStages + kVStages) * kKvBytes, "over the rings");
static_assert(alignof(RowScratch) == 16 && offsetof(RowScratch, q) % 16 == 0 && offsetof(RowScratch, o) % 16 == 0, "16-byte accesses");

// Up to eight query rows (every set bit of `set`, from row `row0` of the segment on) over the segment's key tiles, every warp
// with every sixteenth tile under a running maximum of its own.  Leaves what the epilogue leaves of a row - a finished row or
// the part of one - and the log-sum-exps of the document tiles.
template <int LAYOUT>
__device__ __forceinline__ void rows_from_scratch(const Params& p, RowScratch& sh, int row0, unsigned set) {
    CF_PARAMS;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, lq = bv.q_len, group = n_q_heads / n_kv_heads, rows_total = n_q_heads * lq;
    if (warp < rows::kGroupRows) {                                  // a row of the group per warp; beyond them the last one again
        const int n_rows = min(rows::kGroupRows, __popc(set)), r = row0 + rows::nth_bit(set, min(warp, n_rows - 1)), row = sh.sg.row0 + r, g = row / lq, j = row - g * lq;
        if (lane == 0) sh.row[warp] = r;
        if (threadIdx.x == 0) sh.n_rows = n_rows;
        if (lane < 16)
            sh.q.put(warp, lane, src.q + (size_t)sh.sg.layer * span.q_stride + (((size_t)sh.sg.b * lq + j) * n_q_heads + sh.sg.kvh * group + g) * kD);
    }
    __syncthreads();
    const int j = (sh.sg.row0 + sh.row[lane >> 2]) % lq;
    rows::Stage& stage = sh.stage[warp];
    RowTile(&tile)[2] = sh.tile[warp];
    auto describe = [&](int t, RowTile& x) {
        if (lane == 0) {
            const int n_doc = sh.sg.n_doc, b = sh.sg.b;
            const long long layer = sh.sg.layer;
            long long pitch = (long long)n_kv_heads * kD, at;
            const __nv_bfloat16 *k = src.k, *v = src.v;
            const float2* trig = nullptr;
            int first = -(1 << 30), index = -1, len;
            if (t < n_doc) {
                index = sh.sg.tile0 + t;
                pitch = bv.token_stride;
                at = layer * span.kv_stride + pv.tile_row0[index] * pitch;
                len = pv.tile_len[index];
                trig = pv.trig + (size_t)pv.tile_doc[index] * (kD / 2);
            } else if (t < n_doc + p.n_prefix) {
                const int row0 = (t - n_doc) * kTile;
                k = src.kp;
                v = src.vp;
                at = layer * src.prefix_stride + row0 * pitch;
                len = min(kTile, src.prefix_len - row0);
            } else {
                first = (t - n_doc - p.n_prefix) * kTile;           // causal mask
                k = src.ks;
                v = src.vs;
                at = layer * src.self_stride + ((long long)b * lq + first) * pitch;
                len = min(kTile, lq - first);
            }
            at += sh.sg.kvh * kD;
            x = {k + at, v + at, trig, pitch, len, first, index};
        }
        __syncwarp();
    };
    auto copy_keys = [&](const RowTile& x, int i) { rows::copy_step(stage.k, x.k + i * x.pitch, x.pitch, x.len - i); };
    auto copy_values = [&](const RowTile& x, int i) { rows::copy_step(stage.v, x.v + i * x.pitch, x.pitch, x.len - i); };
    rows::Group acc;
    acc.clear();
    float docs = 0.f, in_tile = 0.f;                                // the parts of acc.l on documents and on the current tile
    int t = sh.sg.t_begin + warp, i = 0, now = 0;                   // the current tile lies in tile[now]
    if (t < sh.sg.t_end) {
        describe(t, tile[0]);
        copy_keys(tile[0], 0);
        rows::copies_end();
        copy_values(tile[0], 0);
        rows::copies_end();
    }
#pragma unroll 1
    while (t < sh.sg.t_end) {
        rows::Keys keys;
        rows::copies_wait();
        keys.read(stage);
        const int visible = min(tile[now].len, j + 1 - tile[now].first) - i;
        const bool last = i + rows::kStepKeys >= tile[now].len, more = !last || t + kRowWarps < sh.sg.t_end;
        const int next = last ? now ^ 1 : now;                      // the tile of the step behind this one
        i = last ? 0 : i + rows::kStepKeys;                         // and its place there
        if (last && more) describe(t + kRowWarps, tile[next]);
        __syncwarp();                                               // every lane has its fragments
        if (more) copy_keys(tile[next], i);
        rows::copies_end();
        const float2* trig = tile[now].trig;
        if (trig) keys.rotate<LAYOUT>(trig);
        float alpha;
        const float sum = acc.scores(sh.q, keys, visible, src.scale_log2, alpha);
        in_tile = fmaf(in_tile, alpha, sum);
        docs = fmaf(docs, alpha, tile[now].trig ? sum : 0.f);
        rows::copies_wait();
        acc.values(stage);
        __syncwarp();
        if (more) copy_values(tile[next], i);
        rows::copies_end();
        if (last) {
            in_tile = rows::over_keys(in_tile);
            const int index = tile[now].index;
            if (index >= 0 && (lane & 3) == 0)                      // (rows beyond the group's repeat its last one)
                ws.tile_lse2[((size_t)sh.sg.layer * ws.max_tiles + index) * rows_total + (size_t)sh.sg.kvh * group * lq + sh.sg.row0 + sh.row[lane >> 2]] =
                    acc.m + log2f(in_tile);
            in_tile = 0.f;
            t += kRowWarps;
            now = next;
            __syncwarp();                                           // the tile has been read
        }
    }
    acc.l = rows::over_keys(acc.l);
    docs = rows::over_keys(docs);
    if ((lane & 3) == 0) {
        sh.m[warp][lane >> 2] = acc.m;
        sh.l[warp][lane >> 2] = acc.l;
        sh.docs[warp][lane >> 2] = docs;
    }
    __syncthreads();
    // join the warps, in order: a row's reference is the largest of theirs (-inf: nothing to attend)
    float weight[2];                                                // of this warp's rows 2 t and 2 t + 1
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const int r = 2 * (lane & 3) + x;
        float top = sh.m[0][r];
        for (int w = 1; w < kRowWarps; ++w) top = fmaxf(top, sh.m[w][r]);
        weight[x] = sh.m[warp][r] > -INFINITY ? exp2f(sh.m[warp][r] - top) : sh.l[warp][r];   // nothing seen: 0 (or not a number)
    }
    for (int w = 0; w < kRowWarps; ++w) {
        if (w == warp)
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    float2& to = *reinterpret_cast<float2*>(&sh.o[2 * (lane & 3) + x][(i >> 2) * 64 + (lane >> 2) * 8 + 2 * (i & 3)]);
                    const float2 was = w == 0 ? make_float2(0.f, 0.f) : to;
                    to = make_float2(fmaf(acc.o[i][x], weight[x], was.x), fmaf(acc.o[i][x + 2], weight[x], was.y));
                }
        __syncthreads();
    }
    if (warp < sh.n_rows) {                                         // a row per warp, four dims per lane
        float top = sh.m[0][warp], l = 0.f, ld = 0.f;
        for (int w = 1; w < kRowWarps; ++w) top = fmaxf(top, sh.m[w][warp]);
        for (int w = 0; w < kRowWarps; ++w) {
            const float f = sh.m[w][warp] > -INFINITY ? exp2f(sh.m[w][warp] - top) : 1.f;
            l = fmaf(sh.l[w][warp], f, l);
            ld = fmaf(sh.docs[w][warp], f, ld);
        }
        const bool whole = sh.sg.t_end - sh.sg.t_begin == sh.sg.n_unit;
        const int row = sh.sg.row0 + sh.row[warp], g = row / lq, jj = row - g * lq;
        const size_t slot = ((size_t)2 * blockIdx.x + (sh.sg.t_begin == 0 ? 1 : 0)) * kRowTile + sh.row[warp];
        const float f = !whole ? 1.f : l == 0.f ? 0.f : 1.f / l;
        const float4 o = *reinterpret_cast<const float4*>(&sh.o[warp][lane * 4]);
        __nv_bfloat16* dst = whole ? out_all + (size_t)sh.sg.layer * span.out_stride + (((size_t)sh.sg.b * lq + jj) * n_q_heads + sh.sg.kvh * group + g) * kD
                                   : reinterpret_cast<__nv_bfloat16*>(ws.part_o) + slot * kD;
        *reinterpret_cast<uint2*>(dst + lane * 4) = make_uint2(pack_bf16(o.x * f, o.y * f), pack_bf16(o.z * f, o.w * f));
        if (lane == 0 && whole) {
            const size_t at = (size_t)sh.sg.lb * rows_total + (size_t)sh.sg.kvh * group * lq + row;
            const float row_lse2 = top + log2f(ld);
            ws.row_lse2[at] = row_lse2 == row_lse2 ? row_lse2 : __int_as_float(0x7fffffff);
            if (lse) lse[at] = (top + log2f(l)) * kLn2;
        } else if (lane == 0) {
            ws.part_m[slot] = l == 0.f ? -INFINITY : top > -INFINITY ? top : 0.f;   // (a sum that is not a number has to be seen)
            ws.part_l[slot] = l;
            if (ws.part_ld) ws.part_ld[slot] = ld;
        }
    }
    __syncthreads();                                                // the shared memory may be used again
}

// The rows of a share that left the range of their reference (their sums are not numbers), segment by segment, in eights of
// neighbours.  Only rows whose logits lie more than 2^80 above the first 16 of the segment come here, and keys that are not
// finite.  A segment's reference is its own, so a row that left it in one share is computed over that share's keys and joins the
// other parts like any other.  In the merge kernel, over all keys of the row (one block of eight warps had to walk them), the path
// cost every merge 0.3 to 0.5 us although nobody took it: one layer of 20 documents, 32/32 heads 48.3 -> 46.6 us, 28 one-layer
// calls over 50 documents, 12/2 heads 574 -> 559.  Calls with such rows: four layers of 50 documents of 160 tokens, 12/2 heads, 44 us
// without, one row a layer 166 -> 79, every row 759 -> 398; one layer of 2 x 60 documents of 180, 32/32 heads, 93 us, 265 -> 166 and
// 1109 -> 646; of 4 x 50 of 160, 28/4 heads, 75 us, 202 -> 130 and 687 -> 720 (few tiles per share leave warps idle).
template <int LAYOUT>
__device__ __forceinline__ void marked_from_scratch(const Params& p, RowScratch& sh, const Line& line) {
    const int group = p.n_q_heads / p.n_kv_heads;
    if (threadIdx.x == 0) sh.x = line.cut(blockIdx.x);
#pragma unroll 1
    while (true) {
        __syncthreads();                                            // the segment before has been read
        if (sh.x >= line.cut(blockIdx.x + 1)) break;
        if (threadIdx.x == 0) sh.sg = segment_at(p.bv, p.pv, p.ws, line, group, sh.x, line.cut(blockIdx.x + 1));
        __syncthreads();
        if (threadIdx.x < kRowTile) {
            const int rows = group * p.bv.q_len;
            float l = 0.f;
            if ((int)threadIdx.x < sh.sg.rows_here)
                l = sh.sg.t_end - sh.sg.t_begin == sh.sg.n_unit
                        ? p.ws.row_lse2[(size_t)sh.sg.lb * p.n_q_heads * p.bv.q_len + (size_t)sh.sg.kvh * rows + sh.sg.row0 + threadIdx.x]
                        : p.ws.part_l[((size_t)2 * blockIdx.x + (sh.sg.t_begin == 0 ? 1 : 0)) * kRowTile + threadIdx.x];
            const unsigned set = __ballot_sync(0xffffffffu, l != l);
            if ((threadIdx.x & 31) == 0) sh.todo[threadIdx.x >> 5] = set;
        }
        if (threadIdx.x == 0) sh.x += sh.sg.t_end - sh.sg.t_begin;
#pragma unroll 1
        while (true) {
            __syncthreads();
            const int w = sh.todo[0] ? 0 : sh.todo[1] ? 1 : sh.todo[2] ? 2 : 3;
            const unsigned set = sh.todo[w];
            if (set == 0) break;
            __syncthreads();
            if (threadIdx.x == 0) sh.todo[w] = set ^ rows::next_group(set);
            rows_from_scratch<LAYOUT>(p, sh, w * 32, set);
        }
    }
}

template <int LAYOUT>
__global__ void __launch_bounds__(kThreads, 1)
attn_tc_kernel(const __grid_constant__ StoreMaps maps, const __grid_constant__ Params p) {
    CF_PARAMS;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t k_base = smem_u32(smem), v_base = k_base + kKStages * kKvBytes;
    Shared& sh = *reinterpret_cast<Shared*>(smem + (kKStages + kVStages) * kKvBytes);
    Barriers& bars = sh.bars;
    volatile int* abort_flag = &bars.abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int group = n_q_heads / n_kv_heads, lq = bv.q_len, rows = group * lq, rows_total = n_q_heads * lq;

    if (warp == kMmaWarp) {
        if (lane == 0) {
            auto init = [](unsigned long long* bar, int n, int count) {
                for (int i = 0; i < n; ++i) mbar_init(smem_u32(bar + i), count);
            };
            init(bars.k_full, kKStages, 1);
            init(bars.k_ready, kKStages, kRotateWarps);
            init(bars.k_empty, kKStages, 1);
            init(bars.v_empty, kVStages, 1);
            init(bars.s_full, 6, 1);
            init(bars.pv_ready, 6, 5);                              // one arrival per warp, one with the copy of V
            init(bars.segment, kSegRing, 1);
            init(&bars.q_ready, 1, 8);
            init(&bars.q_free, 1, 1);
            init(&bars.o_done, 1, 1);
            init(&bars.o_free, 1, 8);
            init(bars.ref_full, 2, 4);
            init(bars.sum_full, 2, 8);
            bars.abort_flag = 0;
            bars.marked = 0;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&bars.tmem_base)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (warp == kLoadWarp && lane < 2 * kBoxes)
        asm volatile("prefetch.tensormap [%0];" ::"l"(lane < kBoxes ? &maps.k[lane] : &maps.v[lane - kBoxes]) : "memory");
    chain_next();
    chain_wait();
    if (warp == 0) {
        scan_requests(bv, pv, p.n_prefix + p.n_self, sh.requests);
        __syncwarp();
        if (lane == 0) {
            const Line l = make_line(bv, ws, sh.requests, n_kv_heads, p.row_tiles, p.n_prefix, p.n_self, (int)gridDim.x);
            sh.line = l;
            const int begin = (int)blockIdx.x < l.n_shares ? l.cut(blockIdx.x) : 0, end = (int)blockIdx.x < l.n_shares ? l.cut(blockIdx.x + 1) : 0;
            if (begin < end) sh.segments[0] = segment_at(bv, pv, ws, l, group, begin, end);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const Line& line = sh.line;
    const uint32_t tmem = bars.tmem_base;
    const int x_begin = (int)blockIdx.x < line.n_shares ? line.cut(blockIdx.x) : 0, x_end = (int)blockIdx.x < line.n_shares ? line.cut(blockIdx.x + 1) : 0;
    const int n_items = x_end - x_begin;                            // 0: this CTA has no share, its roles find nothing to do

    if (n_items == 0) {
    } else if (warp == kLoadWarp) {
        // ------------------------------------------------------------------ key and value loads, tile descriptions
        if (lane == 0) {
            constexpr int kAhead = 3;                               // keys run ahead of values: S(n + 3) is issued beside PV(n)
            Segment sg = sh.segments[0];
            int t = sg.t_begin, x = x_begin, row0, len, index, doc = 0, segments = 1;
            auto fetch = [&]() {                                    // tile t of the segment
                if (t < sg.n_doc) {
                    index = sg.tile0 + t;
                    row0 = __ldg(pv.tile_row0 + index);
                    len = __ldg(pv.tile_len + index);
                    doc = __ldg(pv.tile_doc + index);
                } else if (t < sg.n_doc + line.n_prefix) {
                    index = kKindPrefix;
                    row0 = (t - sg.n_doc) * kTile;
                    len = min(kTile, src.prefix_len - row0);
                } else {
                    const int n = t - sg.n_doc - line.n_prefix;
                    index = kKindSelf - n;
                    row0 = sg.b * lq + n * kTile;
                    len = min(kTile, lq - n * kTile);
                }
            };
            fetch();
            ShareHead head = {};
            int ks = 0, kp = 1, vs = 0, vp = 1, ps = 0;             // the first lap's waits pass: the phase before a fresh barrier's first
            for (int n = 0; n < n_items + kAhead; ++n) {
                if (n < n_items) {
                    const int4 m = make_int4(len | (t == sg.t_begin ? kFirstOfSegment : 0) | (t == sg.t_end - 1 ? kLastOfSegment : 0), index, row0,
                                             sg.kvh | (sg.layer << 20));
                    const float2* trig = pv.trig + (size_t)doc * (kD / 2);
                    ++x;
                    if (++t == sg.t_end && x < x_end) {
                        sg = segment_at(bv, pv, ws, line, group, x, x_end);
                        t = sg.t_begin;
                        sh.segments[segments & (kSegRing - 1)] = sg;
                        mbar_arrive(smem_u32(&bars.segment[segments & (kSegRing - 1)]));
                        ++segments;
                    }
                    if (x < x_end) fetch();                         // the next tile's description travels under this one's wait
                    if (!mbar_wait(smem_u32(&bars.k_empty[ks]), kp, abort_flag)) break;
                    sh.meta[n & (kMetaRing - 1)] = m;
                    const uint32_t bar = smem_u32(&bars.k_full[ks]), dst = k_base + ks * kKvBytes;
                    const int boxes = m.y >= 0 ? ((m.x & 0xff) + 15) >> 4 : kBoxes;
                    const CUtensorMap* map = m.y >= 0 ? &maps.k[boxes - 1] : m.y == kKindPrefix ? &maps.kp : &maps.ks;
                    mbar_expect_tx(bar, (boxes << 12) + (m.y >= 0 ? kTrigBytes : 0));
                    if (m.y >= 0) bulk_load(smem_u32(sh.trig[ks]), trig, kTrigBytes, bar);
                    tma_load_4d(dst, map, 0, m.w & 0xfffff, m.z, m.w >> 20, bar);
                    tma_load_4d(dst + kKvHalf, map, 64, m.w & 0xfffff, m.z, m.w >> 20, bar);
                    if (++ks == kKStages) {
                        ks = 0;
                        kp ^= 1;
                    }
                }
                if (n >= kAhead) {
                    if (!mbar_wait(smem_u32(&bars.v_empty[vs]), vp, abort_flag)) break;
                    const int4 m = sh.meta[(n - kAhead) & (kMetaRing - 1)];
                    const uint32_t bar = smem_u32(&bars.pv_ready[ps]), dst = v_base + vs * kKvBytes;
                    const int boxes = m.y >= 0 ? ((m.x & 0xff) + 15) >> 4 : kBoxes;
                    const CUtensorMap* map = m.y >= 0 ? &maps.v[boxes - 1] : m.y == kKindPrefix ? &maps.vp : &maps.vs;
                    mbar_expect_tx(bar, boxes << 12);
                    tma_load_4d(dst, map, 0, m.w & 0xfffff, m.z, m.w >> 20, bar);
                    tma_load_4d(dst + kKvHalf, map, 64, m.w & 0xfffff, m.z, m.w >> 20, bar);
                    if (++ps == 6) ps = 0;
                    if (++vs == kVStages) {
                        vs = 0;
                        vp ^= 1;
                    }
                }
            }
            // sg is the share's last segment
            if (sg.t_begin == 0 && sg.t_end < sg.n_unit) {
                head.n_parts = line.share_of(x_end - sg.t_end + sg.n_unit - 1) - (int)blockIdx.x + 1;
                head.lb = sg.lb;
                head.layer = sg.layer;
                head.b = sg.b;
                head.row_first = sg.kvh * rows + sg.row0;
                head.rows_here = sg.rows_here;
            }
            sh.head = head;
        }
    } else if (warp == kMmaWarp) {
        // ------------------------------------------------------------------ MMA issue: the warp walks, one lane issues
        const bool lead = elect_one();
        const uint32_t idesc_o = instr_desc(kD, true), idesc_s0 = instr_desc(0, false);
        const uint64_t bk_desc = smem_desc(k_base, 16, 1024), bv_desc = smem_desc(v_base, kKvHalf, 1024);
        const uint32_t bar_k_ready = smem_u32(bars.k_ready), bar_k_empty = smem_u32(bars.k_empty), bar_v_empty = smem_u32(bars.v_empty);
        const uint32_t bar_s_full = smem_u32(bars.s_full), bar_pv_ready = smem_u32(bars.pv_ready);
        // One rolled loop (unrolled by the rings' period of six it was some instructions per tile shorter, and every lap's first
        // pass through it cost 2 to 3 thousand cycles per tile of instruction fetches).
        struct Ring {
            int it, j, parity;                                      // tile, tile mod 6, parity of its lap
        } s = {0, 0, 0}, v = {0, 0, 0};
        auto next = [](Ring& r) {
            ++r.it;
            if (++r.j == 6) {
                r.j = 0;
                r.parity ^= 1;
            }
        };
        int segments_s = 0, segments = 0;                           // segments begun by QK^T, finished by PV
        bool ok = true;
        while (v.it < n_items && ok) {
            // QK^T runs up to three tiles ahead; into the next segment only once its query tile is there
            bool do_s = s.it < n_items && s.it < v.it + kSBuffers;
            int m = 0;
            if (do_s) {
                ok = warp_wait(bar_k_ready + s.j * 8, s.parity, abort_flag);
                if (!ok) break;
                m = sh.meta[s.it & (kMetaRing - 1)].x;
                if (m & kFirstOfSegment) {
                    const uint32_t bar = smem_u32(&bars.q_ready);
                    if (s.it == v.it) ok = warp_wait(bar, segments_s & 1, abort_flag);
                    else do_s = __all_sync(0xffffffffu, mbar_try_wait(bar, segments_s & 1));
                    if (!ok) break;
                    if (do_s) ++segments_s;
                }
            }
            if (do_s) {
                tc_fence_after();
                const uint32_t idesc = idesc_s0 | ((uint32_t)(((m & 0xff) + 15) >> 4) << 18);
                const uint64_t b0 = bk_desc + (uint64_t)(s.j * (kKvBytes >> 4));
                const uint32_t s_tmem = tmem + kColS + (s.j >= 3 ? s.j - 3 : s.j) * kTile, q_tmem = tmem + kColQ;
                if (lead) {
                    umma_ts_lit<false>(s_tmem, q_tmem, b0, idesc);
#pragma unroll
                    for (int kk = 1; kk < 8; ++kk)                  // 16 dims per instruction
                        umma_ts_lit<true>(s_tmem, q_tmem + kk * 8, b0 + (uint64_t)(((kk >> 2) * kKvHalf + (kk & 3) * 32) >> 4), idesc);
                    umma_commit(bar_s_full + s.j * 8);
                    umma_commit(bar_k_empty + s.j * 8);
                    if (m & kLastOfSegment) umma_commit(smem_u32(&bars.q_free));
                }
                __syncwarp();
                next(s);
                if (s.it < v.it + kSBuffers && s.it < n_items) continue;
            }
            m = sh.meta[v.it & (kMetaRing - 1)].x;
            ok = warp_wait(bar_pv_ready + v.j * 8, v.parity, abort_flag);
            if (ok && (m & kFirstOfSegment) && segments > 0) ok = warp_wait(smem_u32(&bars.o_free), (segments - 1) & 1, abort_flag);
            if (!ok) break;
            tc_fence_after();
            const int steps = ((m & 0xff) + 15) >> 4;               // 16 keys = 8 packed columns per instruction
            const int buffer = v.j >= 3 ? v.j - 3 : v.j;            // both of the S buffers and of the value stages
            const uint64_t b0 = bv_desc + (uint64_t)(buffer * (kKvBytes >> 4));
            const uint32_t p_tmem = tmem + kColS + buffer * kTile, o_tmem = tmem + kColO;
            if (lead) {
                umma_ts(o_tmem, p_tmem, b0, idesc_o, (m & kFirstOfSegment) ? 0u : 1u);
                for (int kk = 1; kk < steps; ++kk) umma_ts_lit<true>(o_tmem, p_tmem + kk * 8, b0 + (uint64_t)(kk * 128), idesc_o);
                umma_commit(bar_v_empty + buffer * 8);
                if (m & kLastOfSegment) umma_commit(smem_u32(&bars.o_done));
            }
            __syncwarp();
            if (m & kLastOfSegment) ++segments;
            next(v);
        }
    } else if (warp >= 8) {
        // ------------------------------------------------------------------ key rotation (Eq. 5)
        const int rw = warp == 8 ? 0 : warp < kMmaWarp ? warp - 9 : warp - 10, rt = rw * 32 + lane;   // 0 .. 191
        const int chunk = rt & 7, rsub = rt >> 3;                   // 16-byte chunk of each half row; first row
        int stage = 0, phase = 0;
        for (int it = 0; it < n_items; ++it) {
            if (!warp_wait(smem_u32(&bars.k_full[stage]), phase, abort_flag)) break;
            const int2 meta = *reinterpret_cast<const int2*>(&sh.meta[it & (kMetaRing - 1)]);
            if (meta.y >= 0) {                                      // a document's tile: its table came with the keys
                const int len = meta.x & 0xff;
                uint64_t c2[4], s2[4], n2[4];                       // cosines, sines and their negatives as pairs for the packed arithmetic
                const float4* trig = reinterpret_cast<const float4*>(sh.trig[stage]);
#pragma unroll
                for (int e = 0; e < 4; ++e) {                       // half layout: slices chunk*8 .. +7; interleaved: chunk*4 .. +3 of either half
                    const float4 cs = trig[LAYOUT == CF_ROPE_HALF ? chunk * 4 + e : (e >> 1) * 16 + chunk * 2 + (e & 1)];
                    c2[e] = pack_f2(cs.x, cs.z);
                    s2[e] = pack_f2(cs.y, cs.w);
                    n2[e] = pack_f2(-cs.y, -cs.w);
                }
                // rows 24 apart keep their swizzle phase: one pointer walks
                unsigned char* at = smem + (size_t)stage * kKvBytes + swz(rsub, chunk);
#pragma unroll 2
                for (int r = rsub; r < len; r += kRotateWarps * 4, at += kRotateWarps * 4 * 128) {
                    uint4* pa = reinterpret_cast<uint4*>(at);
                    uint4* pb = reinterpret_cast<uint4*>(at + kKvHalf);
                    const uint4 va = *pa, vb = *pb;
                    uint32_t wa[4] = {va.x, va.y, va.z, va.w}, wb[4] = {vb.x, vb.y, vb.z, vb.w};
                    if (LAYOUT == CF_ROPE_HALF) {
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const uint64_t fa = pack_f2(__uint_as_float(wa[e] << 16), __uint_as_float(wa[e] & 0xffff0000u));
                            const uint64_t fb = pack_f2(__uint_as_float(wb[e] << 16), __uint_as_float(wb[e] & 0xffff0000u));
                            float y0, y1;
                            unpack_f2(fma_f2(fa, c2[e], mul_f2(fb, n2[e])), y0, y1);
                            wa[e] = pack_bf16(y0, y1);
                            unpack_f2(fma_f2(fa, s2[e], mul_f2(fb, c2[e])), y0, y1);
                            wb[e] = pack_bf16(y0, y1);
                        }
                    } else {
#pragma unroll
                        for (int e = 0; e < 4; ++e) {               // the two elements of a word are a slice; words in pairs
                            uint32_t& w0 = e < 2 ? wa[2 * e] : wb[2 * e - 4];
                            uint32_t& w1 = e < 2 ? wa[2 * e + 1] : wb[2 * e - 3];
                            const uint64_t fa = pack_f2(__uint_as_float(w0 << 16), __uint_as_float(w1 << 16));
                            const uint64_t fb = pack_f2(__uint_as_float(w0 & 0xffff0000u), __uint_as_float(w1 & 0xffff0000u));
                            float a0, a1, b0, b1;
                            unpack_f2(fma_f2(fa, c2[e], mul_f2(fb, n2[e])), a0, a1);
                            unpack_f2(fma_f2(fa, s2[e], mul_f2(fb, c2[e])), b0, b1);
                            w0 = pack_bf16(a0, b0);
                            w1 = pack_bf16(a1, b1);
                        }
                    }
                    *pa = make_uint4(wa[0], wa[1], wa[2], wa[3]);
                    *pb = make_uint4(wb[0], wb[1], wb[2], wb[3]);
                }
                fence_proxy_async();
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bars.k_ready[stage]));
            if (++stage == kKStages) {
                stage = 0;
                phase ^= 1;
            }
        }
    } else {
        // ------------------------------------------------------------------ softmax, one row per thread
        const int w = warp >> 2, r = tid & 127;                     // warpgroup; row of the tile = TMEM lane
        const uint32_t lane_tmem = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        const uint64_t scale2 = pack_f2(src.scale_log2, src.scale_log2);
        const uint32_t bar_s_full = smem_u32(bars.s_full), bar_pv_ready = smem_u32(bars.pv_ready);
        int k = w, phase = 0;                                       // this warpgroup's next tile, mod 6, and its parity
        int it0 = 0;                                                // tiles before the current segment
        float ref = 0.f, l_run = 0.f, l_docs = 0.f;
        const bool wide_out = ((reinterpret_cast<uintptr_t>(out_all) | (uintptr_t)(span.out_stride * 2)) & 31) == 0;   // rows start at 32-byte addresses
        bool ok = true;
        for (int seg = 0; ok; ++seg) {
            const bool more = it0 < n_items;
            const int slot = seg & (kSegRing - 1);
            if (more && seg > 0) {
                ok = warp_wait(smem_u32(&bars.segment[slot]), (seg / kSegRing) & 1 ^ (slot == 0 ? 1 : 0), abort_flag);
                if (!ok) break;
            }
            const Segment& sg = sh.segments[slot];
            if (more) {
                // the query tile of the segment goes into tensor memory, half of every row by each warpgroup (before the
                // epilogue of the last segment)
                const bool active = (warp & 3) * 32 < sg.rows_here;
                const int row = sg.row0 + min(r, sg.rows_here - 1), g = row / lq, j = row - g * lq;
                const uint4* q = reinterpret_cast<const uint4*>(src.q + (size_t)sg.layer * span.q_stride + (((size_t)sg.b * lq + j) * n_q_heads + sg.kvh * group + g) * kD) + w * 8;
                uint32_t qw[32];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const uint4 v = __ldg(q + i);
                    qw[4 * i] = v.x;
                    qw[4 * i + 1] = v.y;
                    qw[4 * i + 2] = v.z;
                    qw[4 * i + 3] = v.w;
                }
                if (seg > 0) ok = warp_wait(smem_u32(&bars.q_free), (seg - 1) & 1, abort_flag);   // read by its last QK^T
                if (!ok) break;
                if (active) {
                    tc_fence_after();
                    tmem_st16_from<0>(lane_tmem + kColQ + w * 32, qw);
                    tmem_st16_from<16>(lane_tmem + kColQ + w * 32 + 16, qw);
                    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                    tc_fence_before();
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bars.q_ready));
            }
            if (seg > 0) {
                // ---- end of a segment: the two sums meet, each warpgroup takes half of the columns of O
                const int par = (seg - 1) & 1;
                sh.sum[par][w][r] = l_run;
                sh.docs[par][w][r] = l_docs;
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bars.sum_full[par]));
                ok = warp_wait(smem_u32(&bars.sum_full[par]), ((seg - 1) >> 1) & 1, abort_flag) && warp_wait(smem_u32(&bars.o_done), par, abort_flag);
                if (!ok) break;
                tc_fence_after();
                const Segment& done = sh.segments[(seg - 1) & (kSegRing - 1)];
                const bool whole = done.t_end - done.t_begin == done.n_unit;
                const int row = done.row0 + r;
                const float l_all = sh.sum[par][0][r] + sh.sum[par][1][r], d_all = sh.docs[par][0][r] + sh.docs[par][1][r];
                const bool row_valid = r < done.rows_here, marked = l_all != l_all;
                const size_t at = (size_t)done.lb * rows_total + (size_t)done.kvh * rows + row;
                if ((warp & 3) * 32 < done.rows_here) {
                    const int g = row / lq, j = row - g * lq;
                    const size_t slot = ((size_t)2 * blockIdx.x + (done.t_begin == 0 ? 1 : 0)) * kRowTile + r;
                    const float f = whole ? (l_all > 0.f ? 1.f / l_all : 0.f) : 1.f;
                    __nv_bfloat16* dst = (whole ? out_all + (size_t)done.layer * span.out_stride + (((size_t)done.b * lq + j) * n_q_heads + done.kvh * group + g) * kD
                                                : reinterpret_cast<__nv_bfloat16*>(ws.part_o) + slot * kD) + w * 64;
#pragma unroll 1
                    for (int c = 0; c < 2; ++c) {
                        uint32_t o[32];
                        tmem_ld32(lane_tmem + kColO + w * 64 + c * 32, o);
                        if (row_valid) {
#pragma unroll
                            for (int i = 0; i < 2; ++i) {           // whole 32-byte sectors: rows are 256 bytes apart
                                uint32_t y[8];
#pragma unroll
                                for (int e = 0; e < 8; ++e) y[e] = pack_bf16(__uint_as_float(o[16 * i + 2 * e]) * f, __uint_as_float(o[16 * i + 2 * e + 1]) * f);
                                if (wide_out) {
                                    store32(dst + c * 32 + i * 16, y);
                                } else {
                                    *reinterpret_cast<uint4*>(dst + c * 32 + i * 16) = make_uint4(y[0], y[1], y[2], y[3]);
                                    *reinterpret_cast<uint4*>(dst + c * 32 + i * 16 + 8) = make_uint4(y[4], y[5], y[6], y[7]);
                                }
                            }
                        }
                    }
                    if (w == 0 && row_valid) {
                        if (!whole) {
                            ws.part_m[slot] = l_all == 0.f ? -INFINITY : ref;   // a row may see none of the segment's keys
                            ws.part_l[slot] = l_all;
                            if (ws.part_ld) ws.part_ld[slot] = d_all;   // what the document scores are measured against
                            if (done.t_begin == 0)            // (the share's last segment)
                                reinterpret_cast<uint32_t*>(ws.row_lse2)[at] =
                                    parts_code(blockIdx.x, line.share_of(x_end - done.t_end + done.n_unit - 1) - (int)blockIdx.x + 1);
                        } else {
                            ws.row_lse2[at] = marked ? __int_as_float(0x7fffffff) : ref + log2f(d_all);
                            if (lse) lse[at] = (ref + log2f(l_all)) * kLn2;
                        }
                        if (marked) bars.marked = 1;
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bars.o_free));
            }
            if (!more) break;
            // ---- the tiles of the segment
            const int n = sg.t_end - sg.t_begin, par = seg & 1;
            const bool active = (warp & 3) * 32 < sg.rows_here, row_valid = r < sg.rows_here;
            const int q_index = (sg.row0 + r) % lq;                 // position of this row's token in the query
            float* tile_lse2 = ws.tile_lse2 + (size_t)sg.layer * ws.max_tiles * rows_total + (size_t)sg.kvh * rows + sg.row0 + r;
            const bool leads = (it0 & 1) == w;                      // this warpgroup has the segment's first tile
            bool have_ref = false, seen_extra = false;
            l_run = l_docs = 0.f;
            for (int i = leads ? 0 : 1; i < n; i += 2) {
                ok = warp_wait(bar_s_full + k * 8, phase, abort_flag);
                if (!ok) break;
                tc_fence_after();
                const int4 meta = sh.meta[(it0 + i) & (kMetaRing - 1)];
                const int len = meta.x & 0xff, n_chunks = (len + 15) >> 4;
                // keys this row may see: a whole tile of a document or of the prefix, the query tokens up to its own (causal
                // mask, footnote to Eq. 1)
                const int vis = meta.y <= kKindSelf ? min(len, q_index + 1 - (kKindSelf - meta.y) * kTile) : len;
                const uint32_t s_addr = lane_tmem + kColS + (k >= 3 ? k - 3 : k) * kTile;
                uint32_t va[16], vb[16];
                if (active) {
                    tmem_ld16_async(s_addr, va);
                    tmem_ld16_wait(va);
                }
                if (i == 0) {                                       // the reference of the segment, from its first 16 keys
                    float m = -INFINITY;
#pragma unroll
                    for (int e = 0; e < 16; ++e) m = fmaxf(m, e < vis ? __uint_as_float(va[e]) : -INFINITY);
                    sh.ref[par][r] = m > -INFINITY ? m * src.scale_log2 : 0.f;   // a row that sees none of them sees none of the tile
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&bars.ref_full[par]));
                }
                if (!have_ref) {
                    ok = warp_wait(smem_u32(&bars.ref_full[par]), (seg >> 1) & 1, abort_flag);
                    if (!ok) break;
                    ref = sh.ref[par][r];
                    have_ref = true;
                }
                if (meta.y < 0 && !seen_extra) {                    // from here on the keys are not the documents'
                    l_docs = l_run;
                    seen_extra = true;
                }
                if (active) {
                    // single pass in chunks of 16 keys: P chunk c goes over the S columns 8c .. 8c + 7, which are in registers by then
                    const uint64_t neg_ref2 = pack_f2(-ref, -ref);
                    uint64_t sum2 = 0;
                    auto finish = [&](uint32_t (&v)[16], int c) {
                        if (vis - c * 16 < 16) {                    // the ragged end of a tile, the causal mask
#pragma unroll
                            for (int e = 0; e < 16; ++e) v[e] = e < vis - c * 16 ? v[e] : 0xff800000u;
                        }
                        chunk16_exp(v, scale2, neg_ref2, sum2);
                        tmem_st8_async(s_addr + c * 8, v);
                    };
#pragma unroll 1
                    for (int c = 0;;) {
                        if (c + 1 < n_chunks) tmem_ld16_async(s_addr + (c + 1) * 16, vb);
                        finish(va, c);
                        if (++c == n_chunks) break;
                        tmem_ld16_wait(vb);
                        if (c + 1 < n_chunks) tmem_ld16_async(s_addr + (c + 1) * 16, va);
                        finish(vb, c);
                        if (++c == n_chunks) break;
                        tmem_ld16_wait(va);
                    }
                    float tile_sum, odd;
                    unpack_f2(sum2, tile_sum, odd);
                    tile_sum += odd;
                    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_pv_ready + k * 8);
                    if (!(tile_sum < kSumLimit)) tile_sum = __int_as_float(0x7fffffff);     // out of range: the row is marked
                    l_run += tile_sum;
                    if (meta.y >= 0 && row_valid) tile_lse2[(size_t)meta.y * rows_total] = ref + __log2f(tile_sum);
                } else if (lane == 0) {
                    mbar_arrive(bar_pv_ready + k * 8);
                }
                k += 2;
                if (k >= 6) {
                    k -= 6;
                    phase ^= 1;
                }
            }
            if (ok && !have_ref) ok = warp_wait(smem_u32(&bars.ref_full[par]), (seg >> 1) & 1, abort_flag);   // every phase is waited for
            if (!have_ref && ok) ref = sh.ref[par][r];
            if (!seen_extra) l_docs = l_run;
            it0 += n;
        }
    }

    // ---------------------------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    if (tid == 0) {
        ShareHead head = {};
        if (n_items > 0) head = sh.head;
        reinterpret_cast<ShareHead*>(ws.marks)[blockIdx.x] = head;
    }
    // every copy has landed and every MMA has read its operands: the rings are free
    if (bars.marked && !bars.abort_flag) marked_from_scratch<LAYOUT>(p, *reinterpret_cast<RowScratch*>(smem), line);
    if (bars.abort_flag) {
        // a wait expired: let the copies in flight land before the shared memory is given back
        if (tid == 0) {
            const long long t0 = clock64();
            while (clock64() - t0 < kWaitLimitCycles / 64) {}
            atomicCAS(pv.status, 0, CF_ERR_TIMEOUT);
        }
        __syncthreads();
    }
    if (warp == kMmaWarp) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
}

constexpr int kMergeThreads = 256;

// Units that lie in several shares: the parts of a row are merged in the order of the line by eight lanes.  A chain of two memory
// latencies: where the parts are was left by the CTA the unit begins in, and four parts of a row are loaded together.
// ROWS = 32: a block has a slice of the unit that begins in one share and goes on behind it.  ROWS = 8, for few units of many parts: a
// block has a slice of one unit and reads from its first row's word how it was cut (blocks that looked at four shares each, of
// which few begin a unit: 28 calls over 50 documents, 12/2 heads, 553 us, this way 530); the parts of a row are cut into four
// runs, walked side by side and joined in order through shared memory.  Either also sees to the (empty) results of requests that
// have nothing to attend.
template <int ROWS>
__global__ void __launch_bounds__(kMergeThreads, 2)
attn_tc_merge_kernel(const __grid_constant__ Params p) {
    CF_PARAMS;
    constexpr bool kByUnit = ROWS < 32;
    constexpr int kRuns = 32 / ROWS, kRunThreads = kMergeThreads / kRuns;
    __shared__ float s_run[kRuns > 1 ? kRuns - 1 : 1][19][kRuns > 1 ? kRunThreads : 1];   // m, l, ld and 16 dims per thread
    const int lq = bv.q_len, rows_total = n_q_heads * lq, rows = n_q_heads / n_kv_heads * lq, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int slices = (int)p.merge_slices.d;
    const int at = p.merge_slices.quotient(blockIdx.x), slice = (int)blockIdx.x - at * slices;          // unit or share; slice of its rows
    ShareHead head;
    int share = at;
    if (kByUnit) {
        const int u = p.tiles_of_rows.quotient(at), row_tile = at - u * p.row_tiles, kvh = p.kv_heads.remainder(u);
        head.lb = p.kv_heads.quotient(u);
        head.layer = p.requests.quotient(head.lb);
        head.b = head.lb - head.layer * bv.n_requests;
        head.row_first = kvh * rows + row_tile * ws.rg_rows;
        head.rows_here = min(ws.rg_rows, rows - row_tile * ws.rg_rows);
    }
    chain_next();
    chain_wait();
    if (kByUnit) {
        if (slice * ROWS >= head.rows_here) return;
        const size_t first = (size_t)head.lb * rows_total + head.row_first + slice * ROWS;
        const uint32_t word = reinterpret_cast<const uint32_t*>(ws.row_lse2)[first];
        if (p.n_prefix + p.n_self == 0 && pv.n_tiles[head.b] == 0) {
            const int n = min(ROWS, head.rows_here - slice * ROWS);
            for (int i = threadIdx.x; i < n * (kD / 8); i += kMergeThreads) {
                const int rg = head.row_first + slice * ROWS + i / (kD / 8), h = rg / lq, j = rg - h * lq;
                reinterpret_cast<uint4*>(out_all + (size_t)head.layer * span.out_stride + (((size_t)head.b * lq + j) * n_q_heads + h) * kD)[i % (kD / 8)] =
                    make_uint4(0u, 0u, 0u, 0u);
            }
            __syncthreads();                                        // every thread has its word
            if (threadIdx.x < n) {
                ws.row_lse2[first + threadIdx.x] = -INFINITY;
                if (lse) lse[first + threadIdx.x] = -INFINITY;
            }
            return;
        }
        if (!is_parts_code(word)) return;                           // finished by its one share
        __syncthreads();                                            // every thread has its word: a row's is written below
        head.n_parts = part_count(word);
        share = first_share(word);
    } else {
        const int4* from = reinterpret_cast<const int4*>(reinterpret_cast<const ShareHead*>(ws.marks) + share);
        const int4 lo = from[0], hi = from[1];
        head = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y};
        if (share == p.max_shares - 1 && p.n_prefix + p.n_self == 0)
            for (int b = slice; b < bv.n_requests; b += slices)
                if (pv.n_tiles[b] == 0)
                    for (int layer = 0; layer < ws.n_layers; ++layer) {
                        uint4* dst = reinterpret_cast<uint4*>(out_all + (size_t)layer * span.out_stride + (size_t)b * rows_total * kD);
                        for (int i = threadIdx.x; i < rows_total * (kD / 8); i += kMergeThreads) dst[i] = make_uint4(0u, 0u, 0u, 0u);
                        const size_t to = ((size_t)layer * bv.n_requests + b) * rows_total;
                        for (int i = threadIdx.x; i < rows_total; i += kMergeThreads) {
                            ws.row_lse2[to + i] = -INFINITY;
                            if (lse) lse[to + i] = -INFINITY;
                        }
                    }
        if (head.n_parts == 0 || slice * ROWS >= head.rows_here) return;
    }
    {
        const int n_parts = head.n_parts;
        const int run = warp / (8 / kRuns), part_end = n_parts * (run + 1) / kRuns;
        const int r = slice * ROWS + (warp - run * (8 / kRuns)) * 4 + (lane >> 3), e0 = (lane & 7) * 16;   // row of the unit; this lane's dims
        const bool valid = run == 0 && r < head.rows_here;
        float acc[16], m = -INFINITY, l = 0.f, ld = 0.f;
#pragma unroll
        for (int e = 0; e < 16; ++e) acc[e] = 0.f;
        // part i: the share's slot for what goes on behind it (i = 0), the others' for what began before them
        const size_t slot0 = ((size_t)2 * share + 1) * kRowTile + min(r, head.rows_here - 1), slot1 = slot0 + kRowTile;
        auto slot_of = [&](int i) { return i == 0 ? slot0 : slot1 + (size_t)(i - 1) * 2 * kRowTile; };
        const __nv_bfloat16* part_o = reinterpret_cast<const __nv_bfloat16*>(ws.part_o) + e0;
        for (int i0 = n_parts * run / kRuns; i0 < part_end; i0 += 4) {
            float mp[4], lp[4], dp[4];
            uint4 o[4][2];
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const size_t slot = slot_of(min(i0 + x, part_end - 1));
                mp[x] = i0 + x < part_end ? ws.part_m[slot] : -INFINITY;
                lp[x] = ws.part_l[slot];
                dp[x] = ws.part_ld ? ws.part_ld[slot] : lp[x];
                o[x][0] = *reinterpret_cast<const uint4*>(part_o + slot * kD);
                o[x][1] = *reinterpret_cast<const uint4*>(part_o + slot * kD + 8);
            }
            const float m_new = fmaxf(fmaxf(m, fmaxf(mp[0], mp[1])), fmaxf(mp[2], mp[3]));
            const float keep = m > -INFINITY ? fast_exp2(m - m_new) : 0.f;
            m = m_new;
            l *= keep;
            ld *= keep;
#pragma unroll
            for (int e = 0; e < 16; ++e) acc[e] *= keep;
#pragma unroll
            for (int x = 0; x < 4; ++x)
                if (mp[x] > -INFINITY) {
                    const float w = fast_exp2(mp[x] - m_new);
                    l = fmaf(lp[x], w, l);
                    ld = fmaf(dp[x], w, ld);
                    const uint32_t pairs[8] = {o[x][0].x, o[x][0].y, o[x][0].z, o[x][0].w, o[x][1].x, o[x][1].y, o[x][1].z, o[x][1].w};
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        acc[2 * e] = fmaf(__uint_as_float(pairs[e] << 16), w, acc[2 * e]);
                        acc[2 * e + 1] = fmaf(__uint_as_float(pairs[e] & 0xffff0000u), w, acc[2 * e + 1]);
                    }
                }
        }
        if (kRuns > 1) {
            if (run > 0) {
                float* mine = &s_run[run - 1][0][threadIdx.x % kRunThreads];
                mine[0] = m;
                mine[kRunThreads] = l;
                mine[2 * kRunThreads] = ld;
#pragma unroll
                for (int e = 0; e < 16; ++e) mine[(3 + e) * kRunThreads] = acc[e];
            }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < kRuns - 1; ++k) {
                if (run > 0) break;
                const float* other = &s_run[k][0][threadIdx.x];
                const float mo = other[0];
                if (mo == -INFINITY) continue;
                const float m_new = fmaxf(m, mo), keep = m > -INFINITY ? fast_exp2(m - m_new) : 0.f, w = fast_exp2(mo - m_new);
                m = m_new;
                l = fmaf(other[kRunThreads], w, l * keep);
                ld = fmaf(other[2 * kRunThreads], w, ld * keep);
#pragma unroll
                for (int e = 0; e < 16; ++e) acc[e] = fmaf(other[(3 + e) * kRunThreads], w, acc[e] * keep);
            }
        }
        const int rg = head.row_first + r, h = p.q_len.quotient(rg), j = rg - h * lq;
        if (valid) {
            const float inv = l == 0.f ? 0.f : 1.f / l;              // a sum that is not a number stays one
            uint4* dst = reinterpret_cast<uint4*>(out_all + (size_t)head.layer * span.out_stride + (((size_t)head.b * lq + j) * n_q_heads + h) * kD + e0);
#pragma unroll
            for (int e = 0; e < 2; ++e)
                dst[e] = make_uint4(pack_bf16(acc[8 * e] * inv, acc[8 * e + 1] * inv), pack_bf16(acc[8 * e + 2] * inv, acc[8 * e + 3] * inv),
                                    pack_bf16(acc[8 * e + 4] * inv, acc[8 * e + 5] * inv), pack_bf16(acc[8 * e + 6] * inv, acc[8 * e + 7] * inv));
            if ((lane & 7) == 0) {
                ws.row_lse2[(size_t)head.lb * rows_total + rg] = ld == 0.f ? -INFINITY : m + log2f(ld);
                if (lse) lse[(size_t)head.lb * rows_total + rg] = (l == 0.f ? -INFINITY : m + log2f(l)) * kLn2;
            }
        }
    }
}

// Exercises the bounded wait by itself: one CTA initialises an mbarrier that nothing ever arrives on,
// every thread waits on it with the given limit, the wait gives up, and the CTA reports
// CF_ERR_TIMEOUT through the status word exactly as the attention kernel does.  No tensor memory,
// no copies in flight: the kernel returns by itself after about `limit_cycles` clocks.
__global__ void __launch_bounds__(128) wait_probe_kernel(int* status, long long limit_cycles) {
    __shared__ unsigned long long bar;
    __shared__ int abort_word;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bar), 1);
        abort_word = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const bool ok = mbar_wait(smem_u32(&bar), 0, &abort_word, limit_cycles);
    __syncthreads();
    if (threadIdx.x == 0 && !ok && abort_word) atomicCAS(status, 0, CF_ERR_TIMEOUT);
}

}  // namespace

int launch_wait_probe(const PlanView& pv, long long limit_cycles, cudaStream_t stream) {
    wait_probe_kernel<<<1, 128, 0, stream>>>(pv.status, limit_cycles);
    return cudaGetLastError() == cudaSuccess ? CF_OK : CF_ERR_CUDA;
}

bool attn_tc_supported(const cf_geom* g, const cf_batch* b) {
    return g->dtype == CF_BF16 && g->head_dim == 128 && b->total_tokens > 0;
}

// Query rows of a tile: the rows that share a kv head, spread evenly over as few 128-row tiles as hold them, whole warps.
int attn_tc_row_tile(const cf_geom* g, const cf_batch* b) {
    const long long rows = (long long)(g->n_q_heads / g->n_kv_heads) * b->q_len, tiles = (rows + kRowTile - 1) / kRowTile;
    return (int)std::min<long long>(kRowTile, ((rows + tiles - 1) / tiles + 31) / 32 * 32);
}

// Two parts per share of the line, one share per SM.
size_t attn_tc_part_rows() { return (size_t)2 * sm_count() * kRowTile; }

int launch_attn_tc(const cf_geom* g, const cf_batch* b, const PlanView& pv, const LayerSpan& span, const void* q,
                   const void* k, const void* v, const void* k_self, const void* v_self, long long self_stride,
                   const void* k_prefix, const void* v_prefix, long long prefix_stride, int prefix_len,
                   float scale_log2, const AttnWorkspace& ws, void* out, float* lse, cudaStream_t stream) {
    const int group = g->n_q_heads / g->n_kv_heads;
    const long long row_tiles = ((long long)group * b->q_len + ws.rg_rows - 1) / ws.rg_rows;
    // the line's positions are 32-bit
    const long long most = ((long long)pv.max_tiles + (long long)b->n_requests * (prefix_len / kTile + b->q_len / kTile + 2)) *
                           g->n_kv_heads * row_tiles * span.n_layers;
    if (most > 0x7fffffffLL || g->n_kv_heads >= (1 << 20)) return CF_ERR_INVALID_ARG;
    StoreMaps maps;
    const unsigned long long rows = (unsigned long long)b->total_tokens, row_bytes = (unsigned long long)b->token_stride * 2;
    const unsigned long long layer_bytes = span.n_layers > 1 ? (unsigned long long)span.kv_stride * 2 : rows * row_bytes;
    for (int i = 0; i < kBoxes; ++i) {
        int rc = make_rows_map(&maps.k[i], k, g->n_kv_heads, rows, row_bytes, span.n_layers, layer_bytes, (i + 1) * 16);
        if (rc == CF_OK) rc = make_rows_map(&maps.v[i], v, g->n_kv_heads, rows, row_bytes, span.n_layers, layer_bytes, (i + 1) * 16);
        if (rc != CF_OK) return rc;
    }
    // further key blocks: dense rows of the kv heads, layers `stride` elements apart
    const unsigned long long dense = (unsigned long long)g->n_kv_heads * kD * 2;
    auto block_maps = [&](CUtensorMap* mk, CUtensorMap* mv, const void* pk, const void* pvv, unsigned long long n, long long stride) {
        const unsigned long long layer = span.n_layers > 1 ? (unsigned long long)stride * 2 : n * dense;
        const int rc = make_rows_map(mk, pk, g->n_kv_heads, n, dense, span.n_layers, layer, kTile);
        return rc != CF_OK ? rc : make_rows_map(mv, pvv, g->n_kv_heads, n, dense, span.n_layers, layer, kTile);
    };
    maps.ks = maps.kp = maps.k[0];
    maps.vs = maps.vp = maps.v[0];
    if (k_self) {
        const int rc = block_maps(&maps.ks, &maps.vs, k_self, v_self, (unsigned long long)b->n_requests * b->q_len, self_stride);
        if (rc != CF_OK) return rc;
    }
    if (prefix_len > 0) {
        const int rc = block_maps(&maps.kp, &maps.vp, k_prefix, v_prefix, (unsigned long long)prefix_len, prefix_stride);
        if (rc != CF_OK) return rc;
    }
    const BatchView bv = make_batch_view(b);
    const int shares = std::min(sm_count(), kMaxCodedShares);
    typedef const __nv_bfloat16* In;
    const RowSources src = {static_cast<In>(q), static_cast<In>(k), static_cast<In>(v), static_cast<In>(k_self), static_cast<In>(v_self),
                            static_cast<In>(k_prefix), static_cast<In>(v_prefix), self_stride, prefix_stride, scale_log2, k_self ? 1 : 0, prefix_len};
    const long long units = (long long)span.n_layers * b->n_requests * g->n_kv_heads * row_tiles;
    // Few units in many shares each: from thirteen parts to a unit on.  Measured (attention and merge of a call over 50 documents of
    // 160 tokens, us, 32 rows against 8): 2 units (50 parts) 25.7 / 17.5; 6 (25) 22.2 / 18.8; 8 (18) 26.4 / 24.9; 10 (15) 24.3 /
    // 23.3; 12 (12) 25.3 / 26.4 and 26.4 / 27.7; 14 (11) 25.1 / 25.1; 16 (9) 26.7 / 28.2; 24 (6) 32.4 / 34.9; 48 (3) 38.9 / 42.2.
    const bool many_parts = units * 13 <= shares;
    const int merge_rows = many_parts ? 8 : 32, slices = (ws.rg_rows + merge_rows - 1) / merge_rows;
    const Params p = {bv, pv, ws, span, src, g->n_q_heads, g->n_kv_heads, (int)row_tiles, (prefix_len + kTile - 1) / kTile,
                      k_self ? (b->q_len + kTile - 1) / kTile : 0, shares, Divisor(b->q_len), Divisor((int)row_tiles), Divisor(g->n_kv_heads),
                      Divisor(b->n_requests), Divisor(slices), static_cast<__nv_bfloat16*>(out), lse};
    static PerDeviceOnce configured[2];
    auto run = [&](auto kernel, int which) {
        if (configure_smem_once(configured[which], kernel, kSmemBytes) != CF_OK) return (int)CF_ERR_CUDA;
        const int rc = launch_chained(kernel, dim3((unsigned)shares), kThreads, kSmemBytes, stream, maps, p);
        if (rc != CF_OK) return rc;
        const unsigned blocks = (unsigned)((many_parts ? units : shares) * slices);
        const auto merge = many_parts ? attn_tc_merge_kernel<8> : attn_tc_merge_kernel<32>;
        return launch_chained(merge, dim3(blocks), kMergeThreads, 0, stream, p);
    };
    return g->rope_layout == CF_ROPE_HALF ? run(attn_tc_kernel<CF_ROPE_HALF>, 0) : run(attn_tc_kernel<CF_ROPE_INTERLEAVED>, 1);
}

}  // namespace cf
