// What the kernels of the fused re-position + query-prefill attention share: the line of all key tiles that is cut into equal shares,
// what a share leaves for the merge, and rows computed from scratch.
#pragma once

#include <cstddef>

#include "cf_row_group.cuh"
#include "cf_tc_util.cuh"

namespace cf {
namespace line {

using namespace tc;

constexpr int kRowTile = 128;
constexpr int kBoxes = kTile / 16;                 // copy boxes are 16, 32, .. kTile rows high
constexpr int kTrigBytes = kD / 2 * 8;
constexpr int kMetaRing = 16, kSegRing = 16;
constexpr int kPrefSlots = 48;
constexpr float kSumLimit = 0x1p80f;               // a larger tile sum leaves the range: 2^47 are left for the values and the other tiles
static_assert(kTile % 32 == 0, "halves of whole groups of 16 keys");

struct StoreMaps {
    CUtensorMap k[kBoxes], v[kBoxes];              // the stores, one map per box height
    CUtensorMap ks, vs;                            // keys and values of the query tokens themselves (whole tiles)
    CUtensorMap kp, vp;                            // keys and values of a shared prefix cache (whole tiles)
};

// Keys of a tile in either CTA of a pair: half of the MMA's columns, which come in 32s.
__device__ __forceinline__ int pair_keys(int len) { return ((len + 31) >> 5) << 4; }

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

// PAIR: a unit is two neighbouring tiles of query rows, of which either CTA of a pair (blockIdx.x & 1) has one.
template <bool PAIR>
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
    sg.row0 = (unit - sg.kvh * line.row_tiles) * (PAIR ? 2 : 1) * ws.rg_rows + (PAIR ? (int)(blockIdx.x & 1) * ws.rg_rows : 0);
    sg.rows_here = max(0, min(ws.rg_rows, group * bv.q_len - sg.row0));
    return sg;
}

// What a CTA leaves for the merge kernel: the unit that begins in its share and goes on behind it (n_parts = 0: none).
struct ShareHead {
    int n_parts, lb, layer, b, row_first, rows_here, unused[2];          // row_first: of the unit among the rows of a request
};
static_assert(sizeof(ShareHead) == 32, "two 16-byte loads");

// Keys and values of a call outside the tensor maps, for rows that are computed from scratch.
struct RowSources {
    const __nv_bfloat16 *q, *k, *v, *ks, *vs, *kp, *vp;
    long long self_stride, prefix_stride;
    float scale_log2;
    int with_self, prefix_len;
};

// Everything the attention and merge kernels are told: one constant, so that the rarely taken paths can be handed its address.
struct Params {
    BatchView bv;
    PlanView pv;
    AttnWorkspace ws;
    LayerSpan span;
    RowSources src;
    int n_q_heads, n_kv_heads, row_tiles, n_prefix, n_self, max_shares;   // row_tiles: units of a kv head; n_prefix, n_self: key tiles; max_shares: CTAs
    int ctas;                                      // of a share
    Divisor q_len, tiles_of_rows, kv_heads, requests, merge_slices;       // of the batch; merge_slices: of a unit's rows in merge blocks
    __nv_bfloat16* out;
    float* lse;
};

// What row_lse2 holds of a row whose unit was cut, until its parts are merged: the share the unit begins in and the number of its
// parts, as a negative quiet NaN (a denominator that is not a number is written as the positive one).
constexpr uint32_t kPartsOf = 0xffc00000u;
constexpr int kMaxCodedShares = 1 << 10;
__device__ __forceinline__ uint32_t parts_code(int share, int n_parts) { return kPartsOf | ((uint32_t)n_parts << 10) | (uint32_t)share; }
__host__ __device__ __forceinline__ bool is_parts_code(uint32_t w) { return (w & kPartsOf) == kPartsOf; }
__host__ __device__ __forceinline__ int first_share(uint32_t w) { return (int)(w & (kMaxCodedShares - 1)); }
__host__ __device__ __forceinline__ int part_count(uint32_t w) { return (int)((w ^ kPartsOf) >> 10); }
// Parts that a merge may read from CTA `first` on, of `all` CTAs every one or every second (`ctas` to a share), where it was told of n.  A CTA whose wait ran out writes no
// words for its rows, so that a merge by units finds what the workspace held before: its results are not used (CF_ERR_TIMEOUT), its
// reads have to stay inside the workspace.  (A merge by shares needs no such bound, since that CTA leaves no ShareHead.)
__host__ __device__ __forceinline__ int bounded_parts(int first, int n, int all, int ctas) {
    const int most = (all - 1 - first >> (ctas == 2 ? 1 : 0)) + 1;      // (0 or less where there is no such CTA)
    return n < most ? n : most;
}

// A part computed from scratch is left in fp32, as the halves of its numbers, and its sum (never negative) says so by its sign: such
// rows are rounded to bf16 once, as results.  (Left in bf16 like other parts, whose probabilities are bf16 too, results of nine to
// fifteen parts were off by 2.3e-3 of their size against the 1.66e-3 of one rounding.  The merge adds the low halves in a loop of its own:
// beside the high ones, in the loop over all parts, they cost every merge 0.45 us, this way 0.15.)
constexpr uint32_t kHasLowHalves = 0x80000000u;
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
constexpr int kRowWarps = 16;
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
static_assert(alignof(RowScratch) == 16 && offsetof(RowScratch, q) % 16 == 0 && offsetof(RowScratch, o) % 16 == 0, "16-byte accesses");

// Up to eight query rows (every set bit of `set`, from row `row0` of the segment on) over the segment's key tiles, every warp
// with every sixteenth tile under a running maximum of its own.  Leaves what the epilogue leaves of a row - a finished row or
// the part of one - and the log-sum-exps of the document tiles.
template <int LAYOUT, bool PAIR>
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
    const bool works = !PAIR || warp < kRowWarps;                   // a pair's other warps keep the barriers
    rows::Stage& stage = sh.stage[works ? warp : 0];
    RowTile(&tile)[2] = sh.tile[works ? warp : 0];
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
    int t = works ? sh.sg.t_begin + warp : sh.sg.t_end, i = 0, now = 0;                     // the current tile lies in tile[now]
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
    if (works && (lane & 3) == 0) {
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
        const int w = works ? warp : 0;
        weight[x] = sh.m[w][r] > -INFINITY ? exp2f(sh.m[w][r] - top) : sh.l[w][r];            // nothing seen: 0 (or not a number)
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
        const float f = l == 0.f ? 0.f : 1.f / l;
        const float4 o = *reinterpret_cast<const float4*>(&sh.o[warp][lane * 4]);
        if (whole) {
            __nv_bfloat16* dst = out_all + (size_t)sh.sg.layer * span.out_stride + (((size_t)sh.sg.b * lq + jj) * n_q_heads + sh.sg.kvh * group + g) * kD;
            *reinterpret_cast<uint2*>(dst + lane * 4) = make_uint2(pack_bf16(o.x * f, o.y * f), pack_bf16(o.z * f, o.w * f));
        } else {                                                    // as they are: high halves where bf16 parts lie, low halves beside them
            const uint32_t x[4] = {__float_as_uint(o.x), __float_as_uint(o.y), __float_as_uint(o.z), __float_as_uint(o.w)};
            *reinterpret_cast<uint2*>(reinterpret_cast<uint16_t*>(ws.part_o) + slot * kD + lane * 4) =
                make_uint2(__byte_perm(x[0], x[1], 0x7632), __byte_perm(x[2], x[3], 0x7632));
            *reinterpret_cast<uint2*>(ws.part_low + slot * kD + lane * 4) = make_uint2(__byte_perm(x[0], x[1], 0x5410), __byte_perm(x[2], x[3], 0x5410));
        }
        if (lane == 0 && whole) {
            const size_t at = (size_t)sh.sg.lb * rows_total + (size_t)sh.sg.kvh * group * lq + row;
            const float row_lse2 = top + log2f(ld);
            ws.row_lse2[at] = row_lse2 == row_lse2 ? row_lse2 : __int_as_float(0x7fffffff);
            if (lse) lse[at] = (top + log2f(l)) * kLn2;
        } else if (lane == 0) {
            ws.part_m[slot] = l == 0.f ? -INFINITY : top > -INFINITY ? top : 0.f;   // (a sum that is not a number has to be seen)
            ws.part_l[slot] = __uint_as_float(__float_as_uint(l) | kHasLowHalves);
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
// 1109 -> 646; of 4 x 50 of 160, 28/4 heads, 75 us
// (64 in pairs), 202 -> 128 and 687 -> 732 (few tiles per share leave warps idle, and this path is where a pair's kernel spills: 96
// registers, 76 to 80 bytes of stores and 120 to 128 of loads, none without it).  With half of the rows out of range 4 x 50 documents,
// 28/4 heads, took 242 us and take 273 to 277, 4 x 100 on 32/8 heads 456 and 486: shares of many such rows walk their keys once per eight.
// Accuracy: a row that leaves its range in every share is off by 1.67e-3 of its size, one rounding, as when the merge computed it; one
// that leaves it in some shares only has ordinary parts, of bf16 probabilities, in the others (two thirds of the shares: 1.67e-3 ->
// 1.74e-3; rows that never leave it: 2.87e-3).
template <int LAYOUT, bool PAIR>
__device__ __forceinline__ void marked_from_scratch(const Params& p, RowScratch& sh, const Line& line) {
    const int group = p.n_q_heads / p.n_kv_heads, share = blockIdx.x >> (PAIR ? 1 : 0);
    if (threadIdx.x == 0) sh.x = line.cut(share);
#pragma unroll 1
    while (true) {
        __syncthreads();                                            // the segment before has been read
        if (sh.x >= line.cut(share + 1)) break;
        if (threadIdx.x == 0) sh.sg = segment_at<PAIR>(p.bv, p.pv, p.ws, line, group, sh.x, line.cut(share + 1));
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
            rows_from_scratch<LAYOUT, PAIR>(p, sh, w * 32, set);
        }
    }
}

// The kernel whose CTAs work in pairs (cf_attn_pair.cu); `shares` of the line, two CTAs each.
int launch_attn_pair(const StoreMaps& maps, const Params& p, int rope_layout, int shares, cudaStream_t stream);

}  // namespace line
}  // namespace cf
