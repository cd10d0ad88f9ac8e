// Tensor-core kernel of the cache-construction attention, C_d <- LLM(C_prefix, d) (Sec. 2.2), for bf16
// storage and head_dim 128: block-diagonal causal attention over a packed store.
//
// A work item is the query rows of as many whole tokens as fit 128 rows of a (layer, document, kv head); rows are numbered
// token-major (r = token * G + g), so that an item's queries are one box of the query tensor and it needs the prefix cache
// and the document's keys up to its last token only.  An item's keys are the sequence [prefix, padded to 16; document
// tokens], cut into tiles of 64.
//   warps 0-3  softmax, one query row per thread (= TMEM lane)
//   warps 4-7  epilogue: O / sum to global memory while the softmax is at the next item
//   warp 8     MMA issue, the warp converged and one lane elected (see elect_one)
//   warp 9     item descriptions and copies
// S = Q K^T and O += P V accumulate in tensor memory (two buffers of 64 columns and 128); P goes back as bf16 over the S
// columns already consumed.  A CTA holds 109 KB of shared memory and 256 tensor-memory columns, so two CTAs share an SM;
// CTAs are persistent.  What bounds an item is the chain QK^T, softmax, PV per key tile: no unit is busy for more than a
// quarter of the time.  So QK^T of the next tile, the next item's first one too, runs while the softmax is at the current
// one (tiles of 128 with one S buffer: the softmax waited 2200 cycles per tile for its S and worked for 2000), and the
// epilogue is taken out of the chain.  Rows pass through 2 KB of staging per warp, so that a store instruction writes 64
// bytes to each of 8 rows: one row per thread in 32-byte pieces kept the warps waiting for 2100 cycles per item.
// Softmax: one fixed reference per row, the maximum over the item's first 16 keys (every row sees the first one); P and the
// sums keep their relative precision up to 80 (log2 units) above that maximum.  A row that leaves this range ends as not a
// number and is computed again when the CTA's items are done.
// Bound by HBM for a few query heads per kv head: with 6 heads and a 64-token prefix 123 flops per byte.
// Measured (400 documents of 128-192 tokens, 12/2 heads, 4 layers, prefix 64): 660 us before
// (one issuing thread for copies and MMAs, two passes over S, rows staged through the value buffer), 449 us now; one layer
// of 60 ragged documents with 32 heads and a 41-token prefix 229 -> 100 us.
// Every mbarrier wait is bounded; on expiry the CTA reports CF_ERR_TIMEOUT in the status word.
#include <math_constants.h>

#include <algorithm>

#include "cf_row_group.cuh"
#include "cf_tc_util.cuh"

namespace cf {

namespace {

using namespace tc;

constexpr int kDocMmaWarp = 8, kDocLoadWarp = 9, kDocTcThreads = 320;   // behind four softmax and four epilogue warps
constexpr int kKeys = 64, kKeyChunks = kKeys / 16;           // keys of a tile
constexpr int kKeyHalf = kKeys * 128, kKeyTile = 2 * kKeyHalf;   // bytes: 64 dims of a tile, a tile
constexpr int kDocBoxes = 3;                                 // copy boxes of 16, 32 and 64 rows
constexpr int kItemRing = 8, kSumRing = 4;                   // QK^T runs two tiles, perhaps two items, ahead of PV, and the epilogue one behind
constexpr int kScratchWarps = 8;                             // of the CTA, that compute rows from scratch
constexpr float kDocSumLimit = 0x1p80f;                      // see cf_attn_tc.cu

struct DocMaps {
    CUtensorMap k[kDocBoxes], v[kDocBoxes];        // the documents' keys and values, one map per box height
    CUtensorMap kp[kDocBoxes], vp[kDocBoxes];      // the prefix cache
    CUtensorMap qm;                                // the queries: boxes of 64 dims x G heads x (128 / G) tokens
};

// index w = row tile + row_tiles * (kv head + n_kv_heads * (layer * n_docs + document))
struct DocItem {
    int w, layer, kvh, row_first, r0, rows_here, n_keys;      // n_keys: the padded prefix and the document keys; w < 0: no more items
};

// Shape of the item space.
struct DocGrid {
    int row_tiles, group, rows_per_tile, prefix_len, prefix_pad;
};

__device__ __forceinline__ DocItem doc_item(const DocAttnArgs& a, const DocGrid& dg, int layer, int doc, int kvh, int x) {
    DocItem it;
    it.w = x + dg.row_tiles * (kvh + a.n_kv_heads * (layer * a.n_docs + doc));
    it.layer = layer;
    it.kvh = kvh;
    it.row_first = __ldg(a.doc_offsets + doc);
    const int rows = (__ldg(a.doc_offsets + doc + 1) - it.row_first) * dg.group;
    it.r0 = x * dg.rows_per_tile;
    it.rows_here = min(dg.rows_per_tile, rows - it.r0);
    it.n_keys = dg.prefix_pad + (it.r0 + it.rows_here - 1) / dg.group + 1;   // document tokens up to the last row's
    return it;
}
__device__ __forceinline__ DocItem doc_item(const DocAttnArgs& a, const DocGrid& dg, int w) {
    const int yz = w / dg.row_tiles, z = yz / a.n_kv_heads, layer = z / a.n_docs;
    return doc_item(a, dg, layer, z - layer * a.n_docs, yz - z * a.n_kv_heads, w - yz * dg.row_tiles);
}

// The items of all layers, documents and kv heads lie on a line, each as long as its estimated cost, kItemCost + its keys;
// a CTA takes those that start in its equal share of the line.  Items dealt out in turn instead leave the slowest of 296 CTAs
// with 1.75 times the mean (60 ragged documents with 32 heads), since neighbours on a CTA come from row tiles of like number.
// kItemCost is what an item costs beside its keys, in keys: the first QK^T, the last PV and the epilogue.  Measured (us, for 0 /
// 128 / 256 / 512 / 1024): 60 documents of 47-391 tokens, 32/32 heads 136 / 110 / 114 / 114 / 120; 40 of 24-400, 32/8, two layers
// 120 / 89 / 92 / 93 / 97; 30 of 300-400, 12/2, eight layers 194 / 191 / 191 / 196 / 200; 400 of 128-192, 12/2, four layers 447 /
// 443 / 443 / 445 / 446: what it stands for matters, its value between 128 and 512 does not.
constexpr int kItemCost = 256;
struct DocWalk {
    int layer, doc, kvh, x, tiles, len;                       // the current item; row tiles and tokens of its document
    long long pos, end;                                       // where it starts on the line; where the share ends
};
__device__ __forceinline__ int walk_len(const DocAttnArgs& a, int doc) {
    return doc < a.n_docs ? __ldg(a.doc_offsets + doc + 1) - __ldg(a.doc_offsets + doc) : 0;
}
__device__ __forceinline__ int walk_tiles(const DocGrid& dg, int len) {
    const int tokens = dg.rows_per_tile / dg.group;
    return max(0, min(dg.row_tiles, (len + tokens - 1) / tokens));
}
__device__ __forceinline__ int tile_cost(const DocGrid& dg, int len, int x) {
    return kItemCost + dg.prefix_pad + min((x + 1) * (dg.rows_per_tile / dg.group), len);
}
__device__ __forceinline__ long long doc_cost(const DocGrid& dg, int len) {
    const long long tokens = dg.rows_per_tile / dg.group, tiles = walk_tiles(dg, len);
    return tiles == 0 ? 0 : tiles * (kItemCost + dg.prefix_pad) + tokens * (tiles * (tiles - 1) / 2) + min(tiles * tokens, (long long)len);
}
__device__ __forceinline__ void walk_next(const DocAttnArgs& a, const DocGrid& dg, DocWalk& w) {
    w.pos += tile_cost(dg, w.len, w.x);
    if (++w.x < w.tiles) return;
    w.x = 0;
    if (++w.kvh < a.n_kv_heads) return;
    w.kvh = 0;
    do {
        if (w.pos >= w.end) return;                           // the share ends here, perhaps the line with it
        if (++w.doc == a.n_docs) {
            w.doc = 0;
            ++w.layer;
        }
        w.len = walk_len(a, w.doc);
        w.tiles = walk_tiles(dg, w.len);
    } while (w.tiles == 0);
}
// The first item of this CTA's share, by a whole warp; pos >= end: there is none.
__device__ __forceinline__ DocWalk walk_begin(const DocAttnArgs& a, const DocGrid& dg) {
    const int lane = threadIdx.x & 31;
    DocWalk w = {};
    long long all = 0;
    for (int d = lane; d < a.n_docs; d += 32) all += doc_cost(dg, walk_len(a, d));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) all += __shfl_xor_sync(0xffffffffu, all, o);
    if (all == 0) return w;
    const long long per_layer = all * a.n_kv_heads, line = per_layer * a.n_layers;
    const long long begin = line / gridDim.x * blockIdx.x + line % gridDim.x * blockIdx.x / gridDim.x;
    w.end = line / gridDim.x * (blockIdx.x + 1) + line % gridDim.x * (blockIdx.x + 1) / gridDim.x;
    if (begin == w.end) return w;
    w.layer = (int)(begin / per_layer);
    long long rest = begin - w.layer * per_layer;             // within the layer, then within the document, then within the kv head
    for (int d0 = 0; d0 < a.n_docs; d0 += 32) {
        const int len = walk_len(a, d0 + lane);
        const long long mine = doc_cost(dg, len) * a.n_kv_heads;
        long long upto = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long below = __shfl_up_sync(0xffffffffu, upto, o);
            if (lane >= o) upto += below;
        }
        const unsigned past = __ballot_sync(0xffffffffu, upto > rest);
        if (past) {
            const int at = __ffs((int)past) - 1;
            rest -= __shfl_sync(0xffffffffu, upto - mine, at);
            w.doc = d0 + at;
            w.len = __shfl_sync(0xffffffffu, len, at);
            break;
        }
        rest -= __shfl_sync(0xffffffffu, upto, 31);
    }
    w.tiles = walk_tiles(dg, w.len);
    const long long per_head = doc_cost(dg, w.len);
    w.kvh = (int)(rest / per_head);
    w.pos = begin - (rest - w.kvh * per_head);                // start of the kv head's first item
    while (w.pos < begin) walk_next(a, dg, w);
    return w;
}

// Byte offset of 16-byte piece x (0..3) of row r in a staging block of 32 rows of 64 bytes: eight lanes of consecutive rows, and
// of consecutive pieces, fall on all banks.
__device__ __forceinline__ int stage_at(int r, int x) { return r * 64 + ((x ^ ((r >> 1) & 3)) << 4); }

struct DocShared {
    unsigned char stage[4][32 * 64];

    unsigned long long k_full[2], s_full[2], pv_ready[2], o_done[2];   // of even and of odd key tiles
    unsigned long long q_full, o_full, o_free;               // one phase per item
    unsigned long long item_full[kItemRing], sums_full[kSumRing];
    unsigned int tmem_base;
    volatile int abort_flag;
    int marked;                                               // a row left the range of its reference
    float row_sum[kSumRing][kTile128], row_ref[kSumRing][kTile128];   // sum NaN: the row left the range of its reference
    DocItem item[kItemRing];
    DocWalk walk;                                             // the share's first item
};
constexpr int kDocTcSmem = 3 * kTileBytes + (int)sizeof(DocShared) + 1024;   // Q, K, V tiles
static_assert(2 * (kDocTcSmem + 1024) <= 228 * 1024, "two CTAs per SM");

struct DocParams {
    DocAttnArgs a;
    DocGrid dg;
    const __nv_bfloat16 *q, *k, *v, *kp, *vp;
    __nv_bfloat16* out;
    float* lse;
    int* status;
};
// What a warp that computes rows from scratch holds in the shared memory of the tiles.
struct DocScratch {
    rows::Queries q;
    rows::Stage stage;
};
static_assert(kScratchWarps * sizeof(DocScratch) <= 3 * kTileBytes, "fits the tiles' memory");

// Up to eight rows (r0 + every set bit of `set`) of an item by one warp, under a running maximum.
__device__ __noinline__ void doc_rows_from_scratch(const DocParams& p, DocScratch& sh, int w, int r0, unsigned set) {
    const int lane = threadIdx.x & 31, group = p.dg.group, n_rows = __popc(set);
    const DocItem it = doc_item(p.a, p.dg, w);
    // of a row of the group: its token, and where it lies among the document's rows of queries
    auto token_of = [&](int n) { return (it.r0 + r0 + rows::nth_bit(set, n)) / group; };
    auto place_of = [&](int n) {
        const int row = it.r0 + r0 + rows::nth_bit(set, n), token = row / group;
        return (size_t)(it.row_first + token) * p.a.n_q_heads + it.kvh * group + row - token * group;
    };
    for (int i = 0; i < rows::kGroupRows; i += 2) {
        const int r = i + (lane >> 4);
        sh.q.put(r, lane & 15, p.q + (size_t)it.layer * p.a.q_layer_stride + place_of(r) * kD);
    }
    const int token = token_of(lane >> 2), n_tokens = token_of(n_rows - 1) + 1;    // rows are numbered token by token
    const int prefix_steps = (p.dg.prefix_len + rows::kStepKeys - 1) / rows::kStepKeys;
    const int steps = prefix_steps + (n_tokens + rows::kStepKeys - 1) / rows::kStepKeys;
    auto copy = [&](auto& to, const __nv_bfloat16* prefix, const __nv_bfloat16* tokens, int s) {
        if (s < prefix_steps) {
            const int i = s * rows::kStepKeys;
            const size_t pitch = (size_t)p.a.n_kv_heads * kD;
            rows::copy_step(to, prefix + (size_t)it.layer * p.a.prefix_layer_stride + i * pitch + it.kvh * kD, pitch, p.dg.prefix_len - i);
        } else if (s < steps) {
            const int i = (s - prefix_steps) * rows::kStepKeys;
            rows::copy_step(to, tokens + (size_t)it.layer * p.a.kv_layer_stride + (size_t)(it.row_first + i) * p.a.token_stride + it.kvh * kD,
                            (size_t)p.a.token_stride, n_tokens - i);
        }
        rows::copies_end();
    };
    rows::Group acc;
    acc.clear();
    copy(sh.stage.k, p.kp, p.k, 0);
    copy(sh.stage.v, p.vp, p.v, 0);
    for (int s = 0; s < steps; ++s) {
        const int i = (s < prefix_steps ? s : s - prefix_steps) * rows::kStepKeys;
        rows::Keys keys;
        rows::copies_wait();
        keys.read(sh.stage);
        __syncwarp();                                               // every lane has its fragments
        copy(sh.stage.k, p.kp, p.k, s + 1);
        float alpha;
        acc.scores(sh.q, keys, (s < prefix_steps ? p.dg.prefix_len : token + 1) - i, p.a.scale_log2, alpha);
        rows::copies_wait();
        acc.values(sh.stage);
        __syncwarp();
        copy(sh.stage.v, p.vp, p.v, s + 1);
    }
    const float l = rows::over_keys(acc.l), inv = 1.f / l;
#pragma unroll
    for (int x = 0; x < 2; ++x) {                                   // rows 2 t and 2 t + 1
        const int r = 2 * (lane & 3) + x;
        const float f = __shfl_sync(0xffffffffu, inv, 4 * r);
        __nv_bfloat16* out = p.out + (size_t)it.layer * p.a.out_layer_stride + place_of(r) * kD + 8 * (lane >> 2);
        if (r < n_rows)
#pragma unroll
            for (int i = 0; i < 8; ++i)
                *reinterpret_cast<uint32_t*>(out + (i >> 2) * 64 + 2 * (i & 3)) = pack_bf16(acc.o[i][x] * f, acc.o[i][x + 2] * f);
    }
    if ((lane & 3) == 0 && (lane >> 2) < n_rows && p.lse) {
        const size_t place = place_of(lane >> 2);
        const int h = (int)(place % p.a.n_q_heads);
        p.lse[((size_t)it.layer * p.a.n_q_heads + h) * p.a.total_tokens + it.row_first + token] = (acc.m + log2f(l)) * kLn2;
    }
    __syncwarp();                                                   // the queries have been read
}

// Rows that left the range of their reference, by one of kScratchWarps warps: the share's items are walked once more, the rows that
// are not numbers computed by groups of eight in the memory of the tiles (whose copies and readers are done).  Other rows keep
// what they have, whatever their neighbours' keys are.  Measured (400 documents of 128-192 tokens, 12/2 heads, four layers, 446 us
// without such rows): a key far above the others in one kv head of every tenth document 74 -> 1.3 ms, in every document and head
// 74 -> 6.2 ms, against a warp per row, key after key, and with more than 256 such rows in a CTA all of its rows.
__device__ __noinline__ void doc_marked_from_scratch(const DocParams& p, DocScratch& sh, DocWalk walk) {
    const DocGrid& dg = p.dg;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int turn = 0; walk.pos < walk.end; walk_next(p.a, dg, walk)) {
        const DocItem it = doc_item(p.a, dg, walk.layer, walk.doc, walk.kvh, walk.x);
        for (int r0 = 0; r0 < it.rows_here; r0 += 32) {
            if (turn++ % kScratchWarps != warp) continue;
            const int row = it.r0 + min(r0 + lane, it.rows_here - 1), token = row / dg.group;
            const size_t place = (size_t)(it.row_first + token) * p.a.n_q_heads + it.kvh * dg.group + row - token * dg.group;
            const float first = __bfloat162float(p.out[(size_t)it.layer * p.a.out_layer_stride + place * kD]);
            for (unsigned set = __ballot_sync(0xffffffffu, first != first && r0 + lane < it.rows_here); set;) {
                const unsigned now = rows::next_group(set);
                doc_rows_from_scratch(p, sh, it.w, r0, now);
                set ^= now;
            }
        }
    }
}

__global__ void __launch_bounds__(kDocTcThreads, 2)
docattn_tc_kernel(const __grid_constant__ DocMaps maps, const __grid_constant__ DocParams p) {
    extern __shared__ unsigned char smem_raw[];
    chain_next();
    chain_wait();
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t q_base = smem_u32(smem), k_base = q_base + kTileBytes, v_base = k_base + 2 * kKeyTile;
    DocShared* sh = reinterpret_cast<DocShared*>(smem + 3 * kTileBytes);
    volatile int* abort_flag = &sh->abort_flag;
    const DocGrid& dg = p.dg;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    // rows of the query tile behind the box are never written: zero them once (their results are not stored)
    for (int idx = tid; idx < (kTile128 - dg.rows_per_tile) * 16; idx += kDocTcThreads) {
        const int chunk = idx & 15, r = dg.rows_per_tile + (idx >> 4);
        *reinterpret_cast<uint4*>(smem + (chunk >> 3) * kHalfBytes + swz(r, chunk & 7)) = make_uint4(0u, 0u, 0u, 0u);
    }
    fence_proxy_async();
    if (warp == kDocMmaWarp) {
        if (lane == 0) {
            for (int i = 0; i < 2; ++i) {
                mbar_init(smem_u32(&sh->k_full[i]), 1);
                mbar_init(smem_u32(&sh->s_full[i]), 1);
                mbar_init(smem_u32(&sh->pv_ready[i]), 5);           // P of four warps and the values
                mbar_init(smem_u32(&sh->o_done[i]), 1);
            }
            mbar_init(smem_u32(&sh->q_full), 1);
            for (int i = 0; i < kSumRing; ++i) mbar_init(smem_u32(&sh->sums_full[i]), 4);
            mbar_init(smem_u32(&sh->o_full), 1);
            mbar_init(smem_u32(&sh->o_free), 4);
            for (int i = 0; i < kItemRing; ++i) mbar_init(smem_u32(&sh->item_full[i]), 1);
            sh->abort_flag = 0;
            sh->marked = 0;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;" ::"r"(smem_u32(&sh->tmem_base)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();                                                // barriers are initialised, tensor memory is allocated
    tc_fence_after();
    const uint32_t tmem = sh->tmem_base;

    if (warp == kDocLoadWarp) {
        // -------------------------------------------------------------- items and copies
        // Keys or values of key tile i of an item, the g-th of this CTA: the prefix rows (whole chunks of 16, zeros behind the last row), then the document's.
        auto load = [&](const DocItem& it, int i, int g, bool values) {
            const int k0 = i * kKeys, p_len = max(0, min(kKeys, dg.prefix_pad - k0));
            const int doc_first = max(0, k0 - dg.prefix_pad);
            const int n16 = (min(kKeys, it.n_keys - k0) + 15) >> 4;
            const uint32_t bar = smem_u32(values ? &sh->pv_ready[g & 1] : &sh->k_full[g & 1]), dst = (values ? v_base : k_base) + (g & 1) * kKeyTile;
            mbar_expect_tx(bar, n16 * (16 * 256));
            auto rows = [&](const CUtensorMap* boxes, int at, int n, int row) {   // n chunks of 16 rows to row `at` of the tile
#pragma unroll
                for (int b = kDocBoxes - 1; b >= 0; --b) {
                    if (!(n >> b & 1)) continue;
                    tma_load_4d(dst + at * 128, boxes + b, 0, it.kvh, row, it.layer, bar);
                    tma_load_4d(dst + kKeyHalf + at * 128, boxes + b, 64, it.kvh, row, it.layer, bar);
                    at += 16 << b;
                    row += 16 << b;
                }
            };
            if (p_len > 0) rows(values ? maps.vp : maps.kp, 0, p_len >> 4, k0);
            rows(values ? maps.v : maps.k, p_len, n16 - (p_len >> 4), it.row_first + doc_first);
        };
        int n = 0, g = 0;                                           // items and key tiles so far
        bool ok = true;
        DocItem before = {};
        int i_before = 0;
        auto values_before = [&](int g) {                               // the values of tile g - 1
            if (g > 2) ok = warp_wait(smem_u32(&sh->o_done[(g - 1) & 1]), (((g - 1) >> 1) - 1) & 1, abort_flag);   // PV has read those of g - 3
            if (ok && lane == 0) load(before, i_before, g - 1, true);
            __syncwarp();
        };
        DocWalk walk = walk_begin(p.a, dg);
        if (lane == 0) sh->walk = walk;
        for (; ok && walk.pos < walk.end; ++n) {
            const DocItem it = doc_item(p.a, dg, walk.layer, walk.doc, walk.kvh, walk.x);
            if (lane == 0) {
                sh->item[n % kItemRing] = it;
                mbar_arrive(smem_u32(&sh->item_full[n % kItemRing]));
            }
            walk_next(p.a, dg, walk);
            const int tiles = (it.n_keys + kKeys - 1) / kKeys;
            for (int i = 0; i < tiles && ok; ++i, ++g) {                // the values travel one tile behind the keys
                if (g > 1) ok = warp_wait(smem_u32(&sh->s_full[g & 1]), ((g >> 1) - 1) & 1, abort_flag);   // QK^T has read tile g - 2
                if (ok && lane == 0) load(it, i, g, false);
                __syncwarp();
                if (ok && i == 0) {
                    if (g > 0) ok = warp_wait(smem_u32(&sh->s_full[(g - 1) & 1]), ((g - 1) >> 1) & 1, abort_flag);   // and the last queries
                    if (ok && lane == 0) {
                        const uint32_t bar = smem_u32(&sh->q_full);
                        const int token = it.row_first + it.r0 / dg.group;
                        mbar_expect_tx(bar, dg.rows_per_tile * 256);
                        tma_load_4d(q_base, &maps.qm, 0, it.kvh * dg.group, token, it.layer, bar);
                        tma_load_4d(q_base + kHalfBytes, &maps.qm, 64, it.kvh * dg.group, token, it.layer, bar);
                    }
                    __syncwarp();
                }
                if (ok && g > 0) values_before(g);
                before = it;
                i_before = i;
            }
        }
        if (ok && g > 0) values_before(g);
        if (ok && lane == 0) {
            sh->item[n % kItemRing].w = -1;
            mbar_arrive(smem_u32(&sh->item_full[n % kItemRing]));
        }
    } else if (warp == kDocMmaWarp) {
        // -------------------------------------------------------------- MMA issue
        const uint64_t a0 = smem_desc(q_base, 16, 1024), bk = smem_desc(k_base, 16, 1024), bv = smem_desc(v_base, kKeyHalf, 1024);
        const uint32_t idesc_o = instr_desc(kD, true);
        int n16_before = 0, i_before = 0, n_before = 0;             // the tile whose PV is still to be issued (0: none) and its item
        bool last_before = false;
        int g = 0;
        bool ok = true;
        auto issue_pv = [&]() {                                     // PV of tile g - 1
            const int b = (g - 1) & 1;
            ok = warp_wait(smem_u32(&sh->pv_ready[b]), ((g - 1) >> 1) & 1, abort_flag);
            if (!ok) return;
            tc_fence_after();
            if (i_before == 0 && n_before > 0) {                    // the epilogue has read the rows of the item before
                ok = warp_wait(smem_u32(&sh->o_free), (n_before - 1) & 1, abort_flag);
                if (!ok) return;
                tc_fence_after();
            }
            if (elect_one()) {
                for (int kk = 0; kk < n16_before; ++kk)             // 16 keys = 8 packed P columns per instruction
                    umma_ts(tmem + 128, tmem + b * kKeys + kk * 8, bv + (uint64_t)(b * (kKeyTile >> 4) + kk * 128), idesc_o, (i_before > 0 || kk > 0) ? 1u : 0u);
                umma_commit(smem_u32(&sh->o_done[b]));
                if (last_before) umma_commit(smem_u32(&sh->o_full));
            }
            __syncwarp();
        };
        for (int n = 0; ok; ++n) {
            ok = warp_wait(smem_u32(&sh->item_full[n % kItemRing]), (n / kItemRing) & 1, abort_flag);
            if (!ok) break;
            const int n_keys = sh->item[n % kItemRing].w < 0 ? 0 : sh->item[n % kItemRing].n_keys;
            if (n_keys == 0) {
                if (n16_before > 0) issue_pv();
                break;
            }
            for (int i = 0; i * kKeys < n_keys; ++i, ++g) {
                // S of this tile, into the buffer that the PV before the last has read, while the softmax is at the tile before
                const int b = g & 1;
                if (i == 0) ok = warp_wait(smem_u32(&sh->q_full), n & 1, abort_flag);
                if (ok) ok = warp_wait(smem_u32(&sh->k_full[b]), (g >> 1) & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                const int n16 = (min(kKeys, n_keys - i * kKeys) + 15) >> 4;
                const uint32_t idesc = instr_desc(n16 * 16, false);
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk)
                        umma(tmem + b * kKeys, a0 + (uint64_t)(((kk >> 2) * kHalfBytes + (kk & 3) * 32) >> 4),
                             bk + (uint64_t)((b * kKeyTile + (kk >> 2) * kKeyHalf + (kk & 3) * 32) >> 4), idesc, kk > 0);
                    umma_commit(smem_u32(&sh->s_full[b]));
                }
                __syncwarp();
                if (n16_before > 0) issue_pv();
                if (!ok) break;
                n16_before = n16;
                i_before = i;
                n_before = n;
                last_before = (i + 1) * kKeys >= n_keys;
            }
        }
    } else if (warp < 4) {
        // -------------------------------------------------------------- softmax, one row per thread
        const uint32_t lane_tmem = tmem + ((uint32_t)(warp * 32) << 16);
        const uint64_t scale2 = pack_f2(p.a.scale_log2, p.a.scale_log2);
        const int group = dg.group;
        const int hole = dg.prefix_pad > dg.prefix_len ? (dg.prefix_pad >> 4) - 1 : -1;       // the chunk with padding keys
        const int hole_valid = dg.prefix_len - hole * 16;
        int g = 0;
        bool ok = true;
        for (int n = 0; ok; ++n) {
            ok = warp_wait(smem_u32(&sh->item_full[n % kItemRing]), (n / kItemRing) & 1, abort_flag);
            if (!ok) break;
            const DocItem it = sh->item[n % kItemRing];
            if (it.w < 0) break;
            const int last_row = it.r0 + it.rows_here - 1;
            const int row = min(it.r0 + tid, last_row);                 // rows beyond the end follow the last valid one
            const int token = row / group;
            // keys of the sequence that the row sees, and the least and the most among the warp's rows
            const int lim = dg.prefix_pad + token + 1;
            const int lim_lo = __shfl_sync(0xffffffffu, lim, 0), lim_hi = __shfl_sync(0xffffffffu, lim, 31);
            float ref = 0.f, l_run = 0.f;
            uint64_t neg_ref2 = 0;
            const int chunks = (it.n_keys + 15) >> 4;
            for (int c0 = 0; c0 < chunks; c0 += kKeyChunks, ++g) {      // a tile: chunks c0 .. c0 + 3 of the sequence
                const int n16 = min(kKeyChunks, chunks - c0);
                const uint32_t s_addr = lane_tmem + (g & 1) * kKeys;
                ok = warp_wait(smem_u32(&sh->s_full[g & 1]), (g >> 1) & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                const int full = (lim_lo >> 4) - c0, some = min(n16, ((lim_hi + 15) >> 4) - c0);   // chunks every row sees; any row sees
                uint64_t sum2 = 0;
                auto chunk = [&](int c, uint32_t (&v)[16]) {
                    if (c < full && c0 + c != hole) {
                        chunk16_exp(v, scale2, neg_ref2, sum2);
                    } else {
                        chunk16_exp_masked(v, min(lim - (c0 + c) * 16, c0 + c == hole ? hole_valid : 16), scale2, neg_ref2, sum2);
                    }
                    tmem_st8_async(s_addr + c * 8, v);                  // over S columns already in registers
                };
                uint32_t va[16], vb[16];
                tmem_ld16_async(s_addr, va);
                tmem_ld16_wait(va);
                if (c0 == 0) {
                    const float m = chunk16_max(va, min(lim, hole == 0 ? hole_valid : 16));
                    ref = m * p.a.scale_log2;
                    neg_ref2 = pack_f2(-ref, -ref);
                }
                for (int c = 0; c < some; c += 2) {
                    if (c > 0) tmem_ld16_wait(va);
                    if (c + 1 < some) tmem_ld16_async(s_addr + (c + 1) * 16, vb);
                    chunk(c, va);
                    if (c + 1 >= some) break;
                    tmem_ld16_wait(vb);
                    if (c + 2 < some) tmem_ld16_async(s_addr + (c + 2) * 16, va);
                    chunk(c + 1, vb);
                }
                if (some < n16) {
#pragma unroll
                    for (int x = 0; x < 8; ++x) va[x] = 0u;
                    for (int c = max(some, 0); c < n16; ++c) tmem_st8_async(s_addr + c * 8, va);
                }
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&sh->pv_ready[g & 1]));
                float s0, s1;
                unpack_f2(sum2, s0, s1);
                l_run += s0 + s1 <= kDocSumLimit ? s0 + s1 : CUDART_NAN_F;
            }
            if (!ok) break;
            sh->row_sum[n % kSumRing][tid] = l_run;                     // item n - 4 has left: its rows made way for the PV of item n - 2
            sh->row_ref[n % kSumRing][tid] = ref;
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&sh->sums_full[n % kSumRing]));
        }
    } else {
        // -------------------------------------------------------------- epilogue, one row per thread
        const int r = tid - 128;
        const uint32_t o_addr = tmem + 128 + ((uint32_t)((warp & 3) * 32) << 16);
        unsigned char* stage = sh->stage[warp & 3];
        const int group = dg.group;
        bool ok = true;
        for (int n = 0; ok; ++n) {
            ok = warp_wait(smem_u32(&sh->item_full[n % kItemRing]), (n / kItemRing) & 1, abort_flag);
            if (!ok) break;
            const DocItem it = sh->item[n % kItemRing];
            if (it.w < 0) break;
            const int row = it.r0 + min(r, it.rows_here - 1), token = row / group;
            const int at = token * p.a.n_q_heads + it.kvh * group + row - token * group;   // the row among the document's
            __nv_bfloat16* out = p.out + (size_t)it.layer * p.a.out_layer_stride + (size_t)it.row_first * p.a.n_q_heads * kD + (lane & 3) * 8;
            ok = warp_wait(smem_u32(&sh->sums_full[n % kSumRing]), (n / kSumRing) & 1, abort_flag);
            if (!ok) break;
            const float sum = sh->row_sum[n % kSumRing][r], inv = 1.f / sum;
            if (r < it.rows_here) {
                if (p.lse)
                    p.lse[((size_t)it.layer * p.a.n_q_heads + it.kvh * group + row - token * group) * p.a.total_tokens + it.row_first + token] =
                        (sh->row_ref[n % kSumRing][r] + log2f(sum)) * kLn2;
                if (sum != sum) sh->marked = 1;                         // its output row is not a number either
            }
            ok = warp_wait(smem_u32(&sh->o_full), n & 1, abort_flag);
            if (!ok) break;
            tc_fence_after();
            uint32_t o[32];
            tmem_ld32_async(o_addr, o);
#pragma unroll
            for (int c = 0; c < 4; ++c) {                               // 32 dims at a time, four 16-byte pieces
                uint32_t u[16];
                tmem_ld_wait(o);
#pragma unroll
                for (int x = 0; x < 16; ++x) u[x] = pack_bf16(__uint_as_float(o[2 * x]) * inv, __uint_as_float(o[2 * x + 1]) * inv);
                if (c < 3) {
                    tmem_ld32_async(o_addr + (c + 1) * 32, o);
                } else {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&sh->o_free));
                }
                __syncwarp();                                           // the pieces before have been read
#pragma unroll
                for (int x = 0; x < 4; ++x)
                    *reinterpret_cast<uint4*>(stage + stage_at(lane, x)) = make_uint4(u[4 * x], u[4 * x + 1], u[4 * x + 2], u[4 * x + 3]);
                __syncwarp();
#pragma unroll
                for (int x = 0; x < 32; x += 8) {
                    const int rr = x + (lane >> 2);
                    const int to = __shfl_sync(0xffffffffu, at, rr);
                    if ((warp & 3) * 32 + rr < it.rows_here)
                        *reinterpret_cast<uint4*>(out + (size_t)to * kD + c * 32) = *reinterpret_cast<const uint4*>(stage + stage_at(rr, lane & 3));
                }
            }
        }
    }

    // ---------------------------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    if (sh->abort_flag) {
        // a wait expired: let the loads in flight (at most a tile of each operand) land before the shared memory is given back
        if (warp == kDocMmaWarp && lane == 0) {
            const long long t0 = clock64();
            while (clock64() - t0 < kWaitLimitCycles / 64) {}
        }
        if (tid == 0 && p.status) atomicCAS(p.status, 0, CF_ERR_TIMEOUT);
        __syncthreads();
    }
    if (warp == kDocMmaWarp) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" ::"r"(tmem) : "memory");
    }
    if (sh->marked && !sh->abort_flag && warp < kScratchWarps) doc_marked_from_scratch(p, reinterpret_cast<DocScratch*>(smem)[warp], sh->walk);
}

}  // namespace

bool docattn_tc_supported(const cf_geom* g, const cf_doc_batch* docs) {
    return g->dtype == CF_BF16 && g->head_dim == 128 && docs->total_tokens > 0 &&
           g->n_q_heads / g->n_kv_heads <= kTile128;                   // an item holds at least one whole token
}

int launch_docattn_tc(const cf_geom* g, const DocAttnArgs& a, const void* q, const void* k, const void* v,
                      const void* kp, const void* vp, void* out, float* lse, int* status, cudaStream_t stream) {
    const int group = a.n_q_heads / a.n_kv_heads;
    if (group > kTile128) return CF_ERR_UNSUPPORTED;
    const int rows_per_tile = (kTile128 / group) * group;              // whole tokens
    const long long row_tiles = ((long long)a.max_doc_len * group + rows_per_tile - 1) / rows_per_tile;
    const long long total = row_tiles * a.n_kv_heads * (long long)a.n_docs * a.n_layers;   // work items, empty ones included
    if (row_tiles <= 0 || total > 0x7fffffffLL - 65536) return CF_ERR_INVALID_ARG;
    DocMaps maps;
    const unsigned long long row_bytes = (unsigned long long)a.token_stride * 2;
    const unsigned long long layer_bytes = a.n_layers > 1 ? (unsigned long long)a.kv_layer_stride * 2
                                                          : (unsigned long long)a.total_tokens * row_bytes;
    const unsigned long long prow = (unsigned long long)a.n_kv_heads * kD * 2;
    const unsigned long long player = a.n_layers > 1 ? (unsigned long long)a.prefix_layer_stride * 2
                                                     : (unsigned long long)a.prefix_len * prow;
    for (int i = 0; i < kDocBoxes; ++i) {
        int rc = make_rows_map(&maps.k[i], k, a.n_kv_heads, (unsigned long long)a.total_tokens, row_bytes, a.n_layers, layer_bytes, 16 << i);
        if (rc == CF_OK)
            rc = make_rows_map(&maps.v[i], v, a.n_kv_heads, (unsigned long long)a.total_tokens, row_bytes, a.n_layers, layer_bytes, 16 << i);
        if (rc == CF_OK && a.prefix_len > 0) {
            rc = make_rows_map(&maps.kp[i], kp, a.n_kv_heads, (unsigned long long)a.prefix_len, prow, a.n_layers, player, 16 << i);
            if (rc == CF_OK)
                rc = make_rows_map(&maps.vp[i], vp, a.n_kv_heads, (unsigned long long)a.prefix_len, prow, a.n_layers, player, 16 << i);
        }
        if (rc != CF_OK) return rc;
    }
    {   // queries [layers][tokens][q heads][128] as (64 dims, q heads, tokens, layers); the two halves are fetched one by one
        EncodeTiledFn fn = encode_fn();
        if (!fn) return CF_ERR_CUDA;
        const unsigned long long qrow = (unsigned long long)a.n_q_heads * kD * 2;
        const unsigned long long qlayer = a.n_layers > 1 ? (unsigned long long)a.q_layer_stride * 2
                                                          : (unsigned long long)a.total_tokens * qrow;
        const cuuint64_t dims[4] = {(cuuint64_t)kD, (cuuint64_t)a.n_q_heads, (cuuint64_t)a.total_tokens, (cuuint64_t)a.n_layers};
        const cuuint64_t strides[3] = {(cuuint64_t)kD * 2, (cuuint64_t)qrow, (cuuint64_t)qlayer};
        const cuuint32_t box[4] = {64, (cuuint32_t)group, (cuuint32_t)(kTile128 / group), 1};
        const cuuint32_t elem[4] = {1, 1, 1, 1};
        if (fn(&maps.qm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(q), dims, strides, box, elem,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return CF_ERR_CUDA;
    }
    static PerDeviceOnce configured;
    if (configure_smem_once(configured, docattn_tc_kernel, kDocTcSmem) != CF_OK) return CF_ERR_CUDA;
    const int ctas = sm_count() > 0 ? 2 * sm_count() : 296;         // persistent: two CTAs per SM
    const unsigned grid = (unsigned)std::min<long long>(total, ctas);
    typedef const __nv_bfloat16* In;
    const DocParams p = {a, {(int)row_tiles, group, rows_per_tile, a.prefix_len, (a.prefix_len + 15) & ~15},
                         static_cast<In>(q), static_cast<In>(k), static_cast<In>(v), static_cast<In>(kp), static_cast<In>(vp),
                         static_cast<__nv_bfloat16*>(out), lse, status};
    return launch_chained(docattn_tc_kernel, dim3(grid), kDocTcThreads, kDocTcSmem, stream, maps, p);
}

}  // namespace cf
