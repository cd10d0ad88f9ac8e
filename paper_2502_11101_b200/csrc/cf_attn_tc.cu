// Fused re-position + query-prefill attention on the Blackwell tensor cores (bf16, head_dim 128).
//
// Eq. 5 fused into Eq. 1: key tiles are streamed from the un-repositioned store by TMA into 128B-swizzled shared memory,
// rotated there in place by their document's delta (fp32, one rounding: bit for bit what cf_reposition_keys writes) and
// handed to the tensor cores.
//
// Kv heads with several tiles of query rows are worked on by pairs of CTAs where shares are long enough (cf_attn_pair.cu).
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
// for every phase in order, since a wait for a parity passes early where it skipped one (what a pair's softmax does instead stands at
// softmax_role).
#include <algorithm>

#include "cf_attn_roles.cuh"

namespace cf {

using namespace line;

namespace {

constexpr int kThreads = 512;
constexpr int kRotateWarps = 6;
constexpr int kKvHalf = kTile * 128;               // one 64-column half of a key or value tile
constexpr int kKvBytes = 2 * kKvHalf;
constexpr int kKStages = 6, kVStages = 3;          // with the three S buffers of two warpgroups: everything repeats after six tiles
constexpr int kSBuffers = 3;
constexpr int kLoadWarp = 9, kMmaWarp = 12;
constexpr uint32_t kColO = 0, kColQ = 128, kColS = 192;
static_assert(kColS + kSBuffers * kTile <= 512, "tensor memory columns");
static_assert(kTile % 16 == 0 && kTile <= 96, "three S buffers");
static_assert(kKStages == 6 && kVStages == 3 && kSBuffers == 3, "rings of one period");

struct R {
    static constexpr bool kPair = false;
    static constexpr int kSoftmaxGroups = 2, kKStages = 6, kSBuffers = 3;
    static constexpr uint32_t kColO = 0, kColQ = 128, kColS = 192;
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

struct Shared {
    Barriers bars;
    int4 meta[kMetaRing];                          // tiles in flight: length and flags, tile index or kind, first row, kv head and layer
    Segment segments[kSegRing];                    // of the share
    ShareHead head;
    Line line;
    float ref[2][kRowTile];                        // [segment parity][row]
    alignas(16) float2 trig[kKStages][kD / 2];     // cosines and sines of the documents of the key stages
    Sums<2> sums;
    Requests requests;
};
constexpr int kSmemBytes = (kKStages + kVStages) * kKvBytes + (int)sizeof(Shared) + 1024;
static_assert(kSmemBytes <= 227 * 1024, "shared memory of one CTA");
static_assert(sizeof(RowScratch) <= (kKStages + kVStages) * kKvBytes, "over the rings");

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
    const int group = n_q_heads / n_kv_heads, lq = bv.q_len, rows = group * lq;

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
            if (begin < end) sh.segments[0] = segment_at<false>(bv, pv, ws, l, group, begin, end);
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
                        sg = segment_at<false>(bv, pv, ws, line, group, x, x_end);
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
                    umma_ts_lit<1, false>(s_tmem, q_tmem, b0, idesc);
#pragma unroll
                    for (int kk = 1; kk < 8; ++kk)                  // 16 dims per instruction
                        umma_ts_lit<1, true>(s_tmem, q_tmem + kk * 8, b0 + (uint64_t)(((kk >> 2) * kKvHalf + (kk & 3) * 32) >> 4), idesc);
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
                for (int kk = 1; kk < steps; ++kk) umma_ts_lit<1, true>(o_tmem, p_tmem + kk * 8, b0 + (uint64_t)(kk * 128), idesc_o);
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
                rotate_rows<LAYOUT>(smem + (size_t)stage * kKvBytes, kKvHalf, reinterpret_cast<const float4*>(sh.trig[stage]), chunk, rsub, kRotateWarps * 4, len);
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
        softmax_role<R>(p, sh, sh.sums, nullptr, tmem, blockIdx.x, x_end, n_items);
    }

    // ---------------------------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    if (tid == 0) {
        ShareHead head = {};
        if (n_items > 0 && !bars.abort_flag) head = sh.head;       // (roles that gave up may not have come to the share's last segment)
        reinterpret_cast<ShareHead*>(ws.marks)[blockIdx.x] = head;
    }
    // every copy has landed and every MMA has read its operands: the rings are free
    if (bars.marked && !bars.abort_flag) marked_from_scratch<LAYOUT, false>(p, *reinterpret_cast<RowScratch*>(smem), line);
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
// have nothing to attend.  Weights are exp2f's, which keeps numbers below 2^-126: the documents' share of a row whose prefix lies
// that far above them is what their scores are measured against (with ex2.approx.ftz it was 0 and the scores infinite).
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
        const int u = p.tiles_of_rows.quotient(at), row_tile = at - u * (int)p.tiles_of_rows.d, kvh = p.kv_heads.remainder(u);
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
        share = first_share(word);                                  // (the CTA, for pairs that of this tile of rows)
        head.n_parts = bounded_parts(share, part_count(word), p.max_shares, p.ctas);
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
        uint32_t scratch = 0;
#pragma unroll
        for (int e = 0; e < 16; ++e) acc[e] = 0.f;
        // part i: the CTA's slot for what goes on behind its share (i = 0), the others' for what began before theirs
        const size_t slot0 = ((size_t)2 * share + 1) * kRowTile + min(r, head.rows_here - 1), slot1 = slot0 - kRowTile;
        auto slot_of = [&](int i) { return i == 0 ? slot0 : slot1 + (size_t)i * p.ctas * 2 * kRowTile; };
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
            const float keep = m > -INFINITY ? exp2f(m - m_new) : 0.f;
            m = m_new;
            l *= keep;
            ld *= keep;
            scratch |= __float_as_uint(lp[0]) | __float_as_uint(lp[1]) | __float_as_uint(lp[2]) | __float_as_uint(lp[3]);
#pragma unroll
            for (int e = 0; e < 16; ++e) acc[e] *= keep;
#pragma unroll
            for (int x = 0; x < 4; ++x)
                if (mp[x] > -INFINITY) {
                    const float w = exp2f(mp[x] - m_new);
                    l = fmaf(fabsf(lp[x]), w, l);
                    ld = fmaf(fabsf(dp[x]), w, ld);
                    const uint32_t pairs[8] = {o[x][0].x, o[x][0].y, o[x][0].z, o[x][0].w, o[x][1].x, o[x][1].y, o[x][1].z, o[x][1].w};
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        acc[2 * e] = fmaf(__uint_as_float(pairs[e] << 16), w, acc[2 * e]);
                        acc[2 * e + 1] = fmaf(__uint_as_float(pairs[e] & 0xffff0000u), w, acc[2 * e + 1]);
                    }
                }
        }
        if (scratch & kHasLowHalves) {                              // what the high halves leave of the parts computed from scratch
#pragma unroll 1
            for (int i = n_parts * run / kRuns; i < part_end; ++i) {
                const size_t slot = slot_of(i);
                const float mp = ws.part_m[slot];
                if (mp == -INFINITY || !(__float_as_uint(ws.part_l[slot]) & kHasLowHalves)) continue;
                const float w = exp2f(mp - m);
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    const uint32_t high = (uint32_t)reinterpret_cast<const uint16_t*>(part_o)[slot * kD + e] << 16;
                    const float part = __uint_as_float(high), rest = __uint_as_float(high | ws.part_low[slot * kD + e0 + e]) - part;
                    acc[e] = fmaf(fabsf(part) < INFINITY ? rest : 0.f, w, acc[e]);
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
                const float m_new = fmaxf(m, mo), keep = m > -INFINITY ? exp2f(m - m_new) : 0.f, w = exp2f(mo - m_new);
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

extern "C" int cf_debug_cut_row(uint32_t word, int32_t n_ctas, int32_t ctas_per_share, int32_t* first, int32_t* n_parts) {
    if (n_ctas <= 0 || (ctas_per_share != 1 && ctas_per_share != 2) || !first || !n_parts) return CF_ERR_INVALID_ARG;
    *first = is_parts_code(word) ? first_share(word) : -1;
    *n_parts = is_parts_code(word) ? bounded_parts(*first, part_count(word), n_ctas, ctas_per_share) : 0;
    return CF_OK;
}

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

// Whether CTAs work in pairs on two tiles of query rows (cf_attn_pair.cu).  A pair copies and rotates every key tile once for both,
// but starts later and leaves one of its CTAs without rows where their number is odd: what counts is how many key tiles a pair's share
// has.  Measured, attention and merge of a call (us, alone / in pairs; tiles of a share in brackets, documents of 160 tokens).
// Two tiles of rows, 32/8 heads: 25 documents (5) 31.7 / 31.7; 50 (11) 37.9 / 35.8; 4 x 50 (43) 74.7 / 60.4; four layers of 4 x 100 (346)
// 419 / 292.  Four, 28/4: 25 (5) 31.7 / 31.7; 4 x 12 (10) 35.8 / 33.8; 4 x 50 (43) 72.7 / 58.4; 12/2, 50 (5) 29.7 / 31.7.  Three, 12/2:
// 50 (5) 23.6 / 29.7; 4 x 100 (43) 58.4 / 58.4; four layers of that (173) 167 / 150; 28/4, 4 x 50 (43) 58.4 / 58.4; 4 x 100 (86) 95.2 /
// 89.1.  Five, 28/4: 4 x 12 (16) 37.9 / 37.9; 4 x 50 (65) 85.0 / 74.7.  The tiles are those the host knows of, a bound.  Without a hint
// that is all documents, however few are left (30 of 4 x 100 kept, 12/2, three tiles: 25.0 / 28.4; 3 kept: 12.5 / 15.0): an odd number,
// which gains a tenth at most, then stays alone.  An even one gains up to a third and loses 1 to 2 us with three kept (32/8, 3 of
// 4 x 100: 17.0 / 18.9).
static bool work_in_pairs(const cf_geom* g, const cf_batch* b, int n_layers, long long row_tiles, int more_tiles) {
    const long long documents = std::min((long long)b->n_requests * tiles_per_request_bound(b), (long long)b->n_docs_total + b->total_tokens / kTile + 1);
    const long long tiles = (documents + (long long)b->n_requests * more_tiles) * g->n_kv_heads * n_layers * ((row_tiles + 1) / 2);
    if (row_tiles % 2) return row_tiles > 1 && b->tiles_hint > 0 && tiles >= 44LL * (sm_count() / 2);
    return tiles >= 8LL * (sm_count() / 2);
}

static int more_tiles(const cf_batch* b, int prefix_len, bool with_self) {
    return (prefix_len + kTile - 1) / kTile + (with_self ? (b->q_len + kTile - 1) / kTile : 0);
}

extern "C" int cf_debug_attn_kernel(const cf_geom* geom, const cf_batch* batch, int32_t n_layers, int32_t prefix_len, int32_t with_self, int32_t* which) {
    if (!batch || !which || n_layers <= 0 || prefix_len < 0) return CF_ERR_INVALID_ARG;
    const int rc = validate(geom, batch);
    if (rc != CF_OK) return rc;
    const int rg_rows = attn_tc_row_tile(geom, batch);
    const long long rows = (long long)(geom->n_q_heads / geom->n_kv_heads) * batch->q_len;
    *which = attn_path() != 0 || !attn_tc_supported(geom, batch) ? 0
             : work_in_pairs(geom, batch, n_layers, (rows + rg_rows - 1) / rg_rows, more_tiles(batch, prefix_len, with_self != 0)) ? 2 : 1;
    return CF_OK;
}

int launch_attn_tc(const cf_geom* g, const cf_batch* b, const PlanView& pv, const LayerSpan& span, const void* q,
                   const void* k, const void* v, const void* k_self, const void* v_self, long long self_stride,
                   const void* k_prefix, const void* v_prefix, long long prefix_stride, int prefix_len,
                   float scale_log2, const AttnWorkspace& ws, void* out, float* lse, cudaStream_t stream) {
    const int group = g->n_q_heads / g->n_kv_heads;
    long long row_tiles = ((long long)group * b->q_len + ws.rg_rows - 1) / ws.rg_rows;
    const int n_prefix = (prefix_len + kTile - 1) / kTile, n_self = k_self ? (b->q_len + kTile - 1) / kTile : 0;
    const int ctas = work_in_pairs(g, b, span.n_layers, row_tiles, more_tiles(b, prefix_len, k_self != nullptr)) ? 2 : 1;      // of a share
    row_tiles = (row_tiles + ctas - 1) / ctas;                      // units of a kv head
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
        const int rc = make_rows_map(mk, pk, g->n_kv_heads, n, dense, span.n_layers, layer, kTile / ctas);
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
    const int shares = std::min(sm_count(), kMaxCodedShares) / ctas;   // of the line
    typedef const __nv_bfloat16* In;
    const RowSources src = {static_cast<In>(q), static_cast<In>(k), static_cast<In>(v), static_cast<In>(k_self), static_cast<In>(v_self),
                            static_cast<In>(k_prefix), static_cast<In>(v_prefix), self_stride, prefix_stride, scale_log2, k_self ? 1 : 0, prefix_len};
    const long long units = (long long)span.n_layers * b->n_requests * g->n_kv_heads * row_tiles;
    // Few units in many shares each: from thirteen parts to a unit on.  Measured (attention and merge of a call over 50 documents of
    // 160 tokens, us, 32 rows against 8): 2 units (50 parts) 25.7 / 17.5; 6 (25) 22.2 / 18.8; 8 (18) 26.4 / 24.9; 10 (15) 24.3 /
    // 23.3; 12 (12) 25.3 / 26.4 and 26.4 / 27.7; 14 (11) 25.1 / 25.1; 16 (9) 26.7 / 28.2; 24 (6) 32.4 / 34.9; 48 (3) 38.9 / 42.2.
    const bool many_parts = units * 13 <= shares;
    const int merge_rows = many_parts ? 8 : 32, slices = (ws.rg_rows + merge_rows - 1) / merge_rows;
    const Params p = {bv, pv, ws, span, src, g->n_q_heads, g->n_kv_heads, (int)row_tiles, n_prefix, n_self, shares * ctas, ctas, Divisor(b->q_len), Divisor((int)row_tiles * ctas), Divisor(g->n_kv_heads),
                      Divisor(b->n_requests), Divisor(slices), static_cast<__nv_bfloat16*>(out), lse};
    static PerDeviceOnce configured[2];
    auto run = [&](auto kernel, int which) {
        if (configure_smem_once(configured[which], kernel, kSmemBytes) != CF_OK) return (int)CF_ERR_CUDA;
        return launch_chained(kernel, dim3((unsigned)shares), kThreads, kSmemBytes, stream, maps, p);
    };
    const int rc = ctas == 2 ? launch_attn_pair(maps, p, g->rope_layout, shares, stream)
                             : g->rope_layout == CF_ROPE_HALF ? run(attn_tc_kernel<CF_ROPE_HALF>, 0) : run(attn_tc_kernel<CF_ROPE_INTERLEAVED>, 1);
    if (rc != CF_OK) return rc;
    const unsigned blocks = (unsigned)((many_parts ? units : shares) * ctas * slices);
    const auto merge = many_parts ? attn_tc_merge_kernel<8> : attn_tc_merge_kernel<32>;
    return launch_chained(merge, dim3(blocks), kMergeThreads, 0, stream, p);
}

}  // namespace cf
