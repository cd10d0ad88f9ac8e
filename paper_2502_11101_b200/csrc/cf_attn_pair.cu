// Fused re-position + query-prefill attention for kv heads with more than one tile of 128 query rows (cf_attn_tc.cu: the line of key
// tiles, its shares, what they leave for the merge, the softmax): the two CTAs of a cluster work on the same key tiles with a tile of
// query rows each, as one tcgen05 CTA pair (cta_group::2, M = 256).
//
// With a CTA per tile of query rows every key tile is copied and rotated once per tile of rows (28 query heads on 4, 64 query
// tokens: four times), and rotation is as many instructions as the softmax.  A pair shares both: the B operand of a pair's MMA
// lies half in either CTA, so each copies and rotates half of a tile's keys and copies half of the dims of its values.  What
// that leaves free in shared memory takes the query tile (the A operand of Q K^T) out of tensor memory, where a fourth S buffer
// takes its place.
//   warps 0-11   three softmax warpgroups, key tiles in turn (thread = query row = TMEM lane)
//   warps 12-15  key rotation, a tile per warp: the chain from wait to arrival is 2 to 4 thousand cycles, four run side by side
//   warp 16      key loads: first to run, it finds the line and the first segment itself and loads while the others still wait
//   warp 17      value loads     warp 18  S = Q K^T     warp 19  O += P V     (18 of the first CTA issues for both; 19 of the
//                second CTA passes on that its half of V has landed)
// Measured per tile of 80 keys and 2 x 128 rows (4 x 100 documents, 28/4 heads; cycles; a CTA by itself takes 1890 for its 128 rows):
// one warp for all loads and one for all MMAs 1680, bound by the 1500 cycles the MMA warp's instructions take and by keys that
// wait for the values before them; 4 S buffers instead of 3 1620; loads and MMAs by warps of their own 1600, now bound by rotation,
// eight warps on one tile; rotation a tile per warp 1520, bound by two softmax warpgroups (2500 per tile and 500 between tiles each);
// three warpgroups 1250, where their exponentials take half of the MUFU's time.  32 keys to a softmax chunk instead of 16: no gain.
// Barriers the MMA warps wait on are those of the first CTA.  An arrival from the second is an ordinary one (release at CTA scope).
// By the letter of the memory model that does not order the second CTA's writes for a thread of the first; that it is enough here is
// an assumption about the hardware: what has to be ordered are writes to the second CTA's own shared and tensor memory, which fence.proxy.async
// and the tcgen05 fences have completed for its own SM's tensor core before the arrival is issued, and nobody else reads them.  Release at
// cluster scope costs more than pairs gain, since it waits for global stores: 2870 cycles per tile from the warps themselves, and from
// one relaying warp per barrier that stores nothing itself 89 -> 134 us a call (4 x 100 documents, 32/8 heads).  No CTA leaves, and none computes rows from scratch over its rings, before the other is done with the barriers.
#include "cf_attn_roles.cuh"

namespace cf {
namespace line {

namespace {

constexpr int kRotateWarps = 4;
constexpr int kJointTiles = 2;

struct R {
    static constexpr bool kPair = true;
    static constexpr int kSoftmaxGroups = 3;
    static constexpr int kSBuffers = 4, kKStages = 8;
    static constexpr uint32_t kColO = 0, kColS = 128, kColQ = 0;   // (the query tile lies in shared memory)
};
constexpr int kSoftmaxGroups = R::kSoftmaxGroups, kSBuffers = R::kSBuffers, kVStages = kSBuffers, kKStages = R::kKStages;
constexpr uint32_t kColO = R::kColO, kColS = R::kColS;
constexpr int kKeyHalf = kTile / 2 * 128;          // one 64-column half of a CTA's half of a key tile
constexpr int kStageBytes = 2 * kKeyHalf;          // as much as its half of the dims of a value tile
constexpr int kQueryBytes = 2 * kRowTile * 128;
constexpr int kTrigAt = (kKStages + kVStages) * kStageBytes + kQueryBytes;      // cosines and sines of the documents of the key stages
constexpr int kRingBytes = kTrigAt + kKStages * kTrigBytes;
constexpr int kRotateWarp = 4 * kSoftmaxGroups, kKeyWarp = kRotateWarp + kRotateWarps, kValueWarp = kKeyWarp + 1, kScoreWarp = kKeyWarp + 2, kPvWarp = kKeyWarp + 3;
constexpr int kThreads = 32 * (kPvWarp + 1);
static_assert(kColS + kSBuffers * kTile <= 512, "tensor memory columns");
static_assert(kStageBytes % 1024 == 0 && kKeyHalf % 1024 == 0 && kStageBytes == kTile * 128, "whole swizzle atoms");

struct Barriers {
    unsigned long long k_full[kKStages], k_ready[kKStages], k_empty[kKStages], v_empty[kVStages];
    unsigned long long s_full[kKStages], pv_ready[kKStages];      // [tile mod stages]; pv_ready: P is stored and V has landed
    unsigned long long segment[kSegRing];                               // the description of the segment is there
    unsigned long long q_ready, q_free, o_done, o_free;                 // one phase per segment
    unsigned long long ref_full[2], sum_full[2];                        // [segment parity]
    unsigned int tmem_base;
    volatile int abort_flag;
    volatile int last_segment;                     // number of the share's last segment (from 0)
    volatile int marked;                           // a row of the share has to be computed from scratch
};

struct Shared {
    Barriers bars;
    int4 meta[kMetaRing];                          // tiles in flight: length and flags, tile index or kind, first row, kv head and layer
    Segment segments[kSegRing];                    // of the share
    ShareHead head;
    Line line;
    float ref[2][kRowTile];                        // [segment parity][row]
    Requests requests;
};
constexpr int kSmemBytes = kRingBytes + (int)sizeof(Shared) + (int)sizeof(Sums<kSoftmaxGroups>) + 1024;
static_assert(kSmemBytes <= 227 * 1024 && sizeof(Shared) % 4 == 0, "shared memory of one CTA");
static_assert(sizeof(RowScratch) <= kRingBytes, "over the rings");

template <int LAYOUT>
__global__ void __launch_bounds__(kThreads, 1)
attn_pair_kernel(const __grid_constant__ StoreMaps maps, const __grid_constant__ Params p) {
    CF_PARAMS;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t k_base = smem_u32(smem), v_base = k_base + kKStages * kStageBytes, q_base = v_base + kVStages * kStageBytes;
    Shared& sh = *reinterpret_cast<Shared*>(smem + kRingBytes);
    Sums<kSoftmaxGroups>& sums = *reinterpret_cast<Sums<kSoftmaxGroups>*>(smem + kRingBytes + sizeof(Shared));
    Barriers& bars = sh.bars;
    volatile int* abort_flag = &bars.abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int group = n_q_heads / n_kv_heads, lq = bv.q_len, rows = group * lq;
    const int share = blockIdx.x >> 1, rank = blockIdx.x & 1;
    if (warp == kKeyWarp) {
        if (lane == 0) {
            auto init = [](unsigned long long* bar, int n, int count) {
                for (int i = 0; i < n; ++i) mbar_init(smem_u32(bar + i), count);
            };
            init(bars.k_full, kKStages, 1);
            init(bars.k_ready, kKStages, 2 * kRotateWarps);
            init(bars.k_empty, kKStages, 1);
            init(bars.v_empty, kVStages, 1);
            init(bars.s_full, kKStages, 1);
            // an arrival per softmax warp, one with the copy of V, one passed on by the second CTA, which waits for its copy only
            init(bars.pv_ready, kKStages, rank == 0 ? 10 : 1);
            init(bars.segment, kSegRing, 1);
            init(&bars.q_ready, 1, 2 * 8);
            init(&bars.q_free, 1, 1);
            init(&bars.o_done, 1, 1);
            init(&bars.o_free, 1, 2 * 8);
            init(bars.ref_full, 2, 4);
            init(bars.sum_full, 2, 4 * kSoftmaxGroups);
            bars.abort_flag = 0;
            bars.marked = 0;
            bars.last_segment = 0;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        if (lane < 2 * kBoxes) asm volatile("prefetch.tensormap [%0];" ::"l"(lane < kBoxes ? &maps.k[lane] : &maps.v[lane - kBoxes]) : "memory");
    } else if (warp == kScoreWarp) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&bars.tmem_base)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    chain_next();
    chain_wait();
    const Line& line = sh.line;
    if (warp == kKeyWarp) {
        // ------------------------------------------------------------------ key loads, tile descriptions
        // First the line and this share's first segment.  The other warps wait for them; this one goes on to its loads at once.
        scan_requests(bv, pv, p.n_prefix + p.n_self, sh.requests);
        __syncwarp();
        if (lane == 0) {
            const Line l = make_line(bv, ws, sh.requests, n_kv_heads, p.row_tiles, p.n_prefix, p.n_self, (int)gridDim.x >> 1);
            sh.line = l;
            const int begin = share < l.n_shares ? l.cut(share) : 0, end = share < l.n_shares ? l.cut(share + 1) : 0;
            if (begin < end) sh.segments[0] = segment_at<true>(bv, pv, ws, l, group, begin, end);
        }
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        const int x_begin = share < line.n_shares ? line.cut(share) : 0, x_end = share < line.n_shares ? line.cut(share + 1) : 0;
        if (x_begin < x_end) {
            Segment sg = sh.segments[0];
            int t = sg.t_begin, x = x_begin, segments = 1, base;
            // Descriptions of the documents' tiles base .. base + 63 of the segment, two of them per lane, loaded together: one after
            // the other they held the first loads 700 cycles apart.
            int row0[2], len[2], doc[2];
            auto fetch = [&](int half) {
                const int i = base + 32 * half + lane;
                if (i < sg.n_doc && i < sg.t_end) {
                    row0[half] = __ldg(pv.tile_row0 + sg.tile0 + i);
                    len[half] = __ldg(pv.tile_len + sg.tile0 + i);
                    doc[half] = __ldg(pv.tile_doc + sg.tile0 + i);
                }
            };
            auto start = [&]() {
                base = t;
                fetch(0);
                fetch(1);
            };
            start();
            int ks = 0, kp = 1;                                     // the first lap's waits pass: the phase before a fresh barrier's first
            for (int n = 0; n < x_end - x_begin; ++n) {
                if (t - base == 32) {
                    base = t;
                    row0[0] = row0[1];
                    len[0] = len[1];
                    doc[0] = doc[1];
                    fetch(1);
                }
                int4 m;
                const int from = t - base, tile_doc = __shfl_sync(0xffffffffu, doc[0], from);
                m.x = __shfl_sync(0xffffffffu, len[0], from);
                m.z = __shfl_sync(0xffffffffu, row0[0], from);
                m.y = sg.tile0 + t;
                if (t >= sg.n_doc + line.n_prefix) {
                    const int i = t - sg.n_doc - line.n_prefix;
                    m.y = kKindSelf - i;
                    m.z = sg.b * lq + i * kTile;
                    m.x = min(kTile, lq - i * kTile);
                } else if (t >= sg.n_doc) {
                    m.y = kKindPrefix;
                    m.z = (t - sg.n_doc) * kTile;
                    m.x = min(kTile, src.prefix_len - m.z);
                }
                const int tile_len = m.x;
                m.x |= (t == sg.t_begin ? kFirstOfSegment : 0) | (t == sg.t_end - 1 ? kLastOfSegment : 0);
                m.w = sg.kvh | (sg.layer << 20);
                if (!warp_wait(smem_u32(&bars.k_empty[ks]), kp, abort_flag)) break;
                if (lane == 0) {
                    sh.meta[n & (kMetaRing - 1)] = m;
                    const uint32_t bar = smem_u32(&bars.k_full[ks]), dst = k_base + ks * kStageBytes;
                    const int cta_keys = pair_keys(tile_len), boxes = m.y < 0 ? kBoxes / 2 : cta_keys >> 4, first = m.z + rank * cta_keys;
                    const CUtensorMap* map = m.y >= 0 ? &maps.k[boxes - 1] : m.y == kKindPrefix ? &maps.kp : &maps.ks;
                    mbar_expect_tx(bar, (boxes << 12) + (m.y >= 0 ? kTrigBytes : 0));
                    tma_load_4d(dst, map, 0, m.w & 0xfffff, first, m.w >> 20, bar);
                    tma_load_4d(dst + kKeyHalf, map, 64, m.w & 0xfffff, first, m.w >> 20, bar);
                    if (m.y >= 0) bulk_load(k_base + kTrigAt + ks * kTrigBytes, pv.trig + (size_t)tile_doc * (kD / 2), kTrigBytes, bar);
                }
                __syncwarp();
                if (++ks == kKStages) {
                    ks = 0;
                    kp ^= 1;
                }
                ++x;
                if (++t == sg.t_end && x < x_end) {
                    sg = segment_at<true>(bv, pv, ws, line, group, x, x_end);
                    t = sg.t_begin;
                    if (lane == 0) {
                        sh.segments[segments & (kSegRing - 1)] = sg;
                        mbar_arrive(smem_u32(&bars.segment[segments & (kSegRing - 1)]));
                    }
                    ++segments;
                    start();
                }
            }
            for (int i = 0; i < kKStages; ++i) {                    // what the first CTA's MMAs signal has arrived before this CTA leaves
                if (!warp_wait(smem_u32(&bars.k_empty[ks]), kp, abort_flag)) break;
                if (++ks == kKStages) {
                    ks = 0;
                    kp ^= 1;
                }
            }
            ShareHead head = {};
            if (sg.t_begin == 0 && sg.t_end < sg.n_unit) {          // sg is the share's last segment
                head.n_parts = line.share_of(x_end - sg.t_end + sg.n_unit - 1) - share + 1;
                head.lb = sg.lb;
                head.layer = sg.layer;
                head.b = sg.b;
                head.row_first = sg.kvh * rows + sg.row0;
                head.rows_here = sg.rows_here;
            }
            if (lane == 0) sh.head = head;
        }
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    } else {
        tc_fence_before();
        cluster_sync();                                             // the other CTA's barriers are there
        tc_fence_after();
    }
    const uint32_t tmem = bars.tmem_base;
    const int x_begin = share < line.n_shares ? line.cut(share) : 0, x_end = share < line.n_shares ? line.cut(share + 1) : 0;
    const int n_items = x_end - x_begin;                            // 0: this CTA has no share, its roles find nothing to do

    if (n_items == 0 || warp == kKeyWarp) {
    } else if (warp == kValueWarp) {
        // ------------------------------------------------------------------ value loads, once the description of the tile is there
        if (lane == 0) {
            int ks = 0, kp = 0, vs = 0, vp = 1;
            for (int n = 0; n < n_items; ++n) {
                if (!mbar_wait(smem_u32(&bars.k_full[ks]), kp, abort_flag) || !mbar_wait(smem_u32(&bars.v_empty[vs]), vp, abort_flag)) break;
                const int4 m = sh.meta[n & (kMetaRing - 1)];
                const uint32_t bar = smem_u32(&bars.pv_ready[ks]), dst = v_base + vs * kStageBytes;
                const int boxes = m.y >= 0 ? ((m.x & 0xff) + 15) >> 4 : kBoxes;
                const CUtensorMap* map = m.y >= 0 ? &maps.v[boxes - 1] : m.y == kKindPrefix ? &maps.vp : &maps.vs;
                mbar_expect_tx(bar, boxes << 11);
                tma_load_4d(dst, map, 64 * rank, m.w & 0xfffff, m.z, m.w >> 20, bar);
                if (++ks == kKStages) {
                    ks = 0;
                    kp ^= 1;
                }
                if (++vs == kVStages) {
                    vs = 0;
                    vp ^= 1;
                }
            }
            for (int i = 0; i < kVStages; ++i) {                    // as above
                if (!mbar_wait(smem_u32(&bars.v_empty[vs]), vp, abort_flag)) break;
                if (++vs == kVStages) {
                    vs = 0;
                    vp ^= 1;
                }
            }
        }
    } else if (warp == kPvWarp && rank == 1) {
        // ------------------------------------------------------------------ the first CTA issues; here its warp learns of V
        int j = 0, parity = 0;
        for (int it = 0; it < n_items; ++it) {
            if (!warp_wait(smem_u32(&bars.pv_ready[j]), parity, abort_flag)) break;
            if (lane == 0) mbar_arrive_first(smem_u32(&bars.pv_ready[j]));
            if (++j == kKStages) {
                j = 0;
                parity ^= 1;
            }
        }
    } else if (warp == kScoreWarp && rank == 1) {
    } else if (warp == kScoreWarp) {
        // ------------------------------------------------------------------ S = Q K^T: the warp walks, one lane issues
        const bool lead = elect_one();
        const uint32_t idesc_s0 = instr_desc(0, false, 256);
        const uint64_t bk_desc = smem_desc(k_base, 16, 1024), q_desc = smem_desc(q_base, 16, 1024);
        int j = 0, parity = 0, vs = 0, vp = 1, segments = 0;        // key stage; S buffer, which PV of the tile before in it leaves
        for (int it = 0; it < n_items; ++it) {
            if (!mma_wait<true>(smem_u32(&bars.k_ready[j]), parity, abort_flag)) break;
            const int m = sh.meta[it & (kMetaRing - 1)].x;
            if ((m & kFirstOfSegment) && !mma_wait<true>(smem_u32(&bars.q_ready), segments++ & 1, abort_flag)) break;
            if (!mma_wait<true>(smem_u32(&bars.v_empty[vs]), vp, abort_flag)) break;
            tc_fence_after();
            const uint32_t idesc = idesc_s0 | ((uint32_t)(pair_keys(m & 0xff) >> 3) << 18);
            const uint64_t b0 = bk_desc + (uint64_t)(j * (kStageBytes >> 4));
            const uint32_t s_tmem = tmem + kColS + vs * kTile;
            if (lead) {
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) {                    // 16 dims per instruction
                    const uint64_t b = b0 + (uint64_t)(((kk >> 2) * kKeyHalf + (kk & 3) * 32) >> 4);
                    umma_pair(s_tmem, q_desc + (uint64_t)(((kk >> 2) * 128 * 128 + (kk & 3) * 32) >> 4), b, idesc, kk > 0);
                }
                umma_commit<2>(smem_u32(&bars.s_full[j]));
                umma_commit<2>(smem_u32(&bars.k_empty[j]));
                if (m & kLastOfSegment) umma_commit<2>(smem_u32(&bars.q_free));
            }
            __syncwarp();
            if (++j == kKStages) {
                j = 0;
                parity ^= 1;
            }
            if (++vs == kSBuffers) {
                vs = 0;
                vp ^= 1;
            }
        }
    } else if (warp == kPvWarp) {
        // ------------------------------------------------------------------ O += P V, by a warp of its own: both chains are long
        const bool lead = elect_one();
        const uint32_t idesc_o = instr_desc(kD, true, 256);
        const uint64_t bv_desc = smem_desc(v_base, kStageBytes, 1024);
        int j = 0, parity = 0, vs = 0, segments = 0;
        for (int it = 0; it < n_items; ++it) {
            if (!mma_wait<true>(smem_u32(&bars.pv_ready[j]), parity, abort_flag)) break;
            const int m = sh.meta[it & (kMetaRing - 1)].x;
            if ((m & kFirstOfSegment) && segments > 0 && !mma_wait<true>(smem_u32(&bars.o_free), (segments - 1) & 1, abort_flag)) break;
            tc_fence_after();
            const int steps = ((m & 0xff) + 15) >> 4;               // 16 keys = 8 packed columns per instruction
            const uint64_t b0 = bv_desc + (uint64_t)(vs * (kStageBytes >> 4));
            const uint32_t p_tmem = tmem + kColS + vs * kTile, o_tmem = tmem + kColO;
            if (lead) {
                umma_ts<2>(o_tmem, p_tmem, b0, idesc_o, (m & kFirstOfSegment) ? 0u : 1u);
                for (int kk = 1; kk < steps; ++kk) umma_ts_lit<2, true>(o_tmem, p_tmem + kk * 8, b0 + (uint64_t)(kk * 128), idesc_o);
                umma_commit<2>(smem_u32(&bars.v_empty[vs]));
                if (m & kLastOfSegment) umma_commit<2>(smem_u32(&bars.o_done));
            }
            __syncwarp();
            if (m & kLastOfSegment) ++segments;
            if (++j == kKStages) {
                j = 0;
                parity ^= 1;
            }
            if (++vs == kVStages) vs = 0;
        }
    } else if (warp >= kRotateWarp) {
        // ------------------------------------------------------------------ key rotation (Eq. 5)
        // The first tiles by all warps together, which is what a short share waits for; from then on a group of warps has every
        // kGroups-th tile: the chain of wait, tables, rows, fence and arrival is long, and so several of them run side by side.
        constexpr int kGroups = 4, kGroupWarps = kRotateWarps / kGroups;
        static_assert(kKStages % kGroups == 0, "a group waits for every phase of the stages it comes to");
        const int rw = warp - kRotateWarp, chunk = lane & 7;                  // 16-byte chunk of each half row
        int stage = 0, phase = 0;
        for (int it = 0; it < n_items;) {
            const bool joint = it < kJointTiles;
            if (!joint && it < kJointTiles + kGroups && it - kJointTiles != rw / kGroupWarps) {          // on to the group's first tile
                ++it;
                if (++stage == kKStages) {
                    stage = 0;
                    phase ^= 1;
                }
                continue;
            }
            if (!warp_wait(smem_u32(&bars.k_full[stage]), phase, abort_flag)) break;
            const int2 meta = *reinterpret_cast<const int2*>(&sh.meta[it & (kMetaRing - 1)]);
            if (meta.y >= 0) {                                      // a document's tile: its table came with the keys
                const int keys = pair_keys(meta.x & 0xff), len = min(keys, (meta.x & 0xff) - rank * keys);
                rotate_rows<LAYOUT>(smem + (size_t)stage * kStageBytes, kKeyHalf, reinterpret_cast<const float4*>(smem + kTrigAt + stage * kTrigBytes), chunk,
                                    (joint ? rw : rw % kGroupWarps) * 4 + (lane >> 3), (joint ? kRotateWarps : kGroupWarps) * 4, len);
                fence_proxy_async();
            }
            __syncwarp();
            if (lane == 0) mbar_arrive_first(smem_u32(&bars.k_ready[stage]), joint ? 1 : kGroups);                    // kRotateWarps in all
            const int ahead = joint ? 1 : kGroups;
            it += ahead;
            if ((stage += ahead) >= kKStages) {
                stage -= kKStages;
                phase ^= 1;
            }
        }
    } else {
        softmax_role<R>(p, sh, sums, smem + (q_base - k_base), tmem, share, x_end, n_items);
    }

    // ---------------------------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    // the signal of the last QK^T to the query tile, which nobody else waits for, and the other CTA's last arrivals
    if (tid == 0 && n_items > 0) mbar_wait(smem_u32(&bars.q_free), bars.last_segment & 1, abort_flag);
    __syncwarp();
    cluster_sync();
    if (tid == 0) {
        ShareHead head = {};
        if (n_items > 0 && !bars.abort_flag) head = sh.head;       // (as in cf_attn_tc.cu)
        reinterpret_cast<ShareHead*>(ws.marks)[blockIdx.x] = head;
    }
    // every copy has landed and every MMA has read its operands: the rings are free
    if (bars.marked && !bars.abort_flag) marked_from_scratch<LAYOUT, true>(p, *reinterpret_cast<RowScratch*>(smem), line);
    if (bars.abort_flag) {
        // a wait expired: let the copies in flight land before the shared memory is given back
        if (tid == 0) {
            const long long t0 = clock64();
            while (clock64() - t0 < kWaitLimitCycles / 64) {}
            atomicCAS(pv.status, 0, CF_ERR_TIMEOUT);
        }
        __syncthreads();
    }
    if (warp == kScoreWarp) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
}

}  // namespace

int launch_attn_pair(const StoreMaps& maps, const Params& p, int rope_layout, int shares, cudaStream_t stream) {
    static PerDeviceOnce configured[2];
    auto run = [&](auto kernel, int which) {
        if (configure_smem_once(configured[which], kernel, kSmemBytes) != CF_OK) return (int)CF_ERR_CUDA;
        return launch_chained_clusters(kernel, dim3((unsigned)(2 * shares)), kThreads, kSmemBytes, 2, stream, maps, p);
    };
    return rope_layout == CF_ROPE_HALF ? run(attn_pair_kernel<CF_ROPE_HALF>, 0) : run(attn_pair_kernel<CF_ROPE_INTERLEAVED>, 1);
}

}  // namespace line
}  // namespace cf
