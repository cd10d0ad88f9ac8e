// Roles of the attention kernels: softmax (one query row per thread, warpgroups on the key tiles in turn) and key rotation.
#pragma once

#include "cf_attn_line.cuh"

namespace cf {
namespace line {

// Sums of a row's probabilities, of all keys and of those of documents: [segment parity][warpgroup][row].
template <int GROUPS>
struct Sums {
    float all[2][GROUPS][kRowTile], docs[2][GROUPS][kRowTile];
};

// Rows first, first + step, .. below `len` of a key tile (halves of 64 columns, `key_half` bytes apart, 128-byte swizzle) rotated in place:
// this thread's 16-byte chunk of either half (Eq. 5; fp32, one rounding).  trig: cosines and sines of the document.
template <int LAYOUT>
__device__ __forceinline__ void rotate_rows(unsigned char* base, int key_half, const float4* trig, int chunk, int first, int step, int len) {
    uint64_t c2[4], s2[4], n2[4];                       // cosines, sines and their negatives as pairs for the packed arithmetic
#pragma unroll
    for (int e = 0; e < 4; ++e) {                       // half layout: slices chunk*8 .. +7; interleaved: chunk*4 .. +3 of either half
        const float4 cs = trig[LAYOUT == CF_ROPE_HALF ? chunk * 4 + e : (e >> 1) * 16 + chunk * 2 + (e & 1)];
        c2[e] = pack_f2(cs.x, cs.z);
        s2[e] = pack_f2(cs.y, cs.w);
        n2[e] = pack_f2(-cs.y, -cs.w);
    }
    // rows 8 apart keep their swizzle phase, rows 4 apart differ in one bit of it (`step` is a multiple of either): one pointer walks
    const uintptr_t flip = (step & 4) << 4;
    unsigned char* at = base + swz(first, chunk);
#pragma unroll 2
    for (int r = first; r < len; r += step, at = reinterpret_cast<unsigned char*>(reinterpret_cast<uintptr_t>(at + step * 128) ^ flip)) {
        uint4* pa = reinterpret_cast<uint4*>(at);
        uint4* pb = reinterpret_cast<uint4*>(at + key_half);
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
}

// R: the rings of the kernel; SHARED: its shared memory (barriers, tile descriptions, segments, references).  `query`: where a pair's
// query tile lies in shared memory.  Two warpgroups load the query tile and take finished rows out.
// Where the groups do not divide the stages a warpgroup skips phases of s_full[k]: it meets tile t there and then tile t + stages *
// groups.  Its wait for tile t can still not pass on the parity of tile t - stages, whose phase is over by then: the warpgroup has seen
// S(t - groups), which was issued once PV(t - groups - buffers) had read its S buffer, and PVs are issued in order, each behind the
// softmax of its tile, which has waited for that tile's S.
template <class R, class SHARED>
__device__ __forceinline__ void softmax_role(const Params& p, SHARED& sh, Sums<R::kSoftmaxGroups>& sums, unsigned char* query, uint32_t tmem, int share, int x_end,
                                             int n_items) {
    CF_PARAMS;
    constexpr bool PAIR = R::kPair;
    static_assert(R::kKStages % R::kSoftmaxGroups == 0 || R::kKStages >= R::kSoftmaxGroups + R::kSBuffers, "the phase before a tile's is over");
    constexpr int kSoftmaxGroups = R::kSoftmaxGroups, kKStages = R::kKStages, kSBuffers = R::kSBuffers;
    constexpr uint32_t kColO = R::kColO, kColQ = R::kColQ, kColS = R::kColS;
    const Line& line = sh.line;
    auto& bars = sh.bars;
    volatile int* abort_flag = &bars.abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int group = n_q_heads / n_kv_heads, lq = bv.q_len, rows = group * lq, rows_total = n_q_heads * lq;
    auto arrive_mma = [&](uint32_t bar) {                           // barriers that the warps of the MMAs wait on
        if (PAIR) mbar_arrive_first(bar);
        else mbar_arrive(bar);
    };
    const int w = warp >> 2, r = tid & 127;                     // warpgroup; row of the tile = TMEM lane
    const uint32_t lane_tmem = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const uint64_t scale2 = pack_f2(src.scale_log2, src.scale_log2);
    const uint32_t bar_s_full = smem_u32(bars.s_full), bar_pv_ready = smem_u32(bars.pv_ready);
    int k = w, phase = 0;                                       // this warpgroup's next tile, mod stages, and its parity
    int it0 = 0;                                                // tiles before the current segment
    int leader = 0;                                             // warpgroup that has its first tile
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
        if (more && (kSoftmaxGroups == 2 || w < 2)) {
            // the query tile of the segment goes into tensor memory, half of every row by each of two warpgroups (before
            // the epilogue of the last segment)
            const bool active = (warp & 3) * 32 < sg.rows_here;
            const int row = PAIR ? min(sg.row0 + r, rows - 1) : sg.row0 + min(r, sg.rows_here - 1), g = row / lq, j = row - g * lq;
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
            if (PAIR) {                                         // .. or into shared memory, where a pair has room
                unsigned char* at = query + w * 128 * 128;
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    *reinterpret_cast<uint4*>(at + swz(r, i)) = make_uint4(qw[4 * i], qw[4 * i + 1], qw[4 * i + 2], qw[4 * i + 3]);
                fence_proxy_async();
            } else if (active) {
                tc_fence_after();
                tmem_st16_from<0>(lane_tmem + kColQ + w * 32, qw);
                tmem_st16_from<16>(lane_tmem + kColQ + w * 32 + 16, qw);
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                tc_fence_before();
            }
            __syncwarp();
            if (lane == 0) arrive_mma(smem_u32(&bars.q_ready));
        }
        if (seg > 0) {
            // ---- end of a segment: the two sums meet, each warpgroup takes half of the columns of O
            const int par = (seg - 1) & 1;
            sums.all[par][w][r] = l_run;
            sums.docs[par][w][r] = l_docs;
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bars.sum_full[par]));
            ok = warp_wait(smem_u32(&bars.sum_full[par]), ((seg - 1) >> 1) & 1, abort_flag) && (w >= 2 || warp_wait(smem_u32(&bars.o_done), par, abort_flag));
            if (!ok) break;
            if (kSoftmaxGroups == 2 || w < 2) {
                tc_fence_after();
                const Segment& done = sh.segments[(seg - 1) & (kSegRing - 1)];
                const bool whole = done.t_end - done.t_begin == done.n_unit;
                const int row = done.row0 + r;
                float l_all = sums.all[par][0][r], d_all = sums.docs[par][0][r];
#pragma unroll
                for (int x = 1; x < kSoftmaxGroups; ++x) {
                    l_all += sums.all[par][x][r];
                    d_all += sums.docs[par][x][r];
                }
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
                                    parts_code(blockIdx.x, line.share_of(x_end - done.t_end + done.n_unit - 1) - share + 1);
                        } else {
                            ws.row_lse2[at] = marked ? __int_as_float(0x7fffffff) : ref + log2f(d_all);
                            if (lse) lse[at] = (ref + log2f(l_all)) * kLn2;
                        }
                        if (marked) bars.marked = 1;
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) arrive_mma(smem_u32(&bars.o_free));
            }
        }
        if (!more) {
            if constexpr (PAIR)
                if (tid == 0) bars.last_segment = seg - 1;
            break;
        }
        // ---- the tiles of the segment
        const int n = sg.t_end - sg.t_begin, par = seg & 1;
        const bool active = (warp & 3) * 32 < sg.rows_here, row_valid = r < sg.rows_here;
        const int q_index = (sg.row0 + r) % lq;                 // position of this row's token in the query
        float* tile_lse2 = ws.tile_lse2 + (size_t)sg.layer * ws.max_tiles * rows_total + (size_t)sg.kvh * rows + sg.row0 + r;
        bool have_ref = false, seen_extra = false;
        l_run = l_docs = 0.f;
        for (int i = w >= leader ? w - leader : w - leader + kSoftmaxGroups; i < n; i += kSoftmaxGroups) {
            ok = warp_wait(bar_s_full + k * 8, phase, abort_flag);
            if (!ok) break;
            tc_fence_after();
            const int4 meta = sh.meta[(it0 + i) & (kMetaRing - 1)];
            const int len = meta.x & 0xff, n_chunks = (len + 15) >> 4;
            // keys this row may see: a whole tile of a document or of the prefix, the query tokens up to its own (causal
            // mask, footnote to Eq. 1)
            const int vis = meta.y <= kKindSelf ? min(len, q_index + 1 - (kKindSelf - meta.y) * kTile) : len;
            const uint32_t s_addr = lane_tmem + kColS + (k >= kSBuffers ? k - kSBuffers : k) * kTile;
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
                if (lane == 0) arrive_mma(bar_pv_ready + k * 8);
                if (!(tile_sum < kSumLimit)) tile_sum = __int_as_float(0x7fffffff);     // out of range: the row is marked
                l_run += tile_sum;
                if (meta.y >= 0 && row_valid) tile_lse2[(size_t)meta.y * rows_total] = ref + __log2f(tile_sum);
            } else if (lane == 0) {
                arrive_mma(bar_pv_ready + k * 8);
            }
            k += kSoftmaxGroups;
            if (k >= kKStages) {
                k -= kKStages;
                phase ^= 1;
            }
        }
        if (ok && !have_ref) ok = warp_wait(smem_u32(&bars.ref_full[par]), (seg >> 1) & 1, abort_flag);   // every phase is waited for
        if (!have_ref && ok) ref = sh.ref[par][r];
        if (!seen_extra) l_docs = l_run;
        it0 += n;
        leader = (leader + n) % kSoftmaxGroups;
    }
}

}  // namespace line
}  // namespace cf
