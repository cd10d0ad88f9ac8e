// Eight query rows against sixteen keys at a time by one warp, with mma.sync: what the tensor-core kernels use for rows that left
// the range of their fixed softmax reference.  Such rows are few and scattered and no reason to start a pipeline of roles; what
// counts is that one row does not become a chain of thousands of memory latencies, and that many rows share the loads of their
// keys.  (One row by one warp, key after key, took 0.4 to 1.3 us a key: one row in a call of 8000 keys cost 3 ms, seventy times
// the call, a head of such rows 10 ms.)  The keys and values of the next step are on their way into shared memory (cp.async)
// while the warp computes the current one from registers; with plain loads, whose targets have to find room beside the sums of
// the rows, a step takes a third longer.
//
// Lane = 4 g + t (g = lane / 4, t = lane % 4).  Its row of the group is g; its dims of queries and keys are 32 c + 8 t .. + 7 for
// c = 0 .. 3, so that both halves of a rotary slice (p and p + 64, or neighbours) sit in one lane.
//   S = Q K^T  m16n8k16, rows = queries (eight of sixteen), columns = keys; the contraction index is permuted alike on both sides
//   O^T += V^T P^T  m16n8k16, rows = dims, columns = queries; S's accumulators are P^T's fragments
// Probabilities enter as the sum of two bf16 values (2^-17 off), the sums are fp32; running maximum, as many keys as come.
#pragma once

#include "cf_common.cuh"

namespace cf {
namespace rows {

constexpr int kDim = 128;
constexpr int kGroupRows = 8, kStepKeys = 16;

__device__ __forceinline__ void mma16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t shared_at(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// Sixteen bytes of shared memory, read here and not earlier.
__device__ __forceinline__ void read16(const void* p, uint32_t (&w)[4]) {
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(shared_at(p)) : "memory");
}

// The queries of a group.  Rows 320 bytes apart: the pieces that eight lanes read together fall on all banks.
struct alignas(16) Queries {
    __nv_bfloat16 row[kGroupRows][kDim + 32];
    // Row r of the group, by sixteen lanes (piece = 0 .. 15).
    __device__ __forceinline__ void put(int r, int piece, const __nv_bfloat16* from) {
        *reinterpret_cast<uint4*>(&row[r][8 * piece]) = __ldg(reinterpret_cast<const uint4*>(from + 8 * piece));
    }
};

// A warp's step on its way: sixteen keys and sixteen values.  The pitches keep the fragments of either free of bank conflicts.
struct alignas(16) Stage {
    __nv_bfloat16 k[kStepKeys][kDim + 32], v[kStepKeys][kDim + 8];
};
static_assert(sizeof(Stage) % 16 == 0 && (kDim + 32) * 2 % 16 == 0 && (kDim + 8) * 2 % 16 == 0, "16-byte pieces");
// Copies rows first .. first + 15 (rows `pitch` elements apart, of which n exist; the others repeat the last one) by a warp.
template <int PITCH>
__device__ __forceinline__ void copy_step(__nv_bfloat16 (&to)[kStepKeys][PITCH], const __nv_bfloat16* first, size_t pitch, int n) {
    const int lane = threadIdx.x & 31, piece = 8 * (lane & 15);
#pragma unroll 2
    for (int i = 0; i < kStepKeys / 2; ++i) {
        const int r = 2 * i + (lane >> 4);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(shared_at(&to[r][piece])), "l"(first + (size_t)min(r, n - 1) * pitch + piece) : "memory");
    }
}
__device__ __forceinline__ void copies_end() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// All groups of copies but the youngest one have landed, for the whole warp.
__device__ __forceinline__ void copies_wait() {
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncwarp();
}

// The lane's fragments of a step's keys.
struct Keys {
    uint32_t k[2][4][4];
    __device__ __forceinline__ void read(const Stage& st) {
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int c = 0; c < 4; ++c) read16(&st.k[8 * j + (lane >> 2)][8 * (lane & 3) + 32 * c], k[j][c]);
    }
    // Eq. 5, rounded to the storage type; trig: cosines and sines of the document.
    template <int LAYOUT>
    __device__ __forceinline__ void rotate(const float2* trig) {
        const int t = threadIdx.x & 3;
        auto lo = [](uint32_t w) { return __uint_as_float(w << 16); };
        auto hi = [](uint32_t w) { return __uint_as_float(w & 0xffff0000u); };
        auto both = [](float a, float b) {
            const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
            return *reinterpret_cast<const uint32_t*>(&h);
        };
        float a0, b0, a1, b1;
        if (LAYOUT == CF_ROPE_HALF) {
#pragma unroll
            for (int c = 0; c < 2; ++c)
#pragma unroll
                for (int e = 0; e < 4; ++e) {                       // slices 32 c + 8 t + 2 e and the next one
                    const float4 cs = *reinterpret_cast<const float4*>(trig + 32 * c + 8 * t + 2 * e);
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        uint32_t &x = k[j][c][e], &y = k[j][c + 2][e];
                        rotate_pair(lo(x), lo(y), cs.x, cs.y, a0, b0);
                        rotate_pair(hi(x), hi(y), cs.z, cs.w, a1, b1);
                        x = both(a0, a1);
                        y = both(b0, b1);
                    }
                }
        } else {
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int e = 0; e < 4; ++e) {                       // slice 16 c + 4 t + e
                    const float2 cs = trig[16 * c + 4 * t + e];
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        rotate_pair(lo(k[j][c][e]), hi(k[j][c][e]), cs.x, cs.y, a0, b0);
                        k[j][c][e] = both(a0, b0);
                    }
                }
        }
    }
};

// Running softmax of a group: `m` and the sums belong to row g (the sums to this lane's share of the keys), o to rows 2 t and
// 2 t + 1: o[4 h + i][0], [2] are dims 64 h + 8 g + 2 i and the next of row 2 t, [1], [3] those of row 2 t + 1.
struct Group {
    float o[8][4], m, l;
    uint32_t p[2], rest[2];                                         // probabilities of the step: bf16, and what bf16 leaves of them
    __device__ __forceinline__ void clear() {
        m = -INFINITY;
        l = 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) o[i][e] = 0.f;
    }
    // Row g sees the first `visible` keys of the step.  Returns the lane's sum of the step's probabilities; `alpha`: what sums
    // kept beside l have to be scaled by.
    __device__ __forceinline__ float scores(const Queries& queries, const Keys& keys, int visible, float scale_log2, float& alpha) {
        const int lane = threadIdx.x & 31, t = lane & 3;
        // a short accumulation per chunk, joined in fp32, since mma.sync truncates what it adds: log-sum-exps near 200 were up to
        // 4.2e-5 off with one chain of eight, 3.0e-5 this way, 2.8e-5 with fused multiply-adds (one unit of the last place: 1.5e-5)
        float s[2][2] = {};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            uint32_t q[4];
            read16(&queries.row[lane >> 2][8 * t + 32 * c], q);
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                float part[4] = {};
                mma16816(part, q[0], 0u, q[1], 0u, keys.k[j][c][0], keys.k[j][c][1]);
                mma16816(part, q[2], 0u, q[3], 0u, keys.k[j][c][2], keys.k[j][c][3]);
                s[j][0] += part[0];
                s[j][1] += part[1];
            }
        }
        float e[4] = {s[0][0] * scale_log2, s[0][1] * scale_log2, s[1][0] * scale_log2, s[1][1] * scale_log2};
#pragma unroll
        for (int i = 0; i < 4; ++i)                                 // keys 2 t, 2 t + 1, 2 t + 8, 2 t + 9
            if (2 * t + (i & 1) + 8 * (i >> 1) >= visible) e[i] = -INFINITY;
        float top = fmaxf(fmaxf(e[0], e[1]), fmaxf(e[2], e[3]));
        top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, 1));
        top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, 2));
        top = fmaxf(top, m);
        const float ref = top > -INFINITY ? top : 0.f;              // no key seen yet: nothing to scale, all probabilities 0
        alpha = exp2f(m - ref);
        m = top;
        const float a0 = __shfl_sync(0xffffffffu, alpha, 8 * t), a1 = __shfl_sync(0xffffffffu, alpha, 8 * t + 4);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            o[i][0] *= a0;
            o[i][1] *= a1;
            o[i][2] *= a0;
            o[i][3] *= a1;
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            e[2 * i] = exp2f(e[2 * i] - ref);
            e[2 * i + 1] = exp2f(e[2 * i + 1] - ref);
            const __nv_bfloat162 h = __floats2bfloat162_rn(e[2 * i], e[2 * i + 1]);
            const float2 f = __bfloat1622float2(h);
            const __nv_bfloat162 r = __floats2bfloat162_rn(e[2 * i] - f.x, e[2 * i + 1] - f.y);
            p[i] = *reinterpret_cast<const uint32_t*>(&h);
            rest[i] = *reinterpret_cast<const uint32_t*>(&r);
        }
        const float sum = (e[0] + e[1]) + (e[2] + e[3]);
        l = fmaf(l, alpha, sum);
        return sum;
    }
    __device__ __forceinline__ void values(const Stage& st) {
        const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint32_t v[4][4];                                       // keys 2 t, 2 t + 1, 2 t + 8, 2 t + 9
#pragma unroll
            for (int j = 0; j < 4; ++j) read16(&st.v[2 * t + (j & 1) + 8 * (j >> 1)][8 * g + 64 * h], v[j]);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t a0 = __byte_perm(v[0][i], v[1][i], 0x5410), a1 = __byte_perm(v[0][i], v[1][i], 0x7632);
                const uint32_t a2 = __byte_perm(v[2][i], v[3][i], 0x5410), a3 = __byte_perm(v[2][i], v[3][i], 0x7632);
                mma16816(o[4 * h + i], a0, a1, a2, a3, p[0], p[1]);
                mma16816(o[4 * h + i], a0, a1, a2, a3, rest[0], rest[1]);
            }
        }
    }
};

// A lane's share of a sum of row g made whole.
__device__ __forceinline__ float over_keys(float x) {
    x += __shfl_xor_sync(0xffffffffu, x, 1);
    return x + __shfl_xor_sync(0xffffffffu, x, 2);
}

// The n-th (from 0) set bit of `set`, the first one where there are fewer; `set` is not 0.
__device__ __forceinline__ int nth_bit(unsigned set, int n) {
    for (unsigned s = set; s; s &= s - 1)
        if (n-- == 0) return __ffs((int)s) - 1;
    return __ffs((int)set) - 1;
}
// The lowest kGroupRows set bits.
__device__ __forceinline__ unsigned next_group(unsigned set) {
    unsigned rest = set;
    for (int i = 0; i < kGroupRows; ++i) rest &= rest - 1;
    return set ^ rest;
}

}  // namespace rows
}  // namespace cf
