// The softmax of a 128-key tile on its way from scores to weights, in tensor memory (thread = row = TMEM lane).
//
// What bounds the tile kernels is not the exponentials alone but the instructions around them: the loops of the roles run side by side
// and share the SM's instruction caches, a softmax loop unrolled over 128 keys is 10 KB of code, and the thread that issues the
// MMAs waits for its own few instructions behind it (690 to 790 cycles for 8 MMAs of 64, 150 to 220 for a look at a barrier that has long completed).  So
// the code is kept small and the scores are read twice: once, all of them, for the row's maximum, and again 32 at a time in a loop that
// is not unrolled; packed fp32 arithmetic and three-operand maxima halve the instructions.  The weights of 32 keys (16 columns of 16-bit pairs, for
// bf16 16 more with what their rounding dropped) take the columns of the keys' own scores, so that nothing unread is overwritten.
// Measured on the one-CTA kernel, us a call, unrolled with the scores in registers / this: 30 ragged chunks x 32 heads, fp16, back to back 502 / 478
// (64 columns 302 / 290, bf16 431 / 361), 30 chunks of 32 to 128 rows bf16 104 / 92, a prompt of 2048 in eight calls 128 / 120.  In the CTA-pair
// kernel, whose loops are smaller, the same form is slower (mixed 13B-shaped batch 747 / 760).
#pragma once
#include "tc5_ptx.cuh"

namespace hat {
namespace softmax_tile {

// column of the 16 weights that MMA step ks (16 keys) multiplies, relative to the tile's first; the remainders are 16 columns on
__host__ __device__ constexpr uint32_t weight_col(int ks) { return (ks >> 1) * 32 + (ks & 1) * 8; }

// Scores of keys past `lim` become -inf.  For the warps with such a key: the few tiles at the end of a row's range.
template <int N>
__device__ __forceinline__ void mask(uint32_t scores, int lim) {
    if (!__any_sync(0xffffffffu, lim < N - 1)) return;
#pragma unroll 1
    for (int c = 0; c < N; c += 32) {
        uint32_t x[32];
        tc5::tmem_ld32(scores + c, x);
        tc5::tmem_ld_wait();
#pragma unroll
        for (int k = 0; k < 32; ++k) x[k] = k <= lim - c ? x[k] : 0xff800000u;
        tc5::tmem_st32(scores + c, x);
    }
    tc5::tmem_st_wait();
}

template <int N>
__device__ __forceinline__ float row_max(uint32_t scores) {
    float s[N], m[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};      // four independent chains
#pragma unroll
    for (int c = 0; c < N; c += 32) tc5::tmem_ld32(scores + c, reinterpret_cast<uint32_t*>(s) + c);
    tc5::tmem_ld_wait();
#pragma unroll
    for (int k = 0; k < N; k += 8) {
#pragma unroll
        for (int v = 0; v < 4; ++v) asm("max.f32 %0, %0, %1, %2;\n" : "+f"(m[v]) : "f"(s[k + 2 * v]), "f"(s[k + 2 * v + 1]));
    }
    return fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3]));
}

// exp2(score * scale + offset), its sum, and its 16-bit form in TMEM
template <bool BF16>
struct Weigh {
    uint64_t scale, offset, sum[4];
    __device__ __forceinline__ Weigh(float sc, float off) : scale(tc5::f2_pack(sc, sc)), offset(tc5::f2_pack(off, off)), sum{0, 0, 0, 0} {}
    // 32 keys; dst: the column of the first one's score
    __device__ __forceinline__ void keys32(const uint32_t (&x)[32], uint32_t dst) {
        uint32_t p[16], rest[16];
#pragma unroll
        for (int k = 0; k < 32; k += 2) {
            float e0, e1;
            tc5::f2_unpack(tc5::f2_fma(tc5::f2_pack(__uint_as_float(x[k]), __uint_as_float(x[k + 1])), scale, offset), e0, e1);
            e0 = tc5::fast_exp2(e0); e1 = tc5::fast_exp2(e1);
            const uint64_t e = tc5::f2_pack(e0, e1);
            sum[(k >> 1) & 3] = tc5::f2_add(sum[(k >> 1) & 3], e);
            p[k / 2] = tc5::pack2<BF16>(e0, e1);
            if constexpr (BF16) {
                float r0, r1;
                tc5::f2_unpack(tc5::f2_sub(e, tc5::f2_pack(__uint_as_float(p[k / 2] << 16), __uint_as_float(p[k / 2] & 0xffff0000u))), r0, r1);
                rest[k / 2] = tc5::pack2<true>(r0, r1);
            }
        }
        tc5::tmem_st16(dst, p);
        if constexpr (BF16) tc5::tmem_st16(dst + 16, rest);
    }
    // a tile of 128 keys whose first 32 scores are on their way to `first`
    __device__ __forceinline__ void keys128(uint32_t (&first)[32], uint32_t scores) {
        uint32_t next[32];
        tc5::tmem_ld_wait();
#pragma unroll 1
        for (int c = 0; c < 128; c += 64) {
            tc5::tmem_ld32(scores + c + 32, next);
            keys32(first, scores + c);
            tc5::tmem_ld_wait();
            tc5::tmem_ld32(scores + 64, first);      // the second time unused: nothing is on its way where the loop comes round
            keys32(next, scores + c + 32);
            tc5::tmem_ld_wait();
        }
    }
    __device__ __forceinline__ float total() const {
        float a, b;
        tc5::f2_unpack(tc5::f2_add(tc5::f2_add(sum[0], sum[1]), tc5::f2_add(sum[2], sum[3])), a, b);
        return a + b;
    }
};

}  // namespace softmax_tile
}  // namespace hat
