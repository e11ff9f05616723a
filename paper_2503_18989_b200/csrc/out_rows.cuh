// Output rows of the tile kernels: a thread holds consecutive columns of its own row (thread = row = TMEM lane).
// Stored as they are, every 32-byte store of a warp touches 32 rows, each its own 128-byte line, and the lines are what
// bounds the store path: 128 rows x 512 bytes take 3750 cycles to issue.  With lanes 2 k and 2 k + 1 exchanging halves of 64
// bytes first, a store touches 16 lines: 1770 cycles, shuffles included (a quad's 128 bytes 2090; rows through shared memory and
// stored whole 1650, but a longer drain).  Where a CTA has one unit only, the launch waits for just that: one request of 256 rows x
// 32 heads in 8 chunks 155 -> 151 us.  Where the CTA's other units compute meanwhile, the shuffles cost more than the
// stores (1 % of a ragged prefill batch), so there rows are stored as they are.
#pragma once
#include "hat_internal.h"
#include "tc5_ptx.cuh"

namespace hat {
namespace out_rows {

// before: 16 words of this lane's row; after: words 8 (lane & 1) .. of the even lane's row, then of the odd lane's
__device__ __forceinline__ void swap_halves(uint32_t (&v)[16], bool odd) {
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const uint32_t got = __shfl_xor_sync(0xffffffffu, odd ? v[e] : v[8 + e], 1);
        if (odd) v[e] = got; else v[8 + e] = got;
    }
}
__device__ __forceinline__ void store_32(void* p, const uint32_t* v, bool wide) {
    if (wide) {
        asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n"
                     ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
    } else {
        static_cast<uint4*>(p)[0] = make_uint4(v[0], v[1], v[2], v[3]);
        static_cast<uint4*>(p)[1] = make_uint4(v[4], v[5], v[6], v[7]);
    }
}

// Columns [col, col + N) of D of the warp's rows, scaled by each lane's `inv`, for query head h.  `at` is the lane's row in the
// output (final rows, in whichever type the call wants) or in the partial rows; rows_left counts the rows from the
// lane's own to the end of the chunk (not positive: the lane has none).  With SWAP all lanes of the warp call it.
template <int N, int D, bool SWAP>
__device__ __forceinline__ void store(const AttnArgs& a, const float (&o)[N], float inv, bool final_rows, int64_t at, int rows_left,
                                      int h, int col, int lane) {
    const bool odd = SWAP && (lane & 1);
    const int64_t pitch = (int64_t)a.plan.num_heads * D;
    if (!SWAP && rows_left <= 0) return;
    if (final_rows && a.out16 != nullptr) {
        uint16_t* dst = static_cast<uint16_t*>(a.out16) + (at - odd) * pitch + h * D + col + 16 * odd;
        const bool wide = (reinterpret_cast<uintptr_t>(a.out16) & 31) == 0;
        if constexpr (N == 16) {
            static_assert(!SWAP, "16 columns are one 32-byte store");
            uint32_t v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = pack_out16(o[2 * e] * inv, o[2 * e + 1] * inv, a.out16_bf16);
            store_32(dst, v, wide);
            return;
        }
#pragma unroll
        for (int k = 0; k + 32 <= N; k += 32) {
            uint32_t v[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) v[e] = pack_out16(o[k + 2 * e] * inv, o[k + 2 * e + 1] * inv, a.out16_bf16);
            if constexpr (SWAP) {
                swap_halves(v, odd);
                if (rows_left + odd > 0) store_32(dst + k, v, wide);
                if (rows_left + odd > 1) store_32(dst + pitch + k, v + 8, wide);
            } else {
                store_32(dst + k, v, wide);
                store_32(dst + k + 16, v + 8, wide);
            }
        }
    } else {
        float* base = final_rows ? a.out : a.part_out;
        float* dst = base + (at - odd) * pitch + h * D + col + 8 * odd;
        const bool wide = (reinterpret_cast<uintptr_t>(base) & 31) == 0;
#pragma unroll
        for (int k = 0; k < N; k += 16) {
            uint32_t v[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) v[e] = __float_as_uint(o[k + e] * inv);
            if constexpr (SWAP) {
                swap_halves(v, odd);
                if (rows_left + odd > 0) store_32(dst + k, v, wide);
                if (rows_left + odd > 1) store_32(dst + pitch + k, v + 8, wide);
            } else {
                store_32(dst + k, v, wide);
                store_32(dst + k + 8, v + 8, wide);
            }
        }
    }
}

}  // namespace out_rows
}  // namespace hat
