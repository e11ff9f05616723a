// KV append inside the tile kernels.
//
// A call that appends hands the tile kernels k_new / v_new: the tiles of a unit that hold chunk positions are loaded from
// there instead of from the pool (8-row boxes of the packed rows into the same places, hence the same bits in the result),
// so that nothing has to be appended before the kernel starts.  The pool is written on the way: one unit per (request, K/V
// head, page) stores the page from the ring slot it was loaded into (TMA store, no registers, no second read).  A page that
// the chunk shares with the prefix (prefix not a multiple of 16) is gathered row by row, and a page that the chunk shares or
// does not fill is stored row by row.  A kernel of its own in front takes 34 us on 30 ragged chunks (218 MB) and 2 to 4 us on a
// single 256-row chunk; append_is_apart (hat_api.cu) says where that is the cheaper way all the same.
#pragma once
#include "hat_internal.h"
#include "tc5_ptx.cuh"

namespace hat {
namespace tile_append {

// Where the keys of a page come from and go to; key0 = first key of the page.
struct Chunk {
    int P, C, row_base, hk;
    __device__ __forceinline__ bool fresh(int key0) const { return key0 >= P; }                                // all of it from k_new / v_new
    __device__ __forceinline__ bool whole(int key0) const { return key0 >= P && key0 + kPageSize <= P + C; }    // stored by TMA
    __device__ __forceinline__ bool partly(int key0) const { return key0 + kPageSize > P && key0 < P + C && !whole(key0); }
};

// The page that holds both prefix and chunk rows, gathered row by row into its place in a tile: COLS columns from col0 on;
// rows of 8 are group_bytes apart, column halves 1 KiB.  Asynchronous copies of the calling warp.
template <int COLS>
__device__ __forceinline__ void gather_edge(const AttnArgs& a, const Chunk& ck, const void* pool, const void* fresh, int head_dim, int col0,
                                            int page, int key0, uint32_t dst, uint32_t group_bytes, int lane) {
#pragma unroll 4
    for (int idx = lane; idx < 16 * (COLS / 8); idx += 32) {
        const int r = idx / (COLS / 8), c = idx % (COLS / 8), key = key0 + r;
        const bool in = key < ck.P + ck.C;
        const uint16_t* src = static_cast<const uint16_t*>(pool);
        if (key < ck.P) src += (int64_t)page * a.cache.stride_page + (int64_t)r * a.cache.stride_token + (int64_t)ck.hk * a.cache.stride_head + col0 + c * 8;
        else if (in) src = static_cast<const uint16_t*>(fresh) + ((int64_t)(ck.row_base + key - ck.P) * a.plan.num_kv_heads + ck.hk) * head_dim + col0 + c * 8;
        tc5::cp_async16(dst + (r >> 3) * group_bytes + (c >> 3) * 1024 + (r & 7) * 128 + (((c & 7) ^ (r & 7)) << 4), src, in);
    }
}
// The calling warp's copies have landed and may be read by the tensor core.
__device__ __forceinline__ void gathered() {
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    __syncwarp();
}

// The chunk rows of a page that is not whole: from k_new / v_new to the pool.
template <int COLS>
__device__ __forceinline__ void store_rows(const AttnArgs& a, const Chunk& ck, void* pool, const void* fresh, int head_dim, int col0, int page,
                                           int key0, int lane) {
    const int first = max(ck.P - key0, 0), last = min(ck.P + ck.C - key0, (int)kPageSize);   // rows of the page
    for (int idx = lane; idx < (last - first) * (COLS / 8); idx += 32) {
        const int r = first + idx / (COLS / 8), c = idx % (COLS / 8);
        const uint4 x = __ldg(reinterpret_cast<const uint4*>(static_cast<const uint16_t*>(fresh) +
                                                             ((int64_t)(ck.row_base + key0 + r - ck.P) * a.plan.num_kv_heads + ck.hk) * head_dim + col0) + c);
        *reinterpret_cast<uint4*>(static_cast<uint16_t*>(pool) + (int64_t)page * a.cache.stride_page + (int64_t)r * a.cache.stride_token +
                                  (int64_t)ck.hk * a.cache.stride_head + col0 + c * 8) = x;
    }
}

// Ring slots the warp's stores still read must not be refilled.
__device__ __forceinline__ void stores_read() { asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory"); }
__device__ __forceinline__ void stores_done() { asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory"); }
__device__ __forceinline__ void stores_commit() { asm volatile("cp.async.bulk.commit_group;\n" ::: "memory"); }

}  // namespace tile_append
}  // namespace hat
