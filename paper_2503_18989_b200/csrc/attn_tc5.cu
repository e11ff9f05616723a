// Prefill-chunk attention on the 5th-generation tensor cores (tcgen05 + TMEM), fed by TMA.
//
// Persistent kernel, one CTA per SM.  A work unit = up to 256 query rows (two 128-row query tiles) of one request x
// one head x one key range; CTAs draw units (longest first) from a global counter until none is left.  Both query
// tiles of a unit use the same K/V tiles in shared memory, and while one tile's softmax runs the tensor pipe works
// for the other.  Roles:
//   warp 0      draws the next unit and publishes it to the other roles; TMA producer: the unit's Q tiles, then K
//               and V tiles of 128 keys (8 pages, a box each, 128-byte swizzle) into a two-slot K ring
//               and a three-slot V ring, completion on mbarriers.  It runs ahead across units: the next unit's Q and
//               first K/V tiles are already landing while the current unit's last tiles and its output are processed
//   warp 1      one thread issues tcgen05.mma: S_t = Q_t K^T for query tile t, then O_t += P_t V with P read
//               from TMEM; tcgen05.commit signals the consumers and frees the ring slots.  Owns the TMEM allocation
//   warps 2-5, 6-9   one warpgroup per query tile, thread = query row = TMEM lane: tcgen05.ld of S, scale/mask/online
//               softmax in registers (reference maximum only moved when it grows by more than 2^8, so O is rarely
//               rescaled), P written back to TMEM as the 16-bit A operand; at the end of a unit O is pulled into
//               registers (which frees the accumulator for the next unit), divided by l and stored with the lse
// TMEM columns: S0 [0,128) S1 [128,256) O0 [256,384) O1 [384,512).  P_t(j) overwrites S_t(j) in place (softmax_tile.cuh);
// S_t(j+1) is issued after P_t V(j) by the same thread, and
// tcgen05 executes one thread's MMAs in issue order, so no extra barrier guards the reuse.
// A unit of at most 128 rows uses both column pairs for the SAME query tile: two chains over alternating key tiles,
// merged by the first chain's warpgroup when the unit ends (see Unit::split).
// Every wait is bounded (about a second by default); a wait that gives up sets the plan's status word, raises a
// CTA-wide abort flag that all other waits observe, and the CTA still frees its TMEM and exits normally.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "hat_internal.h"
#include "tma_desc.h"
#include "tc5_ptx.cuh"
#include "out_rows.cuh"
#include "softmax_tile.cuh"
#include "tile_append.cuh"

namespace hat {
namespace {
using namespace tc5;

constexpr int kRows = 128;      // query rows per CTA (MMA M)
constexpr int kKeys = 128;      // keys per tile (MMA N of S, K extent of PV)
constexpr int kStagesK = 2;     // ring slots for K tiles
constexpr int kStagesV = 3;     // ring slots for V tiles (V is requested later in a step than K, so it gets the deeper ring)
// one K or V tile, or the Q tile: 128 rows of head_dim 16-bit values (32 KiB at head_dim 128, 16 KiB at 64), stored as
// head_dim / 64 slabs of 64 columns
template <int D> constexpr uint32_t tile_bytes() { return kKeys * D * 2; }
constexpr uint32_t kSlabBytes = kKeys * 64 * 2;          // 16 KiB: 64 columns of 128 rows
// K and V tiles: 8-row groups (head_dim / 64 blocks of 1 KiB) one after the other; a page is two groups
template <int D> constexpr uint32_t group_bytes() { return 8 * D * 2; }
template <int D> constexpr uint32_t page_bytes() { return 16 * D * 2; }
constexpr float kRescaleThreshold = 8.0f;                // log2 units

struct __align__(8) Barriers {
    uint64_t q_full, q_empty;
    uint64_t k_full[kStagesK], k_empty[kStagesK];
    uint64_t v_full[kStagesV], v_empty[kStagesV];
    uint64_t s_full[2], p_ready[2], o_done[2], o_free[2];   // per query tile
    uint64_t unit_full[2], unit_empty[2];                   // two-slot queue of work units, producer -> other roles
    uint64_t x_ready, x_ready0;                             // split units: (reference maximum, row sum) of chain 1 are in xchg, chain 0's too
    uint64_t peer_ready[8];                                 // kHalves: the softmax warp of the same number in the other CTA has its rows ready
    uint64_t drain;
    volatile long long wait_cycles;                         // bound of every wait below (see waits_begin)
    uint32_t tmem_base;
    volatile int abort_flag;
    volatile int unit_slot[2];                              // unit index, or -1 when the work has run out
    float2 xchg[kRows];                                     // split units: per row, chain 1's reference maximum and row sum
};
template <int D> constexpr uint32_t smem_bytes() { return 1024 /*alignment slack*/ + tile_bytes<D>() * (2 + kStagesK + kStagesV) + sizeof(Barriers); }
static_assert(smem_bytes<128>() <= 227 * 1024, "shared memory of one CTA");
constexpr int kThreads = 320;   // producer warp, MMA warp, two softmax warpgroups

// Bounded wait.  Returns false if the wait gave up or another role already did.  It is inlined some thirty times, so it holds no more
// than it must: the CTA reports to the status word once, at its end (see "Code size" at the kernel).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, Barriers* b) {
    if (mbar_try(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try(bar, parity))
        if (b->abort_flag || clock64() - t0 > b->wait_cycles) {
            b->abort_flag = 1;
            return false;
        }
    return true;
}

// The same for a barrier the cluster's other CTA arrives on, acquiring what it wrote before.
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t* bar, uint32_t parity, Barriers* b) {
    const long long t0 = clock64();
    while (!mbar_try_cluster(bar, parity))
        if (b->abort_flag || clock64() - t0 > b->wait_cycles) {
            b->abort_flag = 1;
            return false;
        }
    return true;
}

// What every role needs to know about a unit; all of them decode it the same way.
struct Unit {
    int h, hk, r, P, C, row_base, row0, kv_begin, kv_end, part;   // h: query head, hk = h / G: the K/V head it reads
    int nq;       // query tiles in use (1 or 2)
    int n_all;    // key tiles of the range
    int n_q0;     // key tiles query tile 0 can see (tile 0 does not see the keys past its own last row)
    // A unit with a single query tile would leave the second accumulator pair and warpgroup idle and the tensor
    // pipe waiting through every softmax.  It runs as two chains instead: chain t takes key tiles t, t+2, t+4, ... with
    // the same Q tile, and the two partial results (disjoint key sets) are merged when the unit ends.
    bool split;
    int n_t0, n_t1;   // key tiles of chain (or query tile) 0 and 1
    __device__ __forceinline__ int n_t(int t) const { return t == 0 ? n_t0 : n_t1; }
    // key tile of step s of chain t
    __device__ __forceinline__ int tile_of(int t, int s) const { return split ? 2 * s + t : s; }
};
__device__ __forceinline__ Unit decode_unit(const AttnArgs& a, const WorkItem* __restrict__ items, int unit) {
    const uint32_t e = __ldg(a.plan.tile_units + unit);      // item | head << 16
    const int4* __restrict__ rec = reinterpret_cast<const int4*>(items + (e & 0xffffu));
    const int4 lo = __ldg(rec), hi = __ldg(rec + 1);
    Unit u;
    u.h = (int)(e >> 16);
    u.hk = u.h / a.plan.group;
    u.r = lo.x; u.row0 = lo.y; u.kv_begin = lo.z; u.kv_end = lo.w;
    u.part = hi.x; u.P = hi.y; u.C = hi.z; u.row_base = hi.w;
    u.nq = min(u.C - u.row0, a.plan.tile_rows) > kRows ? 2 : 1;
    u.n_all = (u.kv_end - u.kv_begin + kKeys - 1) / kKeys;
    const int end0 = min(u.kv_end, u.P + u.row0 + kRows);
    u.n_q0 = u.nq == 1 ? u.n_all : max(0, (end0 - u.kv_begin + kKeys - 1) / kKeys);
    u.split = u.nq == 1;
    u.n_t0 = u.split ? (u.n_all + 1) / 2 : u.n_q0;
    u.n_t1 = u.split ? u.n_all / 2 : (u.nq == 2 ? u.n_all : 0);
    return u;
}

// How the units lie on the CTAs.  A template parameter because the softmax loop's registers are tight: as a branch, the other
// output form cost it 2 %.
//   kMany    CTAs draw units
//   kOne     no CTA has more than one unit (128 columns; rows of 64 store as fast as they are)
//   kHalves  the same, and the CTAs of a cluster of two have the two key ranges of one tile of at most 128 rows: they merge them
//            through each other's shared memory, a quarter of the columns to a warpgroup, instead of through global memory and a launch
//            (one request of 256 rows x 32 heads, us a call: prefix 768
//            19.4 -> 13.4, 1792 23.9 -> 17.9, 4000 38.9 -> 32.3)
enum Form { kMany, kOne, kHalves };
// Code size: the loops of the roles run side by side and have to share the instruction cache; what else the kernel holds, executed or
// not, costs misses.  Calls that append nothing therefore get a kernel without the code for it (APPEND = false), and a wait is
// as short as it can be.  One call of 30 ragged chunks x 32 heads, fp16, nothing appended: 124 KB of code 417 us, 97 KB 387 us (64 columns:
// 358 -> 327 us); instruction cache misses of 12 chunks 1.0 M -> 0.6 M, 133 -> 124 us.
template <bool BF16, int kD, int FORM, bool APPEND>
__global__ void __launch_bounds__(kThreads, 1)
attn_tc5_kernel(AttnArgs a, const WorkItem* __restrict__ items, int total_units, int32_t* work_counter,
                const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_k_new,
                const __grid_constant__ CUtensorMap map_v_new, int fold) {
    constexpr bool ONE = FORM != kMany;
    static_assert(FORM != kOne || kD == 128, "rows of 64 columns store as fast as they are");
    constexpr uint32_t kTileBytes = tile_bytes<kD>();
    constexpr int kSlabs = kD / 64;                              // 64-column slabs of a Q tile
    constexpr uint32_t kGroupBytes = group_bytes<kD>(), kPageBytes = page_bytes<kD>();
    extern __shared__ unsigned char smem_raw[];
    // 1024-byte alignment: the swizzle pattern and the matrix descriptors assume it
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    unsigned char* q_tiles = smem;                               // 2 x 32 KiB
    unsigned char* k_ring = smem + 2 * kTileBytes;
    unsigned char* v_ring = k_ring + kStagesK * kTileBytes;
    Barriers* bars = reinterpret_cast<Barriers*>(v_ring + kStagesV * kTileBytes);

    const int H = a.plan.num_heads;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int32_t* status = a.plan.status;

    if (threadIdx.x == 0) {
        mbar_init(&bars->q_full, 1); mbar_init(&bars->q_empty, 1);
        for (int s = 0; s < kStagesK; ++s) { mbar_init(&bars->k_full[s], 1); mbar_init(&bars->k_empty[s], 1); }
        for (int s = 0; s < kStagesV; ++s) { mbar_init(&bars->v_full[s], 1); mbar_init(&bars->v_empty[s], 1); }
        for (int s = 0; s < 2; ++s) {
            mbar_init(&bars->s_full[s], 1);
            mbar_init(&bars->p_ready[s], 4);                     // one arrival per softmax warp
            mbar_init(&bars->o_done[s], 1);
            mbar_init(&bars->o_free[s], 4);
            mbar_init(&bars->unit_full[s], 1);
            mbar_init(&bars->unit_empty[s], 1 + 8);              // the MMA thread and every softmax warp
        }
        mbar_init(&bars->x_ready, 4);
        mbar_init(&bars->x_ready0, 4);
        for (int w = 0; w < 8; ++w) mbar_init(&bars->peer_ready[w], 1);
        mbar_init(&bars->drain, 1);
        bars->abort_flag = 0;
        bars->wait_cycles = a.overlap ? a.wait_cycles : kNotYet;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\n" ::"r"(smem_u32(&bars->tmem_base)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (FORM == kHalves) {
        cluster_arrive();                                        // the other CTA's barriers are initialised
        cluster_wait();
    }
    tc_fence_after();
    const uint32_t tmem = bars->tmem_base;
    pdl_launch_dependents();
    if (warp == 0) {
        // ------------------------------------------------------------------ unit fetch + TMA producer
        // Lane pg + 8 g moves page pg of a tile: one box (g = 0), or its two 8-row groups where the pool's strides fold neither
        // way and for rows of k_new / v_new.  What this warp does per tile is close to what a tile costs the tensor core, so
        // the tiles that hold nothing of the chunk have a loop of their own with no more than it must hold (ring positions are stepped, page
        // ids fetched a tile ahead): a prompt of 2048 in eight calls 119.4 / 117.4 us, 30 ragged chunks 467 / 459.
        const long long since = clock64();
        // the previous kernel's end, once what the plan's own arrays hold has been read
        auto front_ended = [&]() {
            if (a.overlap) return;
            pdl_wait();
            if (lane == 0) waits_begin(&bars->wait_cycles, since, a.wait_cycles);
        };
        const int pg = lane & 7, grp = lane >> 3;
        const int boxes = fold ? 8 : 16;                         // lanes that move pool pages
        const int c1 = 8 * grp, s3 = fold == 1 ? 1 : 0, s4 = fold == 2 ? 1 : 0;
        const uint32_t lane_off = pg * kPageBytes + grp * kGroupBytes;
        int sk = 0, sv = 0;                                      // ring slots of the next tile
        uint32_t pk = 1, pv = 1;                                 // parities of their "empty" barriers: the first round passes at once
        bool withhold = a.withhold;                              // self test: the first V tile never arrives, its consumers give up
        if constexpr (FORM == kHalves) withhold = withhold && cluster_ctarank() == 0;   // (and the other CTA waits for its rows in vain)
        bool ok = true;
        // the tile before the one being requested, if this unit is the one that appends its pages: stored from its ring slots
        bool owes = false, o_whole = false, stored = false;      // stored: a slot may still be read by its store
        int o_sk = 0, o_sv = 0, o_page = 0, o_hk = 0;
        uint32_t o_pk = 0, o_pv = 0;
        auto pay = [&]() {
            if (!owes) return;
            owes = false;
            ok = mbar_wait(&bars->k_full[o_sk], o_pk, bars) && mbar_wait(&bars->v_full[o_sv], o_pv, bars);
            ok = __all_sync(0xffffffffu, ok);
            if (ok && o_whole) {
                tma_store_5d(&map_k, smem_u32(k_ring) + o_sk * kTileBytes + lane_off, 0, c1, 0, o_hk << s3, o_page << s4);
                tma_store_5d(&map_v, smem_u32(v_ring) + o_sv * kTileBytes + lane_off, 0, c1, 0, o_hk << s3, o_page << s4);
            }
            tile_append::stores_commit();
            stored = true;
        };
        auto step = [&]() {
            if (++sk == kStagesK) { sk = 0; pk ^= 1; }
            if (++sv == kStagesV) { sv = 0; pv ^= 1; }
        };
        for (int un = 0; ok; ++un) {
            const int slot = un & 1;
            if (un >= 2) {
                ok = __all_sync(0xffffffffu, mbar_wait(&bars->unit_empty[slot], ((un >> 1) - 1) & 1, bars));
                if (!ok) break;
            }
            int unit = 0;
            if (lane == 0) {
                // a CTA's first unit is its own number: nothing to wait for
                if (un == 0 && a.static_first) unit = (int)blockIdx.x;
                else if (ONE) unit = -1;
                else unit = atomicAdd(work_counter, 1) + (a.static_first ? (int)gridDim.x : 0);
                if (unit >= total_units) unit = -1;
                bars->unit_slot[slot] = unit;
                mbar_arrive(&bars->unit_full[slot]);             // release: the slot is written before the arrival
            }
            unit = __shfl_sync(0xffffffffu, unit, 0);
            if (unit < 0) {
                // a grid that joins another one may find nothing left: its end still stands for the end of what precedes it
                if (un == 0) front_ended();
                break;
            }
            const Unit u = decode_unit(a, items, unit);
            const int32_t* __restrict__ table = a.plan.block_table + (int64_t)u.r * a.plan.max_pages;
            const int total_pages = (u.kv_end - u.kv_begin + kPageSize - 1) / kPageSize, page0 = u.kv_begin / kPageSize;
            auto page_of = [&](int j) -> int {
                const int at = 8 * j + pg;
                return at < total_pages
                           ? HAT_IN_RANGE(__ldg(table + HAT_IN_RANGE(page0 + at, a.plan.max_pages, status)), a.plan.num_pages, status) : 0;
            };
            int page = page_of(0);
            // Q tiles: the previous unit's last S must have read the old ones
            if (un > 0) {
                ok = __all_sync(0xffffffffu, mbar_wait(&bars->q_empty, (un - 1) & 1, bars));
                if (!ok) break;
            } else {
                front_ended();
            }
            if (lane == 0) mbar_expect_tx(&bars->q_full, u.nq * kTileBytes);
            if (lane < kSlabs * u.nq)       // lane = kSlabs * (query tile) + (column half)
                tma_load_3d(smem_u32(q_tiles) + (lane / kSlabs) * kTileBytes + (lane % kSlabs) * kSlabBytes, &map_q, (lane % kSlabs) * 64, u.h,
                            u.row_base + u.row0 + (lane / kSlabs) * kRows, &bars->q_full);
            // tiles [0, n_plain) hold nothing of the chunk, or the call does not append
            const int n_plain = APPEND ? min(u.n_all, max(0, u.P - u.kv_begin) / kKeys) : u.n_all;
            const int c3 = u.hk << s3;
            const tile_append::Chunk ck{u.P, u.C, u.row_base, u.hk};
            // of the units that read a chunk page, the last row block of the group's first query head appends it
            const bool appends = APPEND && u.h == u.hk * a.plan.group && u.row0 + a.plan.tile_rows >= u.C;
            int j = 0;
#pragma unroll 1
            for (; j < n_plain; ++j) {
                const int npages = min(8, total_pages - 8 * j);
                const int page_next = page_of(j + 1), c4 = page << s4;
                const bool pool = lane < boxes && pg < npages;
                HAT_CHECK(sk < kStagesK && sv < kStagesV, status);
                if (APPEND && stored) { tile_append::stores_read(); stored = false; }
                ok = __all_sync(0xffffffffu, mbar_wait(&bars->k_empty[sk], pk, bars));
                if (!ok) break;
                if (lane == 0) mbar_expect_tx(&bars->k_full[sk], npages * kPageBytes);
                if (pool) tma_load_5d(smem_u32(k_ring) + sk * kTileBytes + lane_off, &map_k, 0, c1, 0, c3, c4, &bars->k_full[sk]);
                ok = __all_sync(0xffffffffu, mbar_wait(&bars->v_empty[sv], pv, bars));
                if (!ok) break;
                if (!withhold) {
                    if (lane == 0) mbar_expect_tx(&bars->v_full[sv], npages * kPageBytes);
                    if (pool) tma_load_5d(smem_u32(v_ring) + sv * kTileBytes + lane_off, &map_v, 0, c1, 0, c3, c4, &bars->v_full[sv]);
                }
                if (APPEND && owes) {                             // the previous unit's last tile
                    pay();
                    if (!ok) break;
                }
                withhold = false;
                page = page_next;
                step();
            }
            if (!ok) break;
            if (!APPEND) continue;
            // tiles with chunk positions
#pragma unroll 1
            for (; j < u.n_all; ++j) {
                const int npages = min(8, total_pages - 8 * j);
                const int page_next = page_of(j + 1), c4 = page << s4;
                const uint32_t k_dst = smem_u32(k_ring) + sk * kTileBytes, v_dst = smem_u32(v_ring) + sv * kTileBytes;
                // in a tile with chunk positions: pages of the chunk alone come from k_new / v_new; a page with both prefix and
                // chunk rows is gathered and completes the barriers last
                const int kb = u.kv_begin + j * kKeys, key0 = kb + pg * kPageSize, pe = (u.P - kb) / kPageSize;
                const bool edge = u.P > kb && u.P % kPageSize != 0 && pe < npages;
                const bool fresh = lane < 16 && pg < npages && ck.fresh(key0);
                const bool pool = lane < boxes && pg < npages && !ck.fresh(key0) && !(edge && pg == pe);
                const uint32_t bytes = (npages - (edge ? 1 : 0)) * kPageBytes;
                const int row = u.row_base + key0 - u.P + 8 * grp;
                HAT_CHECK(sk < kStagesK && sv < kStagesV, status);
                if (APPEND && stored) { tile_append::stores_read(); stored = false; }
                ok = __all_sync(0xffffffffu, mbar_wait(&bars->k_empty[sk], pk, bars));
                if (!ok) break;
                if (lane == 0) { if (edge) mbar_expect_only(&bars->k_full[sk], bytes); else mbar_expect_tx(&bars->k_full[sk], bytes); }
                if (pool) tma_load_5d(k_dst + lane_off, &map_k, 0, c1, 0, c3, c4, &bars->k_full[sk]);
                if (fresh) tma_load_4d(k_dst + lane_off, &map_k_new, 0, row, 0, u.hk, &bars->k_full[sk]);
                ok = __all_sync(0xffffffffu, mbar_wait(&bars->v_empty[sv], pv, bars));
                if (!ok) break;
                if (!withhold) {
                    if (lane == 0) { if (edge) mbar_expect_only(&bars->v_full[sv], bytes); else mbar_expect_tx(&bars->v_full[sv], bytes); }
                    if (pool) tma_load_5d(v_dst + lane_off, &map_v, 0, c1, 0, c3, c4, &bars->v_full[sv]);
                    if (fresh) tma_load_4d(v_dst + lane_off, &map_v_new, 0, row, 0, u.hk, &bars->v_full[sv]);
                }
                if constexpr (APPEND) {
                    if (edge) {
                        const int at = __shfl_sync(0xffffffffu, page, pe);
#pragma unroll 1
                        for (int kv = 0; kv < 2; ++kv)
                            tile_append::gather_edge<kD>(a, ck, kv ? a.cache.v_pool : a.cache.k_pool, kv ? a.v_new : a.k_new, kD, 0, at, kb + pe * kPageSize,
                                                         (kv ? v_dst : k_dst) + pe * kPageBytes, kGroupBytes, lane);
                        tile_append::gathered();
                        if (lane == 0) { mbar_arrive(&bars->k_full[sk]); if (!withhold) mbar_arrive(&bars->v_full[sv]); }
                    }
                    pay();                                       // the tile before, or the previous unit's last
                    if (!ok) break;
                    if (appends && !withhold) {
                        owes = true;
                        o_sk = sk; o_sv = sv; o_pk = pk ^ 1; o_pv = pv ^ 1; o_page = page; o_hk = u.hk;
                        o_whole = lane < boxes && pg < npages && ck.whole(key0);
                        // the pages that are not whole, row by row
                        for (uint32_t left = __ballot_sync(0xffffffffu, lane < 8 && pg < npages && ck.partly(key0)); left; left &= left - 1) {
                            const int from = __ffs(left) - 1, at = __shfl_sync(0xffffffffu, page, from);
#pragma unroll 1
                            for (int kv = 0; kv < 2; ++kv)
                                tile_append::store_rows<kD>(a, ck, kv ? a.v_dst : a.k_dst, kv ? a.v_new : a.k_new, kD, 0, at, kb + from * kPageSize, lane);
                        }
                    }
                }
                withhold = false;
                page = page_next;
                step();
            }
        }
        // The last CTA whose producer draws no more leaves the unit counter at zero for the next call, which then needs no
        // memset in front of it.  work_counter[1] counts them.  (Every draw has returned, so no fence is needed; at the CTA's end, behind
        // one, this held up the next kernel of the stream by about 1 us.)
        if (!ONE && a.tail_reset && lane == 0 && atomicAdd(work_counter + 1, 1) == (int)gridDim.x - 1) {
            work_counter[0] = 0;
            work_counter[1] = 0;
        }
        if constexpr (APPEND) {
            if (ok) pay();
            tile_append::stores_done();
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer (one thread)
        if (lane == 0) {
            constexpr uint32_t fmt = BF16 ? 1u : 0u;
            constexpr uint32_t idesc_s = make_idesc(fmt, 0, kRows, kKeys);   // Q (K-major) x K (K-major)
            constexpr uint32_t idesc_o = make_idesc(fmt, 1, kRows, kD);      // P (TMEM)    x V (MN-major)
            // matrix descriptors of Q tile 0 and of slot 0 of each ring, built once
            const uint64_t q_desc0 = smem_desc(smem_u32(q_tiles), 16, 1024);
            const uint64_t k_desc0 = smem_desc(smem_u32(k_ring), 16, kGroupBytes);
            const uint64_t v_desc0 = smem_desc(smem_u32(v_ring), 1024, kGroupBytes);
            bool ok = true;
            int kt_base = 0;                          // K/V tiles of the units before this one
            // bit t, for tile or chain t: parity of the next completion of p_ready[t] and of o_free[t]; O_t holds a finished unit that its
            // warpgroup may still be reading
            uint32_t p_par = 0, f_par = 0, o_busy = 0;
            for (int un = 0; ok; ++un) {
                const int slot = un & 1;
                ok = mbar_wait(&bars->unit_full[slot], (un >> 1) & 1, bars);
                if (!ok) break;
                const int unit = bars->unit_slot[slot];
                mbar_arrive(&bars->unit_empty[slot]);
                if (unit < 0) break;
                const Unit u = decode_unit(a, items, unit);
                ok = mbar_wait(&bars->q_full, un & 1, bars);
                if (!ok) break;
                // the two kinds of unit get their own copy of the issue loop: every instruction of this thread counts
                auto run_unit = [&](auto split_tag) {
                    constexpr bool SPLIT = decltype(split_tag)::value;
                    int k_ready = -1, v_ready = -1;       // last K / V tile of this unit known to have landed
                    // S_t(s) = Q K(j)^T into TMEM columns [128 t, 128 t + 128), j = the key tile of step s of chain / tile t
                    auto issue_s = [&](int qt, int sidx) {
                        const int j = SPLIT ? 2 * sidx + qt : sidx;
                        const int kt = kt_base + j, st = kt % kStagesK;
                        if (k_ready < j) {
                            ok = mbar_wait(&bars->k_full[st], (kt / kStagesK) & 1, bars);
                            k_ready = j;
                            if (!ok) return;
                        }
                        // descriptors of the first 16 columns; the others differ in the address field only
                        const uint64_t qd = q_desc0 + (uint64_t)((SPLIT ? 0 : qt) * (kTileBytes >> 4));
                        const uint64_t kd = k_desc0 + (uint64_t)(st * (kTileBytes >> 4));
                        tc_fence_after();
#pragma unroll
                        for (int ks = 0; ks < kD / 16; ++ks) {
                            // 16 columns = 32 bytes inside a row of 64; the next 64 columns are 16 KiB (Q) or 1 KiB (K) on
                            const uint32_t q_off = ((ks >> 2) * kSlabBytes + (ks & 3) * 32) >> 4, k_off = ((ks >> 2) * 1024 + (ks & 3) * 32) >> 4;
                            mma_ss(tmem + qt * 128, qd + q_off, kd + k_off, idesc_s, ks > 0);
                        }
                        tc_commit(&bars->s_full[qt]);
                        if (SPLIT || qt == u.nq - 1) {
                            tc_commit(&bars->k_empty[st]);                       // the last reader of this K tile
                            if (j == u.n_all - 1) tc_commit(&bars->q_empty);     // and the unit's last read of the Q tiles
                        }
                    };
                    // O_t (+)= P_t V(j); P sits in the columns S_t was computed in
                    auto issue_pv = [&](int qt, int sidx) {
                        const int j = SPLIT ? 2 * sidx + qt : sidx;
                        const int kt = kt_base + j, st = kt % kStagesV;
                        if (v_ready < j) {
                            ok = mbar_wait(&bars->v_full[st], (kt / kStagesV) & 1, bars);
                            v_ready = j;
                            if (!ok) return;
                        }
                        if (sidx == 0 && (o_busy >> qt) & 1) {
                            // the accumulator still holds the previous unit: wait until its rows are in registers
                            ok = mbar_wait(&bars->o_free[qt], (f_par >> qt) & 1, bars);
                            f_par ^= 1u << qt;
                            o_busy &= ~(1u << qt);
                            if (!ok) return;
                        }
                        ok = mbar_wait(&bars->p_ready[qt], (p_par >> qt) & 1, bars);
                        p_par ^= 1u << qt;
                        if (!ok) return;
                        tc_fence_after();
                        const uint64_t vd = v_desc0 + (uint64_t)(st * (kTileBytes >> 4));
                        const uint32_t tp = tmem + qt * 128, to = tmem + 256 + qt * 128;
                        HAT_CHECK((to & 0xffffu) + 128 <= 512 && (tp & 0xffffu) + 128 <= 256, status);
#pragma unroll
                        for (int ks = 0; ks < kKeys / 16; ++ks) {
                            // 16 keys = one page; inside it 64-column blocks 1 KiB apart (leading), then the next 8-key group
                            const uint64_t vdesc = vd + (uint64_t)((ks * kPageBytes) >> 4);
                            mma_ts(to, tp + softmax_tile::weight_col(ks), vdesc, idesc_o, (sidx > 0) || (ks > 0));
                            if constexpr (BF16) mma_ts(to, tp + softmax_tile::weight_col(ks) + 16, vdesc, idesc_o, true);
                        }
                        if (sidx == u.n_t(qt) - 1) tc_commit(&bars->o_done[qt]);      // before that S(next) tells
                        if (SPLIT || qt == u.nq - 1) tc_commit(&bars->v_empty[st]);
                    };
                    if constexpr (ONE) {
                        // one copy of the products for both tiles or chains: code that a CTA of one unit meets cold (eight calls of one request
                        // 117 / 114 us; where CTAs draw units the addresses that depend on the tile cost more, 64 columns bf16 361 / 390)
#pragma unroll 1
                        for (int sidx = -1; sidx < max(u.n_t0, u.n_t1) && ok; ++sidx) {
#pragma unroll 1
                            for (int qt = 0; qt < 2 && ok; ++qt) {
                                const int n = u.n_t(qt);
                                if (sidx >= n) continue;
                                if (sidx >= 0) issue_pv(qt, sidx);
                                if (ok && sidx + 1 < n) issue_s(qt, sidx + 1);
                            }
                        }
                        return;
                    }
                    if (u.n_t0 > 0) issue_s(0, 0);
                    if (ok && u.n_t1 > 0) issue_s(1, 0);
                    for (int sidx = 0; sidx < max(u.n_t0, u.n_t1) && ok; ++sidx) {
                        // tile 0's P V, then at once its next S: the tensor pipe works on them while tile 1's softmax runs
                        if (sidx < u.n_t0) {
                            issue_pv(0, sidx);
                            if (ok && sidx + 1 < u.n_t0) issue_s(0, sidx + 1);
                        }
                        if (ok && sidx < u.n_t1) {
                            issue_pv(1, sidx);
                            if (ok && sidx + 1 < u.n_t1) issue_s(1, sidx + 1);
                        }
                    }
                };
                if (u.split) run_unit(std::true_type{}); else run_unit(std::false_type{});
                // a unit in which a tile had no keys leaves that tile's earlier hand-over pending
                if (u.n_t0 > 0) o_busy |= 1u;
                if (u.n_t1 > 0) o_busy |= 2u;
                kt_base += u.n_all;
            }
            if (!ok) {
                // gave up: let the MMAs already issued finish (bounded) before TMEM is released
                tc_commit(&bars->drain);
                const long long t0 = clock64();
                while (!mbar_try(&bars->drain, 0) && clock64() - t0 < bars->wait_cycles) { }
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------------ softmax / correction / output
        const int qt = (warp - 2) >> 2;                     // query tile of this warpgroup
        const int quarter = warp & 3;                       // TMEM lanes this warp may touch
        const int t = quarter * 32 + lane;                  // query row inside the tile = TMEM lane
        const uint32_t lane_sel = (uint32_t)(quarter * 32) << 16;
        const uint32_t tm_s = tmem + qt * 128 + lane_sel, tm_o = tmem + 256 + qt * 128 + lane_sel;
        const int wg_tid = (int)threadIdx.x - 64 - qt * 128;
        const float sc = a.scale_log2;
        int kt_base = 0;                                    // K/V tiles of the units before this one
        int s_cnt = 0, o_cnt = 0, x_cnt = 0;                // completions of s_full[qt] / o_done[qt] / x_ready consumed so far
        bool ok = true;
        for (int un = 0; ok; ++un) {
            const int slot = un & 1;
            ok = __all_sync(0xffffffffu, mbar_wait(&bars->unit_full[slot], (un >> 1) & 1, bars));
            if (!ok) break;
            const int unit = bars->unit_slot[slot];
            __syncwarp();                                    // every lane has read the slot
            if (lane == 0) mbar_arrive(&bars->unit_empty[slot]);
            if (unit < 0) break;
            const Unit u = decode_unit(a, items, unit);
            if (qt < u.nq || u.split) {
                const int n_mine = u.n_t(qt);
                const int i_row = u.row0 + (u.split ? 0 : qt * kRows) + t;   // row inside the chunk
                const int last_key = min(u.P + i_row, u.kv_end - 1);
                float m_used = -INFINITY, l = 0.f;           // in units of scale_log2
                for (int sidx = 0; sidx < n_mine; ++sidx) {
                    const int j = u.tile_of(qt, sidx);       // key tile of this step
                    const int kb = u.kv_begin + j * kKeys;
                    ok = __all_sync(0xffffffffu, mbar_wait(&bars->s_full[qt], s_cnt & 1, bars));
                    ++s_cnt;
                    if (!ok) break;
                    tc_fence_after();
                    softmax_tile::mask<kKeys>(tm_s, last_key - kb);   // keys 0 .. last_key - kb of this tile are visible to this row
                    // raw maximum (the scale is positive, so it commutes with max)
                    const float mx = softmax_tile::row_max<kKeys>(tm_s) * sc;
                    uint32_t first[32];
                    tmem_ld32(tm_s, first);
                    // move the reference maximum only when it grew by more than the threshold
                    float alpha = 1.f;
                    bool rescale = false;
                    if (mx > m_used + kRescaleThreshold) {
                        alpha = (m_used == -INFINITY) ? 0.f : fast_exp2(m_used - mx);
                        rescale = (m_used != -INFINITY);
                        m_used = mx;
                    }
                    softmax_tile::Weigh<BF16> weigh(sc, (m_used == -INFINITY) ? 0.f : -m_used);
                    weigh.keys128(first, tm_s);
                    l = l * alpha + weigh.total();

                    // O may only be rescaled once the previous P V product has finished: it was issued, by the same thread, before
                    // this step's S, which is here
                    if (__any_sync(0xffffffffu, rescale)) {
#pragma unroll 1
                        for (int c = 0; c < kD / 32; ++c) {
                            uint32_t o[32];
                            tmem_ld32(tm_o + c * 32, o);
                            tmem_ld_wait();
#pragma unroll
                            for (int k = 0; k < 32; ++k) o[k] = __float_as_uint(__uint_as_float(o[k]) * alpha);
                            tmem_st32(tm_o + c * 32, o);
                        }
                    }
                    tmem_st_wait();
                    // a range that ends inside this tile: V rows past the range were not loaded (or hold stale
                    // slots); zero them so that 0 * garbage cannot produce NaN (both warpgroups may do it: same zeros)
                    if (kb + kKeys > u.kv_end) {
                        const int kt = kt_base + j;
                        ok = __all_sync(0xffffffffu, mbar_wait(&bars->v_full[kt % kStagesV], (kt / kStagesV) & 1, bars));
                        if (!ok) break;
                        unsigned char* vt = v_ring + (kt % kStagesV) * kTileBytes;
                        const int first = u.kv_end - kb;
                        constexpr int kVecs = kD / 8;                              // 16-byte vectors per row
                        for (int idx = wg_tid; idx < (kKeys - first) * kVecs; idx += 128) {
                            const int row = first + idx / kVecs, part = idx % kVecs;
                            *reinterpret_cast<uint4*>(vt + (row >> 3) * kGroupBytes + (part >> 3) * 1024 + (row & 7) * 128 + (part & 7) * 16) = make_uint4(0, 0, 0, 0);
                        }
                        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                    }
                    // one arrival per warp: every lane's P is in TMEM (wait::st) and fenced before the warp meets
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bars->p_ready[qt]);
                }
                if (!ok) break;
                // ---- output of the unit
                if (n_mine > 0) {                            // uniform over the warpgroup
                    ok = __all_sync(0xffffffffu, mbar_wait(&bars->o_done[qt], o_cnt & 1, bars));
                    ++o_cnt;
                    if (!ok) break;
                    tc_fence_after();
                }
                if constexpr (ONE) {
                    // 64 columns at a time, stored with the lanes' halves exchanged (out_rows.cuh).  A split unit: the chains (disjoint keys)
                    // are merged, weights 2^(m_t - m), sums and accumulators add up; each chain's warpgroup does half of the columns
                    const bool have0 = u.split || n_mine > 0, have1 = u.split && u.n_t1 > 0;
                    float w0 = 1.f, w1 = 0.f;
                    if (u.split) {
                        float2* x0 = reinterpret_cast<float2*>(q_tiles + kTileBytes);   // the second query tile's place is free
                        (qt == 0 ? x0 : bars->xchg)[t] = make_float2(m_used, l);
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(qt == 0 ? &bars->x_ready0 : &bars->x_ready);
                        ok = __all_sync(0xffffffffu, mbar_wait(qt == 0 ? &bars->x_ready : &bars->x_ready0, 0, bars));
                        if (!ok) break;
                        tc_fence_after();
                        const float2 c0 = x0[t], c1 = bars->xchg[t];
                        m_used = fmaxf(c0.x, c1.x);
                        w0 = (c0.x == -INFINITY) ? 0.f : fast_exp2(c0.x - m_used);
                        w1 = (c1.x == -INFINITY) ? 0.f : fast_exp2(c1.x - m_used);
                        l = c0.y * w0 + c1.y * w1;
                    }
                    const int64_t orow = u.part < 0 ? u.row_base + i_row : u.part + (i_row - u.row0);
                    HAT_CHECK(i_row >= u.C || (orow >= 0 && orow < (u.part < 0 ? (int64_t)a.plan.total_rows : a.part_rows)), status);
                    const uint32_t tm_a = u.split ? tmem + 256 + lane_sel : tm_o;
                    auto load32 = [&](float* o, int c0) {
                        if (have0) {
                            tmem_ld32(tm_a + c0, reinterpret_cast<uint32_t*>(o));
                            tmem_ld_wait();
                        } else {
#pragma unroll
                            for (int k = 0; k < 32; ++k) o[k] = 0.f;
                        }
                        if (have1) {
                            uint32_t o1[32];
                            tmem_ld32(tm_a + 128 + c0, o1);      // the second chain's accumulator: next 128 columns
                            tmem_ld_wait();
#pragma unroll
                            for (int k = 0; k < 32; ++k) o[k] = o[k] * w0 + __uint_as_float(o1[k]) * w1;
                        }
                    };
                    if constexpr (FORM == kHalves) {
                        // this CTA finishes a quarter of the columns per warpgroup; the other half of the warpgroup's half goes where the Q tile was
                        // (every product that read it has ended), the maximum and sum behind chain 0's
                        constexpr int HALF = kD / 2, QUARTER = kD / 4;
                        const uint32_t rank = cluster_ctarank();
                        float o[HALF], mine[QUARTER];
#pragma unroll
                        for (int c = 0; c < HALF; c += 32) load32(o + c, HALF * qt + c);
                        float4* give = reinterpret_cast<float4*>(q_tiles) + qt * (QUARTER / 4 * kRows) + t;
                        float2* ml = reinterpret_cast<float2*>(q_tiles + kTileBytes) + (1 + qt) * kRows + t;
#pragma unroll
                        for (int k = 0; k < QUARTER / 4; ++k) {
                            const float* lo = o + 4 * k; const float* hi = o + QUARTER + 4 * k;
                            give[k * kRows] = rank == 0 ? make_float4(hi[0], hi[1], hi[2], hi[3]) : make_float4(lo[0], lo[1], lo[2], lo[3]);
#pragma unroll
                            for (int e = 0; e < 4; ++e) mine[4 * k + e] = rank == 0 ? lo[e] : hi[e];
                        }
                        *ml = make_float2(m_used, l);
                        __syncwarp();
                        if (lane == 0) mbar_arrive_cluster(map_to_cta(smem_u32(&bars->peer_ready[warp - 2]), rank ^ 1u));
                        ok = __all_sync(0xffffffffu, mbar_wait_cluster(&bars->peer_ready[warp - 2], 0, bars));
                        if (!ok) break;
                        const float2 other = ld_cluster_f2(map_to_cta(smem_u32(ml), rank ^ 1u));
                        const uint32_t from = map_to_cta(smem_u32(give), rank ^ 1u);
                        const float m_new = fmaxf(m_used, other.x);
                        const float wm = (m_used == -INFINITY) ? 0.f : fast_exp2(m_used - m_new);
                        const float wo = (other.x == -INFINITY) ? 0.f : fast_exp2(other.x - m_new);
                        // the same in both CTAs, whichever piece is its own
                        l = __fadd_rn(__fmul_rn(l, wm), __fmul_rn(other.y, wo));
                        m_used = m_new;
                        const float inv = l > 0.f ? 1.f / l : 0.f;
#pragma unroll
                        for (int k = 0; k < QUARTER / 4; ++k) {
                            const float4 v = ld_cluster_f4(from + k * kRows * 16);
                            mine[4 * k] = mine[4 * k] * wm + v.x * wo; mine[4 * k + 1] = mine[4 * k + 1] * wm + v.y * wo;
                            mine[4 * k + 2] = mine[4 * k + 2] * wm + v.z * wo; mine[4 * k + 3] = mine[4 * k + 3] * wm + v.w * wo;
                        }
                        out_rows::store<QUARTER, kD, kD == 128>(a, mine, inv, true, orow, u.C - i_row, u.h, HALF * qt + QUARTER * (int)rank, lane);
                        if (i_row < u.C && qt == 0 && rank == 0) a.lse[orow * H + u.h] = l > 0.f ? (m_used + log2f(l)) * 0.6931471805599453f : -INFINITY;
                    } else {
                        const float inv = l > 0.f ? 1.f / l : 0.f;
#pragma unroll 1
                        for (int c0 = 0; c0 < kD; c0 += 32) {
                            if (u.split && c0 >> 6 != qt) continue;
                            float o[32];
                            load32(o, c0);
                            out_rows::store<32, kD, true>(a, o, inv, u.part < 0, orow, u.C - i_row, u.h, c0, lane);
                        }
                        if (i_row < u.C && !(u.split && qt == 1))
                            (u.part < 0 ? a.lse : a.part_lse)[orow * H + u.h] = l > 0.f ? (m_used + log2f(l)) * 0.6931471805599453f : -INFINITY;
                    }
                } else if (u.split && qt == 1) {
                    // second chain of a split unit: its accumulator is complete; publish the row's reference maximum
                    // and sum, the first chain's warpgroup reads the accumulator itself (same TMEM lanes) and stores
                    if (n_mine > 0) {
                        bars->xchg[t] = make_float2(m_used, l);
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&bars->x_ready);
                    }
                } else {
                    // 32 columns at a time, one copy of the code for all (see softmax_tile.cuh: 30 chunks of 32 to 128 rows x 32 heads, fp16, 82 / 74 us,
                    // bf16 97 / 83; 30 ragged chunks 459 / 451); with the last ones in registers the accumulator is handed back
                    const bool have1 = u.split && u.n_t1 > 0;
                    float w0 = 1.f, w1 = 0.f;
                    if (have1) {
                        // the second chain (disjoint keys): weights 2^(m_t - m), sums and accumulators add up
                        ok = __all_sync(0xffffffffu, mbar_wait(&bars->x_ready, x_cnt & 1, bars));
                        ++x_cnt;
                        if (!ok) break;
                        tc_fence_after();
                        const float2 other = bars->xchg[t];
                        const float m_new = fmaxf(m_used, other.x);
                        w0 = (m_used == -INFINITY) ? 0.f : fast_exp2(m_used - m_new);
                        w1 = (other.x == -INFINITY) ? 0.f : fast_exp2(other.x - m_new);
                        l = l * w0 + other.y * w1;
                        m_used = m_new;
                    }
                    const float inv = l > 0.f ? 1.f / l : 0.f;
                    const int64_t orow = u.part < 0 ? u.row_base + i_row : u.part + (i_row - u.row0);
                    HAT_CHECK(i_row >= u.C || (orow >= 0 && orow < (u.part < 0 ? (int64_t)a.plan.total_rows : a.part_rows)), status);
#pragma unroll 1
                    for (int c = 0; c < kD; c += 32) {
                        float o[32];
                        if (n_mine > 0) {
                            tmem_ld32(tm_o + c, reinterpret_cast<uint32_t*>(o));
                            tmem_ld_wait();
                        } else {
#pragma unroll
                            for (int k = 0; k < 32; ++k) o[k] = 0.f;
                        }
                        if (have1) {
                            uint32_t o1[32];
                            tmem_ld32(tm_o + 128 + c, o1);           // the second chain's accumulator: next 128 columns
                            tmem_ld_wait();
#pragma unroll
                            for (int k = 0; k < 32; ++k) o[k] = o[k] * w0 + __uint_as_float(o1[k]) * w1;
                        }
                        if (c == kD - 32 && (n_mine > 0 || have1)) {
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) {
                                if (n_mine > 0) mbar_arrive(&bars->o_free[qt]);
                                if (have1) mbar_arrive(&bars->o_free[1]);
                            }
                        }
                        out_rows::store<32, kD, false>(a, o, inv, u.part < 0, orow, u.C - i_row, u.h, c, lane);
                        __syncwarp();                            // rows past the chunk store nothing
                    }
                    if (i_row < u.C) (u.part < 0 ? a.lse : a.part_lse)[orow * H + u.h] = l > 0.f ? (m_used + log2f(l)) * 0.6931471805599453f : -INFINITY;
                }
            }
            kt_base += u.n_all;
        }
    }

    tc_fence_before();
    __syncthreads();
    if (bars->abort_flag) {
        if (threadIdx.x == 0) atomicOr(status, 1);
        settle();
    }
    if constexpr (FORM == kHalves) {
        cluster_arrive();                                        // the other CTA has read what it needs of this one's shared memory
        cluster_wait();
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(tmem) : "memory");
    }
    if (a.overlap && threadIdx.x == 0) pdl_wait();               // the next kernel takes this one's end for the end of both
}

// ---------------------------------------------------------------------------------------------- host side
}  // namespace

bool tc5_layout_supported(int dtype, int head_dim, int num_pages, int H, int64_t stride_page, int64_t stride_token,
                          int64_t stride_head) {
    if ((head_dim != 64 && head_dim != 128) || num_pages <= 0) return false;
    CUtensorMap m;
    // the encoder checks alignment and ranges only; any 16-byte aligned address will do for the probe
    const void* probe = reinterpret_cast<const void*>(uintptr_t(1) << 30);
    int fold;
    return tma_encode_pool_map(&m, dtype == HAT_DTYPE_BF16, probe, head_dim, num_pages, H, stride_page, stride_token, stride_head) &&
           tma_encode_tile_map(&m, dtype == HAT_DTYPE_BF16, probe, head_dim, num_pages, H, stride_page, stride_token, stride_head, &fold);
}

cudaError_t launch_attn_tc5(const hat_plan* plan, const AttnArgs& args, cudaStream_t stream, int grid_limit,
                            bool reset_counter, int first_unit, int num_units, int counter_word, bool overlap) {
    const bool bf16 = plan->dtype == HAT_DTYPE_BF16;
    const CUtensorMap *mk = nullptr, *mv = nullptr;
    const CUtensorMap* mq = plan_q_map(plan, args.q);
    const CUtensorMap *mkn = nullptr, *mvn = nullptr, *mvh = nullptr;
    int fold = 0;
    if (!mq || !plan_tile_maps(plan, args.cache, &mk, &mv, &fold) || !plan_new_maps(plan, args.k_new, args.v_new, &mkn, &mvn, &mvh))
        return cudaErrorInvalidValue;
    // one CTA per SM draws units from a counter that is zero at this point: the last of the previous call's producers cleared it
    // (reset_counter); a grid that joins another one on the same counter leaves it alone
    const int total_units = num_units >= 0 ? num_units : (int)plan->tile_units.size() - first_unit;
    if (total_units <= 0) return cudaSuccess;
    int32_t* counter = plan->dev.status + counter_word;
    AttnArgs a2 = args;
    a2.plan.tile_units = plan->dev.tile_units + first_unit;
    a2.tail_reset = reset_counter ? 1 : 0;
    a2.static_first = a2.tail_reset;            // a counter of its own
    a2.overlap = overlap || args.overlap ? 1 : 0;
    int ctas = std::min(total_units, plan->num_sms);
    if (grid_limit > 0) ctas = std::min(ctas, grid_limit);
    const dim3 grid((unsigned)ctas);
    const bool d128 = plan->head_dim == 128;
    const bool alone = total_units <= ctas && a2.static_first, one = d128 && alone;
    if (plan->tile_clusters && !alone) return cudaErrorInvalidValue;
    auto form = [&](auto b, auto app) {
        constexpr bool B = decltype(b)::value, A = decltype(app)::value;
        return !d128 ? (plan->tile_clusters ? attn_tc5_kernel<B, 64, kHalves, A> : attn_tc5_kernel<B, 64, kMany, A>) : plan->tile_clusters ? attn_tc5_kernel<B, 128, kHalves, A>
               : one ? attn_tc5_kernel<B, 128, kOne, A> : attn_tc5_kernel<B, 128, kMany, A>;
    };
    using Yes = std::true_type;
    using No = std::false_type;
    auto kern = args.k_new ? (bf16 ? form(Yes{}, Yes{}) : form(No{}, Yes{})) : (bf16 ? form(Yes{}, No{}) : form(No{}, No{}));
    const uint32_t smem = d128 ? smem_bytes<128>() : smem_bytes<64>();
    cudaError_t e = smem_attr_once(reinterpret_cast<const void*>(kern), (int)smem);
    if (e != cudaSuccess) return e;
    return launch_pdl_clusters(plan->tile_clusters ? 2 : 1, kern, grid, dim3(kThreads), smem, stream, a2, plan->dev.prefill_items, total_units, counter, *mq, *mk, *mv, *mkn, *mvn, fold);
}

}  // namespace hat
