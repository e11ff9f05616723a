// Streaming (verify-class) chunk attention: up to 16 query rows of one request against a long key range, bound by
// HBM bandwidth.  One launch appends the chunk's K/V rows, attends, and merges requests whose keys were cut.
//
// Persistent kernel, two CTAs per SM (grid = min(units, 2 x SMs)), six warps each.  A unit = one piece of a request's
// pages x one K/V head x one slab of 16 (chunk row, query head of the group) pairs; units are drawn longest piece
// first from a counter in the plan.  What a request's rows see is laid out as a list of 16-key pages:
//   pages 0 .. ceil(P/16)-1   the cached prefix, page by page of the block table (the last one cut at P)
//   page  ceil(P/16)          the chunk's own rows, gathered: from k_new / v_new when the call appends (the pool then
//                             need not be written first), else row by row from the pool; rows beyond the chunk are zero
// so both kinds of call do the same arithmetic in the same order and give the same bits.
//   warp 4      producer: reads its first unit's record and page ids, then waits for the end of the stream's previous kernel; unit
//               after unit without draining in between, the Q tile (cp.async) and the pages, each by two TMA boxes (16 tokens of K and
//               of V, 128-byte swizzle), into a ring of slots on mbarriers
//   warps 0-3   page j of a unit belongs to warp 3 - j mod 4: mma.sync m16n8k16, fp32 accumulate, online softmax whose
//               reference maximum only moves when it grows by more than 2^8, so the accumulator is rarely rescaled.
//               At the end of a unit the partial results pass from warp to warp through one shared-memory buffer; a warp
//               goes on with the next unit as soon as it has handed over.  The warp that consumed the chunk page copies its
//               rows from shared memory to the pool.
//   warp 5      takes the unit's result out of that buffer, normalises and stores it.  A request cut into pieces: every
//               piece stores partial rows and counts itself in; the CTA with the last piece of a (request, head, slab) merges them
//               at its end with all warps, in the order of the pieces.  A warp of its own, so that stores, fence and count (2 us
//               and more) hold up no one, and so that its registers do not weigh on the main loop
//
// A unit of 32 pairs (two warps to a page, K/V once instead of twice for grouped heads with more than 16 pairs) measured
// slower: 16 requests x 8 K/V heads x 16..32 pairs, bf16, 100 us against 89 to 93 in two slabs of 16.  There mma.sync is the limit
// (96 MMAs a page at 16 cycles), the second pass over K/V comes from L2, and slabs balance better.
//
// What bounds it: HBM for large batches (30 requests x 32 heads, 980 MB: 151 us = 6.5 TB/s, which is the measured copy rate; the
// step of append, this kernel and their gap was 163 us, now 157), the start of the pipeline and the tail for medium ones (12
// requests, 250 MB: 63 us of append, attention, merge and gaps per layer, now 46), a chain of latencies for one request
// (4 rows x 700 tokens: 10.9 us a call: 1 us to the Q tile, 1 us to the first page, 1.3 to 2 us of pages, 1.3 to 1.8 from warp to warp,
// 1.3 to store and count, 3.3 to merge).
// Batches of few units therefore run in a short form (CL > 0 below): a CTA for every unit, the warps' results combined by all warps
// at once, the pieces of a request exchanged within a cluster: 8.0 us for that call; pick_short_cluster (hat_api.cu) says which batches.
// Waits on the mbarriers are bounded and report through the plan's status word.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "hat_internal.h"
#include "tma_desc.h"
#include "tc5_ptx.cuh"

namespace hat {
namespace {
using tc5::cp_async16;
using tc5::fast_exp2;
using tc5::mbar_arrive;
using tc5::mbar_expect_tx;
using tc5::mbar_init;
using tc5::mbar_try;
using tc5::smem_u32;

constexpr int kWarps = 4;                   // consumer warps
constexpr int kThreads = kWarps * 32 + 64;
constexpr int kCtasPerSm = 2;
constexpr int kTodo = 48;                   // merges put off to the end of the CTA
constexpr int kBatch = 4;                   // pages requested at a time
constexpr int kAhead = 32;                  // pages prefetched to L2 before the previous kernel's end (a lane has one page id)
constexpr float kMoveThreshold = 8.0f;      // log2 units
constexpr float kLargest = 3.402823466e38f;

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
template <bool BF16>
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    if constexpr (BF16) {
        asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
                     : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                     : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
    } else {
        asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
                     : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                     : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
    }
}
template <bool BF16>
__device__ __forceinline__ uint32_t pack2(float lo, float hi) { return pack_out16(lo, hi, BF16); }
// the barrier's current phase also waits for this thread's copies so far
__device__ __forceinline__ void cp_async_on(uint64_t* bar) {
    asm volatile("cp.async.mbarrier.arrive.shared::cta.b64 [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}

// Byte offset of 16-byte vector c of token row `row` in a page as TMA lays it down: two 2 KiB column halves,
// rows of 128 bytes, the vector index XORed with the row (128-byte swizzle).
template <int D>
__device__ __forceinline__ uint32_t page_off(int row, int c) {
    if constexpr (D == 128) return (uint32_t)((c >> 3) * 2048 + row * 128 + (((c & 7) ^ (row & 7)) << 4));
    else return (uint32_t)(row * 128 + ((c ^ (row & 7)) << 4));
}
// The Q tile is written by ordinary copies: rows of D*2 bytes, vector index XORed with the row.
template <int D>
__device__ __forceinline__ uint32_t q_off(int row, int c) { return (uint32_t)(row * (D * 2) + ((c ^ (row & 7)) << 4)); }

// Shared memory of a CTA: ring slots (one page of K, then of V), the Q tile, the hand-over buffer, barriers.
// Every consumer warp has slots of its own: a parity wait is only sound for a waiter that has seen every earlier phase
// of the barrier, so a slot must not pass from one warp to another.
template <int D> struct Geo {
    static constexpr uint32_t PAGE = 16 * D * 2;                 // K (or V) of one page of one head
    static constexpr uint32_t SLOT = 2 * PAGE;
    static constexpr uint32_t Q = 16 * D * 2;
    static constexpr uint32_t X = (D / 8 + 1) * 512;             // accumulators (and maxima, sums) of one warp
    // as many slots as let two CTAs share an SM (115712 bytes each)
    static constexpr int PER = D == 64 ? 4 : 3;                  // slots of each consumer warp
    static constexpr int SLOTS = kWarps * PER;
};
template <int SLOTS> struct __align__(16) Ctl {
    int4 unit[3];                                                // the unit's StreamItem
    int hs;                                                      // its head * n_sub + slab; -1: no unit left
    uint64_t full[SLOTS], empty[SLOTS];
    uint64_t q_full, q_empty;                                    // Q tile, unit and hs
    int4 job[3];                                                 // the unit whose result is in the hand-over buffer
    uint64_t x_free;                                             // the buffer has been read
    int4 todo[kTodo][2];                                         // merges this CTA owes: it stored the last piece
    int num_todo;
    uint64_t todo_full;                                          // every unit is done, the list is final
    uint64_t hand[kWarps];                                       // warp w has handed over (the last in line: to the output warp)
    volatile int abort_flag;
    volatile long long wait_cycles;                              // bound of every wait (see tc5::waits_begin)
};

template <int SLOTS>
__device__ __forceinline__ bool wait_for(uint64_t* bar, uint32_t parity, Ctl<SLOTS>* ctl, const AttnArgs& a) {
    if (mbar_try(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try(bar, parity)) {
        if (ctl->abort_flag) return false;
        if (clock64() - t0 > ctl->wait_cycles) {
            ctl->abort_flag = 1;
            atomicOr(a.plan.status, 1);
            return false;
        }
    }
    return true;
}

// The same for a barrier that the other CTAs of the cluster arrive on, acquiring what they wrote before.
template <int SLOTS>
__device__ __forceinline__ bool wait_for_cluster(uint64_t* bar, uint32_t parity, Ctl<SLOTS>* ctl, const AttnArgs& a) {
    const long long t0 = clock64();
    while (!tc5::mbar_try_cluster(bar, parity)) {
        if (ctl->abort_flag) return false;
        if (clock64() - t0 > ctl->wait_cycles) {
            ctl->abort_flag = 1;
            atomicOr(a.plan.status, 1);
            return false;
        }
    }
    return true;
}

// The dynamic shared memory from its first 1024-byte boundary on: ring, Q tile, hand-over buffer, control block.
template <int D>
__device__ __forceinline__ Ctl<Geo<D>::SLOTS>* ctl_of(unsigned char* smem) {
    return reinterpret_cast<Ctl<Geo<D>::SLOTS>*>(smem + Geo<D>::SLOTS * Geo<D>::SLOT + Geo<D>::Q + Geo<D>::X);
}

// Final rows of a unit: column chunk c (8 columns) of rows g and g + 8 of the tile, each with its maximum and row sum in ml.
template <int D>
struct RowStore {
    const AttnArgs& a;
    int H, G, h, pair0, pairs, row_base, lane;
    template <typename F>
    __device__ __forceinline__ void rows(const float4& ml, F&& row) const {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            if (e * 8 + (lane >> 2) >= pairs) continue;
            const int pair = pair0 + e * 8 + (lane >> 2), i = pair / G;
            row(e, (int64_t)(row_base + i) * H + h * G + (pair - i * G), e ? ml.y : ml.x, e ? ml.w : ml.z);
        }
    }
    __device__ __forceinline__ void chunk(int c, const float4& o, int e, int64_t at, float inv) const {
        const float v0 = (e ? o.z : o.x) * inv, v1 = (e ? o.w : o.y) * inv;
        const int64_t to = at * D + 2 * (lane & 3) + c * 8;
        if (a.out16 != nullptr) *reinterpret_cast<uint32_t*>(static_cast<uint16_t*>(a.out16) + to) = pack_out16(v0, v1, a.out16_bf16);
        else *reinterpret_cast<float2*>(a.out + to) = make_float2(v0, v1);
    }
    __device__ __forceinline__ void lse(int64_t at, float m, float sum) const {
        if ((lane & 3) != 0) return;
        // ln of m and sum together, rounded once: sum = f 2^k with f near 1, whose logarithm is small, and m + k in two terms
        const int k = (__float_as_int(sum) - 0x3f3504f3) >> 23;
        const float f = __uint_as_float(__float_as_uint(sum) - ((uint32_t)k << 23)), mk = m + (float)k, low = (float)k - (mk - m);
        constexpr float kLn2 = 0.6931471805599453f;
        a.lse[at] = sum > 0.f ? fmaf(mk, kLn2, fmaf(low, kLn2, logf(f))) : -INFINITY;
    }
};

// Partial results of the same rows over other keys, one after the other: maxima and sums of rows g and g + 8 (x, y and z, w).
struct Weights { float m0, m1, l0, l1; };
template <int N>
__device__ __forceinline__ Weights weights_of(const float4 (&ml)[N], float (&w0)[N], float (&w1)[N]) {
    Weights t{-INFINITY, -INFINITY, 0.f, 0.f};
#pragma unroll
    for (int i = 0; i < N; ++i) { t.m0 = fmaxf(t.m0, ml[i].x); t.m1 = fmaxf(t.m1, ml[i].y); }
    const float f0 = t.m0 == -INFINITY ? 0.f : t.m0, f1 = t.m1 == -INFINITY ? 0.f : t.m1;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        w0[i] = fast_exp2(ml[i].x - f0); w1[i] = fast_exp2(ml[i].y - f1);
        t.l0 += ml[i].z * w0[i]; t.l1 += ml[i].w * w1[i];
    }
    return t;
}

// The warps' work.  A warp returns when it is done, or early when a wait gave up.
// CL = 0: persistent, as above.  CL > 0, the short form: as many CTAs as units, each with one: the CTAs of a cluster of CL have the pieces
// (of equal size, the last with the chunk) of one request, K/V head and slab.  The warps' results meet in the ring slots, which nothing will refill, and are
// combined by all warps at once; then the CTAs' through each other's shared memory, every CTA finishing D / CL columns: no chain
// from warp to warp, no output warp, no partial rows, fence, count and merge.
template <bool BF16, int D, int CL>
__device__ __forceinline__ void stream_roles(const AttnArgs& a, unsigned char* smem, const StreamItem* __restrict__ items, int n_sub, int total_units,
                                             int32_t* __restrict__ work_counter, int32_t* __restrict__ piece_counters, const CUtensorMap& map_k,
                                             const CUtensorMap& map_v) {
    using G_ = Geo<D>;
    constexpr int CH = D / 8, ON = D / 8, SLOTS = G_::SLOTS, PER = G_::PER;
    constexpr uint32_t PAGE = G_::PAGE, SLOT = G_::SLOT;
    using Ctl_ = Ctl<SLOTS>;

    unsigned char* q_buf = smem + SLOTS * SLOT;
    float4* xbuf = reinterpret_cast<float4*>(q_buf + G_::Q);
    Ctl_* ctl = ctl_of<D>(smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (tid == 0) {
        for (int s = 0; s < SLOTS; ++s) { mbar_init(&ctl->full[s], 1); mbar_init(&ctl->empty[s], 1); }
        mbar_init(&ctl->q_full, 1);
        mbar_init(&ctl->q_empty, kWarps);
        mbar_init(&ctl->x_free, CL > 1 ? CL * kWarps : 1);
        mbar_init(&ctl->todo_full, 1);
        ctl->num_todo = 0;
        for (int w = 0; w < kWarps; ++w) mbar_init(&ctl->hand[w], CL > 0 ? kWarps : 1);
        ctl->abort_flag = 0;
        ctl->wait_cycles = tc5::kNotYet;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    }
    __syncthreads();
    if constexpr (CL > 1) {
        tc5::cluster_arrive();                                    // the other CTAs' barriers are initialised
        tc5::cluster_wait();
    }
    const int rank = CL > 1 ? (int)tc5::cluster_ctarank() : 0;

    const int H = a.plan.num_heads, G = a.plan.group, Hkv = a.plan.num_kv_heads;
    const int hs_count = Hkv * n_sub;
    const int4* __restrict__ recs = reinterpret_cast<const int4*>(items);
    // chunk row of a (row, query head of the group) pair: pair / G, by a multiplication while that is exact (16 G pairs at most)
    const uint32_t g_inv = ((1u << 20) + G - 1) / G;
    auto pair_row = [&](int pair) { return G < 256 ? (int)(((uint32_t)pair * g_inv) >> 20) : pair / G; };
    bool ok = true;

    if (warp == kWarps) {
        // ------------------------------------------------------------------ producer
        const long long since = clock64();
        const uint16_t* __restrict__ q = static_cast<const uint16_t*>(a.q);
        const bool fused = a.k_new != nullptr;
        // Pages are requested kBatch at a time, lanes 2 k and 2 k + 1 moving K and V of page k: a page at a time (600 cycles of
        // waiting and issuing each) held the kernel at 4.8 TB/s.
        // Page j of a unit goes to way kWarps - 1 - j mod kWarps: where the pages do not come out even, the first in the hand-over line
        // has the fewest.
        const int bk = lane < 2 * kBatch ? lane >> 1 : 0, is_v = lane & 1, way = kWarps - 1 - bk % kWarps;
        int issued = 0;                                           // pages requested for `way` so far
        int unit = CL > 1 ? blockIdx.x / CL : blockIdx.x, un = 0;
        int hs = 0, page_id = 0;
        int4 r0, r1, r2;                                          // the unit's StreamItem; page_id: of its first 32 pages, one per lane
        auto fetch_record = [&](int u, int& hs_, int4& q0, int4& q1, int4& q2) {
            const int item = u / hs_count;
            hs_ = u - item * hs_count;
            q0 = __ldg(recs + item * 3); q1 = __ldg(recs + item * 3 + 1); q2 = __ldg(recs + item * 3 + 2);
        };
        auto fetch_ids = [&](const int4& q0, const int4& q1) {
            const int32_t* __restrict__ t = a.plan.block_table + (int64_t)q0.x * a.plan.max_pages;
            const int pg = q1.x + lane;
            return pg < min(q1.y, (q0.w + kPageSize - 1) / kPageSize) ? __ldg(t + pg) : 0;
        };
        fetch_record(unit, hs, r0, r1, r2);
        if constexpr (CL > 1) {
            const int pages = r1.y;
            r1.x = pages * rank / CL; r1.y = pages * (rank + 1) / CL;
        }
        page_id = fetch_ids(r0, r1);
        {
            // CTAs of this kernel start as those of the one before run out of work: its tail brings their first pages to L2
            // (eight calls of 12 requests x 32 heads one after the other: 376 us without, 366 us with; 12 pages 368)
            const int npre = (r0.w + kPageSize - 1) / kPageSize, h = hs / n_sub;
            if (lane < kAhead && r1.x + lane < min(r1.y, npre)) {
                const int page = HAT_IN_RANGE(page_id, a.plan.num_pages, a.plan.status);
                tc5::tma_prefetch_5d(&map_k, 0, 0, 0, h, page);
                tc5::tma_prefetch_5d(&map_v, 0, 0, 0, h, page);
            }
        }
        tc5::pdl_wait();                                          // up to here only the plan's own arrays were read
        if (lane == 0) tc5::waits_begin(&ctl->wait_cycles, since, a.wait_cycles);
        // the kernel behind may be one that runs beside this one (tile kernels of the same call): what precedes both has ended
        tc5::pdl_launch_dependents();
        for (;;) {
            const bool done = unit >= total_units;
            const int row_base = r0.y, C = r0.z, P = r0.w, page0 = r1.x, page1 = r1.y;
            const int32_t* __restrict__ table = a.plan.block_table + (int64_t)r0.x * a.plan.max_pages;
            const int npre = (P + kPageSize - 1) / kPageSize;
            const int h = hs / n_sub, sub = hs - h * n_sub;
#ifdef HAT_DEBUG_BOUNDS
            if (!done && (r0.x < 0 || C < 1 || C > 16 || P < 0 || row_base < 0 || row_base + C > a.plan.total_rows || page0 < 0 ||
                          page1 < page0 || (CL == 0 && page1 == page0) || page1 > npre + 1 || npre > a.plan.max_pages || r2.x < 1 || r2.x > kMaxSplits)) {
                if (lane == 0) atomicOr(a.plan.status, 2);
                ctl->abort_flag = 1;
                ok = false;
                break;
            }
#endif
            const bool skip = !done && sub * 16 >= C * G;    // this request has fewer pairs
            if constexpr (CL > 0) {
                if (skip) {                                       // of every CTA of the cluster
                    if (lane == 0) { ctl->hs = -1; mbar_arrive(&ctl->q_full); }
                    break;
                }
            }
            if (!skip) {
                if (un >= 1) ok = wait_for(&ctl->q_empty, (un - 1) & 1, ctl, a);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                if (!done) {
                    // this lane copies 16 bytes of every (32 / CH)-th row
                    const int c = lane % CH;
#pragma unroll
                    for (int row = lane / CH; row < 16; row += 32 / CH) {
                        const int pair = sub * 16 + row, i = pair_row(pair);
                        const bool in = i < C;
                        const uint16_t* src = q + (in ? ((int64_t)(row_base + i) * H + h * G + (pair - i * G)) * D + c * 8 : 0);
                        cp_async16(smem_u32(q_buf) + q_off<D>(row, c), src, in);
                    }
                    cp_async_on(&ctl->q_full);
                }
                if (lane == 0) { ctl->unit[0] = r0; ctl->unit[1] = r1; ctl->unit[2] = r2; ctl->hs = done ? -1 : hs; }
                __syncwarp();
                // self test: the first Q tile never arrives (of a cluster, its first CTA's: the others wait for that one's result in vain)
                if (lane == 0 && !(a.withhold && un == 0 && rank == 0)) mbar_arrive(&ctl->q_full);
                ++un;
            }
            if (done) break;
            // The next unit is drawn, its record and its first page ids are fetched while this unit's last pages are requested,
            // one step per batch: fetched at the boundary they cost 2 us without a request in flight.
            int step = 0, drawn = 0, next = 0, next_hs = 0, next_id = 0;
            int4 n0 = r0, n1 = r1, n2 = r2;
            auto look_ahead = [&]() {
                if (step == 0) {
                    if (lane == 0) drawn = atomicAdd(work_counter, 1);
                } else if (step == 1) {
                    next = __shfl_sync(0xffffffffu, drawn, 0) + (int)gridDim.x;
                    if (next < total_units) fetch_record(next, next_hs, n0, n1, n2);
                } else {
                    if (next < total_units) next_id = fetch_ids(n0, n1);
                }
                ++step;
            };
            if (!skip) {
                const int n = page1 - page0;
                int ids = page_id, ids_next = 0;                  // page ids of this and the next 32 pages, one per lane
                for (int j0 = 0; j0 < n; j0 += kBatch) {
                    if (CL == 0 && step < 3 && n - j0 <= 6 * kBatch) look_ahead();
                    if ((j0 & 31) == 0) {
                        if (j0 > 0) ids = ids_next;
                        const int ahead = page0 + j0 + 32 + lane;
                        ids_next = ahead < min(page1, npre) ? __ldg(table + ahead) : 0;
                    }
                    const int page = HAT_IN_RANGE(__shfl_sync(0xffffffffu, ids, (j0 + bk) & 31), a.plan.num_pages, a.plan.status);
                    const int turn = issued + bk / kWarps, slot = way * PER + turn % PER;
                    const bool mine = lane < 2 * kBatch && j0 + bk < n;
                    if (mine && turn >= PER) ok = wait_for(&ctl->empty[slot], (turn / PER - 1) & 1, ctl, a);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    const bool prefix = mine && page0 + j0 + bk < npre;
                    if (prefix && !is_v) mbar_expect_tx(&ctl->full[slot], SLOT);
                    __syncwarp();
                    if (prefix) tc5::tma_load_5d(smem_u32(smem) + slot * SLOT + is_v * PAGE, is_v ? &map_v : &map_k, 0, 0, 0, h, page, &ctl->full[slot]);
                    if (page1 > npre && j0 + kBatch >= n) {
                        // the chunk's rows, one after the other from k_new / v_new or from their slots of the pool
                        const int cslot = __shfl_sync(0xffffffffu, slot, 2 * (n - 1 - j0));
                        const uint32_t dst = smem_u32(smem) + cslot * SLOT;
#pragma unroll 4
                        for (int idx = lane; idx < 16 * CH; idx += 32) {
                            const int row = idx / CH, c = idx % CH;
                            const bool in = row < C;
                            const uint16_t *ks = static_cast<const uint16_t*>(a.cache.k_pool), *vs = static_cast<const uint16_t*>(a.cache.v_pool);
                            if (in && fused) {
                                const int64_t off = ((int64_t)(row_base + row) * Hkv + h) * D + c * 8;
                                ks = static_cast<const uint16_t*>(a.k_new) + off;
                                vs = static_cast<const uint16_t*>(a.v_new) + off;
                            } else if (in) {
                                const int pos = P + row;
                                const int pp = HAT_IN_RANGE(__ldg(table + HAT_IN_RANGE(pos / kPageSize, a.plan.max_pages, a.plan.status)), a.plan.num_pages, a.plan.status);
                                const int64_t off = pp * a.cache.stride_page + (pos % kPageSize) * a.cache.stride_token + h * a.cache.stride_head + c * 8;
                                ks += off; vs += off;
                            }
                            cp_async16(dst + page_off<D>(row, c), ks, in);
                            cp_async16(dst + PAGE + page_off<D>(row, c), vs, in);
                        }
                        cp_async_on(&ctl->full[cslot]);
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&ctl->full[cslot]);
                    }
                    issued += (min(kBatch, n - j0) + way) / kWarps;
                }
                if (!ok) break;
            }
            if constexpr (CL > 0) break;
            while (step < 3) look_ahead();
            unit = next; hs = next_hs; page_id = next_id;
            r0 = n0; r1 = n1; r2 = n2;
        }
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        // the last producer to finish leaves the unit counter at zero for the next call
        if (CL == 0 && lane == 0) {
            __threadfence();
            if (atomicAdd(work_counter + 1, 1) == (int)gridDim.x - 1) {
                work_counter[0] = 0;
                work_counter[1] = 0;
                __threadfence();
            }
        }
        return;
    }

    // Merges of cut requests whose last piece this CTA stored: rows first, first + step, ... of the list, two at a time.  They are
    // put off to the end of the CTA: a round trip to L2 takes 3000 cycles while the pages stream, a merge several of them,
    // and meanwhile the hand-over buffer would be blocked (spec_verify cut into 135 pieces: 9 us per merge).
    auto merge_todo = [&](int first, int step) {
        constexpr int V = D / 32, NP = 8;                         // floats per lane, pieces in flight
        const int n_todo = ctl->num_todo;
        int turn = 0;
        for (int e = 0; e < n_todo; ++e) {
            const int4 j0 = ctl->todo[e][0], j1 = ctl->todo[e][1];
            const int part0 = j0.x, nsplit = j0.y, row_base = j0.z, C = j0.w, pair0 = j1.x, pairs = j1.y, h = j1.z;
            const int64_t hop = (int64_t)C * H;                   // (row, head) pairs from one piece to the next
            for (int p0 = 0; p0 < pairs; p0 += 2, ++turn) {
                if (turn % step != first) continue;
                int64_t at0[2], at[2];
                float w[2], v[2][NP][V], acc[2][V], mx[2], sum[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int pair = pair0 + min(p0 + u, pairs - 1), i = pair_row(pair), hq = h * G + (pair - i * G);
                    at0[u] = ((int64_t)part0 + i) * H + hq;
                    at[u] = (int64_t)(row_base + i) * H + hq;
                    w[u] = lane < nsplit ? __ldcg(a.part_lse + at0[u] + lane * hop) : -INFINITY;
                }
                auto load_pieces = [&](int s0) {
#pragma unroll
                    for (int u = 0; u < 2; ++u)
#pragma unroll
                        for (int s = 0; s < NP; ++s)
                            if (s0 + s < nsplit) {
                                const float* src = a.part_out + (at0[u] + (s0 + s) * hop) * D + lane * V;
                                if constexpr (V == 4) { const float4 y = __ldcg(reinterpret_cast<const float4*>(src)); v[u][s][0] = y.x; v[u][s][1] = y.y; v[u][s][2] = y.z; v[u][s][3] = y.w; }
                                else { const float2 y = __ldcg(reinterpret_cast<const float2*>(src)); v[u][s][0] = y.x; v[u][s][1] = y.y; }
                            }
                };
                load_pieces(0);
#pragma unroll
                for (int u = 0; u < 2; ++u) mx[u] = w[u];
#pragma unroll
                for (int k = 16; k > 0; k >>= 1)
#pragma unroll
                    for (int u = 0; u < 2; ++u) mx[u] = fmaxf(mx[u], __shfl_xor_sync(0xffffffffu, mx[u], k));
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    mx[u] = mx[u] == -INFINITY ? 0.f : mx[u];
                    w[u] = sum[u] = expf(w[u] - mx[u]);           // 0 for empty pieces and idle lanes
                }
#pragma unroll
                for (int k = 16; k > 0; k >>= 1)
#pragma unroll
                    for (int u = 0; u < 2; ++u) sum[u] += __shfl_xor_sync(0xffffffffu, sum[u], k);
#pragma unroll
                for (int u = 0; u < 2; ++u)
#pragma unroll
                    for (int k = 0; k < V; ++k) acc[u][k] = 0.f;
                for (int s0 = 0; s0 < nsplit; s0 += NP) {
                    if (s0 > 0) load_pieces(s0);
#pragma unroll
                    for (int s = 0; s < NP; ++s)
                        if (s0 + s < nsplit) {
#pragma unroll
                            for (int u = 0; u < 2; ++u) {
                                const float ws = __shfl_sync(0xffffffffu, w[u], s0 + s);
#pragma unroll
                                for (int k = 0; k < V; ++k) acc[u][k] += ws * v[u][s][k];
                            }
                        }
                }
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    if (p0 + u >= pairs) break;
                    const float inv = sum[u] > 0.f ? 1.f / sum[u] : 0.f;
#pragma unroll
                    for (int k = 0; k < V; ++k) acc[u][k] *= inv;
                    if (a.out16 != nullptr) {
                        uint16_t* dst = static_cast<uint16_t*>(a.out16) + at[u] * D + lane * V;
                        if constexpr (V == 4)
                            *reinterpret_cast<uint2*>(dst) = make_uint2(pack_out16(acc[u][0], acc[u][1], a.out16_bf16), pack_out16(acc[u][2], acc[u][3], a.out16_bf16));
                        else
                            *reinterpret_cast<uint32_t*>(dst) = pack_out16(acc[u][0], acc[u][1], a.out16_bf16);
                    } else if constexpr (V == 4) {
                        *reinterpret_cast<float4*>(a.out + at[u] * D + lane * V) = make_float4(acc[u][0], acc[u][1], acc[u][2], acc[u][3]);
                    } else {
                        *reinterpret_cast<float2*>(a.out + at[u] * D + lane * V) = make_float2(acc[u][0], acc[u][1]);
                    }
                    if (lane == 0) a.lse[at[u]] = sum[u] > 0.f ? mx[u] + logf(sum[u]) : -INFINITY;
                }
            }
        }
    };

    if (CL == 0 && warp == kWarps + 1) {
        // ------------------------------------------------------------------ output, merge of cut requests
        const int g = lane >> 2, t4 = lane & 3;
        for (int un = 0;; ++un) {
            ok = __all_sync(0xffffffffu, wait_for(&ctl->hand[kWarps - 1], un & 1, ctl, a));
            if (!ok) return;
            const int4 j0 = ctl->job[0], j1 = ctl->job[1], j2 = ctl->job[2];
            const int part0 = j0.x, nsplit = j0.y, row_base = j0.w, C = j1.x, pair0 = j1.y, pairs = j1.z, h = j1.w, part = j2.x;
            if (nsplit < 0) {
                if (lane == 0) mbar_arrive(&ctl->todo_full);
                merge_todo(kWarps, kWarps + 1);
                return;
            }
            {
                float4 o[ON];
                const float4* x = xbuf + lane;
                const float4 ml = x[ON * 32];
#pragma unroll
                for (int c = 0; c < ON; ++c) o[c] = x[c * 32];
                __syncwarp();
                if (lane == 0) mbar_arrive(&ctl->x_free);
                // normalise and store: final rows, or partial rows of a cut request
                constexpr float kLn2 = 0.6931471805599453f;
                const bool to16 = part < 0 && a.out16 != nullptr;    // final rows in the 16-bit output type
                float* obase = part < 0 ? a.out : a.part_out;
                float* lbase = part < 0 ? a.lse : a.part_lse;
                const int64_t first = part < 0 ? row_base : part;
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    if (e * 8 + g >= pairs) continue;
                    const int pair = pair0 + e * 8 + g, i = pair_row(pair), hq = h * G + (pair - i * G);
                    const float m = e ? ml.y : ml.x, sum = e ? ml.w : ml.z, inv = sum > 0.f ? 1.f / sum : 0.f;
                    const int64_t at = ((first + i) * H + hq) * D + 2 * t4;
#pragma unroll
                    for (int c = 0; c < ON; ++c) {
                        const float v0 = (e ? o[c].z : o[c].x) * inv, v1 = (e ? o[c].w : o[c].y) * inv;
                        if (to16) *reinterpret_cast<uint32_t*>(static_cast<uint16_t*>(a.out16) + at + c * 8) = pack_out16(v0, v1, a.out16_bf16);
                        else *reinterpret_cast<float2*>(obase + at + c * 8) = make_float2(v0, v1);
                    }
                    if (t4 == 0) lbase[(first + i) * H + hq] = sum > 0.f ? (m + log2f(sum)) * kLn2 : -INFINITY;
                }
            }
            if (part < 0) continue;
            __syncwarp();
            int arrived = 0;
            if (lane == 0) {
                asm volatile("fence.acq_rel.gpu;\n" ::: "memory");   // every lane's partial rows before the count
                arrived = atomicAdd(piece_counters + j0.z, 1);
            }
            if (__shfl_sync(0xffffffffu, arrived, 0) != nsplit - 1) continue;
            asm volatile("fence.acq_rel.gpu;\n" ::: "memory");
            if (lane == 0) piece_counters[j0.z] = 0;              // for the next call
            if (lane == 0) {
                const int at = ctl->num_todo;
                ctl->todo[at][0] = make_int4(part0, nsplit, row_base, C);
                ctl->todo[at][1] = make_int4(pair0, pairs, h, 0);
                ctl->num_todo = at + 1;
            }
            __syncwarp();
            if (ctl->num_todo == kTodo) {                         // no room for more: pay now
                merge_todo(0, 1);
                __syncwarp();
                if (lane == 0) ctl->num_todo = 0;
                __syncwarp();
            }
        }
    }

    // ---------------------------------------------------------------------- consumers
    const int g = lane >> 2, t4 = lane & 3, mi = lane >> 3;
    const bool append = a.k_new != nullptr;
    const uint32_t k_lane = page_off<D>((mi >> 1) * 8 + (lane & 7), mi & 1), v_lane = page_off<D>((mi & 1) * 8 + (lane & 7), mi >> 1);
    int taken = 0;                                                // pages this warp has consumed so far
    for (int un = 0;; ++un) {
        ok = __all_sync(0xffffffffu, wait_for(&ctl->q_full, un & 1, ctl, a));
        if (!ok) return;
        const int hs = ctl->hs;
        if (CL > 0 && hs < 0) return;
        if (hs < 0) {
            // the end, handed on to the output warp once it has taken the previous result
            if (warp == kWarps - 1) {
                if (un > 0) ok = __all_sync(0xffffffffu, wait_for(&ctl->x_free, (un - 1) & 1, ctl, a));
                if (!ok) return;
                if (lane == 0) { ctl->job[0] = make_int4(0, -1, 0, 0); mbar_arrive(&ctl->hand[warp]); }
            }
            // what is left to merge, with every warp
            ok = __all_sync(0xffffffffu, wait_for(&ctl->todo_full, 0, ctl, a));
            if (ok) merge_todo(warp, kWarps + 1);
            return;
        }
        const int4 r0 = ctl->unit[0], r1 = ctl->unit[1], r2 = ctl->unit[2];
        const int row_base = r0.y, C = r0.z, P = r0.w, page0 = r1.x, n = r1.y - r1.x, part = r1.z;
        const int h = hs / n_sub, sub = hs - h * n_sub;
        const int npre = (P + kPageSize - 1) / kPageSize;
        const int pair0 = sub * 16;                                // the unit's pairs: pair0 .. pair0 + pairs - 1
        const int pairs = min(16, C * G - pair0);                  // at least 1
        const bool low_rows = pairs <= 8;                          // rows 8..15 of the tile hold nothing
        const uint32_t qbase = smem_u32(q_buf);

        uint32_t qf[D / 16][4];
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks) ldsm4(qf[ks], qbase + q_off<D>((mi & 1) * 8 + (lane & 7), ks * 2 + (mi >> 1)));
        __syncwarp();
        if (lane == 0) mbar_arrive(&ctl->q_empty);

        float o[ON][4];
        float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};     // reference maxima (log2 units) and row sums, rows g and g+8
        float top[2] = {-INFINITY, -INFINITY};                      // their highest so far
#pragma unroll
        for (int k = 0; k < ON; ++k) o[k][0] = o[k][1] = o[k][2] = o[k][3] = 0.f;

        for (int j = kWarps - 1 - warp; j < n; j += kWarps, ++taken) {
            const int slot = warp * PER + taken % PER;
            const int pg = page0 + j;
            const bool chunk_page = pg == npre;
            // where the rows this lane will copy to the pool go: looked up ahead of the wait
            int page_a = 0, page_b = 0;
            if (chunk_page && append && sub == 0) {
                const int32_t* __restrict__ table = a.plan.block_table + (int64_t)r0.x * a.plan.max_pages;
                page_a = HAT_IN_RANGE(__ldg(table + HAT_IN_RANGE(P / kPageSize, a.plan.max_pages, a.plan.status)), a.plan.num_pages, a.plan.status);
                page_b = HAT_IN_RANGE(__ldg(table + HAT_IN_RANGE((P + C - 1) / kPageSize, a.plan.max_pages, a.plan.status)), a.plan.num_pages, a.plan.status);
            }
            ok = __all_sync(0xffffffffu, wait_for(&ctl->full[slot], (taken / PER) & 1, ctl, a));
            if (!ok) return;
            const uint32_t kst = smem_u32(smem) + slot * SLOT, vst = kst + PAGE;
            // where this lane's first fragment of K and V lies; the others differ in address bits 5 and 6 and by 2 KiB (page_off)
            const uint32_t ka = kst + k_lane, va = vst + v_lane;
            // keys of the page before `cut` hold the prefix (all 16 but in its last page); the chunk page has its own rule
            const int cut = chunk_page ? kPageSize : min(kPageSize, P - pg * kPageSize);
            if (cut < kPageSize) {
                // slots past the prefix hold stale tokens: zero their V rows so that 0 * garbage cannot produce NaN (their
                // scores are masked below)
                for (int idx = lane; idx < (kPageSize - cut) * CH; idx += 32) {
                    const int row = cut + idx / CH, c = idx % CH;
                    asm volatile("st.shared.v4.b32 [%0], {%1,%1,%1,%1};\n" ::"r"(vst + page_off<D>(row, c)), "r"(0) : "memory");
                }
                asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");   // the slot's next TMA write comes after these
                __syncwarp();
            }

            // S = Q K^T for the 16 keys of the page, even and odd halves of the sum apart (half as long a chain of MMAs)
            float s[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}}, s2[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks) {
                uint32_t b[4];
                ldsm4(b, (ka ^ ((ks & 3) << 5)) + (ks >> 2) * 2048);
                mma16816<BF16>(ks & 1 ? s2[0] : s[0], qf[ks], b[0], b[1]);
                mma16816<BF16>(ks & 1 ? s2[1] : s[1], qf[ks], b[2], b[3]);
            }
            uint32_t pa[4], pl[4];
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
                for (int e = 0; e < 4; ++e) s[k][e] = (s[k][e] + s2[k][e]) * a.scale_log2;
            if (chunk_page || cut < kPageSize) {
                // visible keys of the page, bit c = key c: of the chunk, its causal or tree word; of the prefix, those before `cut`
                uint32_t bits0 = (1u << cut) - 1u, bits1 = bits0;
                if (chunk_page) {
                    const int i0 = pair_row(pair0 + g), i1 = pair_row(pair0 + g + 8);
                    const uint32_t all = (1u << C) - 1u;
                    bits0 = i0 < C ? (2u << i0) - 1u : 0u; bits1 = i1 < C ? (2u << i1) - 1u : 0u;
                    if (a.plan.tree_mask != nullptr) {
                        if (i0 < C) bits0 = __ldg(a.plan.tree_mask + row_base + i0) & all;
                        if (i1 < C) bits1 = __ldg(a.plan.tree_mask + row_base + i1) & all;
                    }
                }
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const int c = k * 8 + 2 * t4;
                    s[k][0] = (bits0 >> c) & 1u ? s[k][0] : -INFINITY;
                    s[k][1] = (bits0 >> (c + 1)) & 1u ? s[k][1] : -INFINITY;
                    s[k][2] = (bits1 >> c) & 1u ? s[k][2] : -INFINITY;
                    s[k][3] = (bits1 >> (c + 1)) & 1u ? s[k][3] : -INFINITY;
                }
            }
            float mx0 = fmaxf(fmaxf(s[0][0], s[0][1]), fmaxf(s[1][0], s[1][1]));
            float mx1 = low_rows ? -INFINITY : fmaxf(fmaxf(s[0][2], s[0][3]), fmaxf(s[1][2], s[1][3]));
            mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 1));
            mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 1));
            mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 2));
            mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 2));
            // move a row's reference maximum only when the new maximum exceeds it by more than the threshold; weights
            // then stay below 2^8 and the accumulators are rescaled only on the (rare) pages where some row moved.
            // In the short form it moves to every page's own maximum (unless that is far below an earlier one, whose weights count for more): the
            // largest weight of each page is then 1, which no rounding changes.  Without it the error against 64 bits was up to 1.29 times that of
            // the persistent kernel's many short pieces, with it 0.82 (fp16) and 0.86 (bf16) of it (geometric means of 60 batches).  No branch
            // around it: packed products in line cost less than the jump (700 tokens x 32 heads bf16 8.5 us, 8.8 with, 8.7 moving rarely).
            if constexpr (CL > 0) {
                top[0] = fmaxf(top[0], mx0); top[1] = fmaxf(top[1], mx1);
                // (an infinite maximum moves it too, so that such a row is NaN as in the other form)
                const bool mv0 = mx0 > fminf(top[0] - kMoveThreshold, kLargest), mv1 = mx1 > fminf(top[1] - kMoveThreshold, kLargest);
                const float al0 = mv0 ? fast_exp2(m[0] - mx0) : 1.f, al1 = low_rows ? al0 : mv1 ? fast_exp2(m[1] - mx1) : 1.f;
                if (mv0) m[0] = mx0;
                if (mv1) m[1] = mx1;
                l[0] *= al0; l[1] *= al1;
                const uint64_t by0 = tc5::f2_pack(al0, al0), by1 = tc5::f2_pack(al1, al1);
#pragma unroll
                for (int k = 0; k < ON; ++k) {
                    tc5::f2_unpack(tc5::f2_mul(tc5::f2_pack(o[k][0], o[k][1]), by0), o[k][0], o[k][1]);
                    tc5::f2_unpack(tc5::f2_mul(tc5::f2_pack(o[k][2], o[k][3]), by1), o[k][2], o[k][3]);
                }
            } else {
                const bool mv0 = mx0 > m[0] + kMoveThreshold, mv1 = mx1 > m[1] + kMoveThreshold;
                if (__any_sync(0xffffffffu, mv0 || mv1)) {
                    const float al0 = mv0 ? ((m[0] == -INFINITY) ? 0.f : fast_exp2(m[0] - mx0)) : 1.f;
                    const float al1 = low_rows ? al0 : mv1 ? ((m[1] == -INFINITY) ? 0.f : fast_exp2(m[1] - mx1)) : 1.f;
                    if (mv0) m[0] = mx0;
                    if (mv1) m[1] = mx1;
                    l[0] *= al0; l[1] *= al1;
#pragma unroll
                    for (int k = 0; k < ON; ++k) { o[k][0] *= al0; o[k][1] *= al0; o[k][2] *= al1; o[k][3] *= al1; }
                }
            }
            const float ref0 = (m[0] == -INFINITY) ? 0.f : m[0], ref1 = (m[1] == -INFINITY) ? 0.f : m[1];
            // P in the A operand's layout: words 0 and 2 are rows 0..7, words 1 and 3 rows 8..15.  bf16 keeps 8 significant bits,
            // so what the rounding of P dropped is multiplied as well: in the idle rows 8..15 where those hold nothing
            // (half the MMAs), else as a second operand.
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                float (&e)[4] = s[k];
                e[0] = fast_exp2(e[0] - ref0); e[1] = fast_exp2(e[1] - ref0);
                l[0] += e[0] + e[1];
                pa[2 * k] = pack2<BF16>(e[0], e[1]);
                if constexpr (BF16)
                    pl[2 * k] = pack2<BF16>(e[0] - __uint_as_float(pa[2 * k] << 16), e[1] - __uint_as_float(pa[2 * k] & 0xffff0000u));
                if (low_rows) {
                    pa[2 * k + 1] = BF16 ? pl[2 * k] : 0u;
                    continue;
                }
                e[2] = fast_exp2(e[2] - ref1); e[3] = fast_exp2(e[3] - ref1);
                l[1] += e[2] + e[3];
                pa[2 * k + 1] = pack2<BF16>(e[2], e[3]);
                if constexpr (BF16)
                    pl[2 * k + 1] = pack2<BF16>(e[2] - __uint_as_float(pa[2 * k + 1] << 16), e[3] - __uint_as_float(pa[2 * k + 1] & 0xffff0000u));
            }
            // O += P V
#pragma unroll
            for (int dn = 0; dn < D / 16; dn += 2) {
                uint32_t b[4], c[4];
                ldsm4t(b, (va ^ ((dn & 3) << 5)) + (dn >> 2) * 2048);
                ldsm4t(c, (va ^ (((dn + 1) & 3) << 5)) + ((dn + 1) >> 2) * 2048);
                mma16816<BF16>(o[2 * dn], pa, b[0], b[1]);
                mma16816<BF16>(o[2 * dn + 1], pa, b[2], b[3]);
                mma16816<BF16>(o[2 * dn + 2], pa, c[0], c[1]);
                mma16816<BF16>(o[2 * dn + 3], pa, c[2], c[3]);
                if (BF16 && !low_rows) {
                    mma16816<BF16>(o[2 * dn], pl, b[0], b[1]);
                    mma16816<BF16>(o[2 * dn + 1], pl, b[2], b[3]);
                    mma16816<BF16>(o[2 * dn + 2], pl, c[0], c[1]);
                    mma16816<BF16>(o[2 * dn + 3], pl, c[2], c[3]);
                }
            }
            if (chunk_page && append && sub == 0) {
                // the chunk's rows on to their slots of the pool, as they lie in shared memory
                const int64_t head = (int64_t)h * a.cache.stride_head;
                for (int idx = lane; idx < C * CH; idx += 32) {
                    const int row = idx / CH, c = idx % CH, pos = P + row;
                    const int page = pos / kPageSize == P / kPageSize ? page_a : page_b;
                    const int64_t at = page * a.cache.stride_page + (pos % kPageSize) * a.cache.stride_token + head + c * 8;
                    *reinterpret_cast<uint4*>(static_cast<uint16_t*>(a.k_dst) + at) = *reinterpret_cast<const uint4*>(smem + slot * SLOT + page_off<D>(row, c));
                    *reinterpret_cast<uint4*>(static_cast<uint16_t*>(a.v_dst) + at) = *reinterpret_cast<const uint4*>(smem + slot * SLOT + PAGE + page_off<D>(row, c));
                }
            }
            if (chunk_page) asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");   // written by copies, next by TMA
            __syncwarp();
            if (lane == 0) mbar_arrive(&ctl->empty[slot]);
        }

        // ---- the warps' results, from warp to warp in order (fragment positions are identical in each)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            l[e] += __shfl_xor_sync(0xffffffffu, l[e], 1);
            l[e] += __shfl_xor_sync(0xffffffffu, l[e], 2);
        }
        if (BF16 && low_rows) {                                    // the second term of the weights was summed in rows 8..15
#pragma unroll
            for (int k = 0; k < ON; ++k) { o[k][0] += o[k][2]; o[k][1] += o[k][3]; }
        }
        if constexpr (CL > 0) {
            const auto result_of = [&](int w) { return reinterpret_cast<float4*>(smem + w * PER * SLOT) + lane; };
            static_assert(PER * SLOT >= G_::X && ON % kWarps == 0, "a warp's result fits its ring slots");
            float4* mine = result_of(warp);
#pragma unroll
            for (int k = 0; k < ON; ++k) mine[k * 32] = make_float4(o[k][0], o[k][1], o[k][2], o[k][3]);
            mine[ON * 32] = make_float4(m[0], m[1], l[0], l[1]);
            __syncwarp();
            if (lane == 0) mbar_arrive(&ctl->hand[0]);
            ok = __all_sync(0xffffffffu, wait_for(&ctl->hand[0], 0, ctl, a));
            if (!ok) return;
            float4 ml[kWarps];
            float w0[kWarps], w1[kWarps];
#pragma unroll
            for (int w = 0; w < kWarps; ++w) ml[w] = result_of(w)[ON * 32];
            const Weights t = weights_of(ml, w0, w1);
            const float4 tml = make_float4(t.m0, t.m1, t.l0, t.l1);
            constexpr int SHARE = ON / kWarps;                       // column chunks a warp combines
            float4 acc[SHARE];
#pragma unroll
            for (int k = 0; k < SHARE; ++k) {
                acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int w = 0; w < kWarps; ++w) {
                    const float4 v = result_of(w)[(warp * SHARE + k) * 32];
                    acc[k].x += v.x * w0[w]; acc[k].y += v.y * w0[w]; acc[k].z += v.z * w1[w]; acc[k].w += v.w * w1[w];
                }
            }
            const RowStore<D> to{a, H, G, h, pair0, pairs, row_base, lane};
            if constexpr (CL == 1) {
                to.rows(tml, [&](int e, int64_t at, float mx, float sum) {
                    const float inv = sum > 0.f ? 1.f / sum : 0.f;
#pragma unroll
                    for (int k = 0; k < SHARE; ++k) to.chunk(warp * SHARE + k, acc[k], e, at, inv);
                    if (warp == 0) to.lse(at, mx, sum);
                });
            } else {
                float4* give = xbuf + lane;
#pragma unroll
                for (int k = 0; k < SHARE; ++k) give[(warp * SHARE + k) * 32] = acc[k];
                if (warp == 0) give[ON * 32] = tml;
                __syncwarp();
                if (lane < CL) tc5::mbar_arrive_cluster(tc5::map_to_cta(smem_u32(&ctl->x_free), lane));
                ok = __all_sync(0xffffffffu, wait_for_cluster(&ctl->x_free, 0, ctl, a));
                if (!ok) return;
                constexpr int OWN = ON / CL;                         // column chunks a CTA finishes
                for (int k = warp; k < OWN; k += kWarps) {
                    const int c = rank * OWN + k;
                    float4 ml2[CL], v[CL];
                    float u0[CL], u1[CL];
#pragma unroll
                    for (int i = 0; i < CL; ++i) {
                        const uint32_t from = tc5::map_to_cta(smem_u32(give), (uint32_t)i);
                        ml2[i] = tc5::ld_cluster_f4(from + ON * 512);
                        v[i] = tc5::ld_cluster_f4(from + c * 512);
                    }
                    const Weights t2 = weights_of(ml2, u0, u1);
                    float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int i = 0; i < CL; ++i) { r.x += v[i].x * u0[i]; r.y += v[i].y * u0[i]; r.z += v[i].z * u1[i]; r.w += v[i].w * u1[i]; }
                    to.rows(make_float4(t2.m0, t2.m1, t2.l0, t2.l1), [&](int e, int64_t at, float mx, float sum) {
                        to.chunk(c, r, e, at, sum > 0.f ? 1.f / sum : 0.f);
                        if (c == 0) to.lse(at, mx, sum);
                    });
                }
            }
            return;
        }
        const bool have = kWarps - 1 - warp < n;                    // this warp worked on the unit
        float4* x = xbuf + lane;
        if (warp > 0) ok = wait_for(&ctl->hand[warp - 1], un & 1, ctl, a);
        else if (un > 0) ok = wait_for(&ctl->x_free, (un - 1) & 1, ctl, a);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) return;
        if (warp > 0 && have) {
            const float4 ml = x[ON * 32];
            const float n0 = fmaxf(m[0], ml.x), n1 = fmaxf(m[1], ml.y);
            const float f0 = n0 == -INFINITY ? 0.f : n0, f1 = n1 == -INFINITY ? 0.f : n1;
            const float w0 = fast_exp2(m[0] - f0), w1 = fast_exp2(m[1] - f1), x0 = fast_exp2(ml.x - f0), x1 = fast_exp2(ml.y - f1);
            m[0] = n0; m[1] = n1;
            l[0] = l[0] * w0 + ml.z * x0;
            l[1] = l[1] * w1 + ml.w * x1;
#pragma unroll
            for (int k = 0; k < ON; ++k) {
                if (low_rows) {
                    const float2 v = *reinterpret_cast<const float2*>(x + k * 32);
                    o[k][0] = o[k][0] * w0 + v.x * x0; o[k][1] = o[k][1] * w0 + v.y * x0;
                } else {
                    const float4 v = x[k * 32];
                    o[k][0] = o[k][0] * w0 + v.x * x0; o[k][1] = o[k][1] * w0 + v.y * x0;
                    o[k][2] = o[k][2] * w1 + v.z * x1; o[k][3] = o[k][3] * w1 + v.w * x1;
                }
            }
        }
        if (have || warp == 0) {
#pragma unroll
            for (int k = 0; k < ON; ++k) {
                if (low_rows) *reinterpret_cast<float2*>(x + k * 32) = make_float2(o[k][0], o[k][1]);
                else x[k * 32] = make_float4(o[k][0], o[k][1], o[k][2], o[k][3]);
            }
            x[ON * 32] = make_float4(m[0], m[1], l[0], l[1]);
        }
        if (warp == kWarps - 1 && lane == 0) {
            ctl->job[0] = make_int4(r1.w, r2.x, r2.y + hs, row_base);
            ctl->job[1] = make_int4(C, pair0, pairs, h);
            ctl->job[2] = make_int4(part, 0, 0, 0);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&ctl->hand[warp]);
    }
}

template <bool BF16, int D>
__global__ void __launch_bounds__(kThreads, kCtasPerSm)
attn_stream_kernel(const __grid_constant__ AttnArgs a, const StreamItem* __restrict__ items, int n_sub, int total_units, int32_t* __restrict__ work_counter,
                   int32_t* __restrict__ piece_counters, const __grid_constant__ CUtensorMap map_k,
                   const __grid_constant__ CUtensorMap map_v) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    stream_roles<BF16, D, 0>(a, smem, items, n_sub, total_units, work_counter, piece_counters, map_k, map_v);
    __syncthreads();
    if (ctl_of<D>(smem)->abort_flag) tc5::settle();
}

constexpr int kShortThreads = kWarps * 32 + 32;       // no output warp

template <bool BF16, int D, int CL>
__global__ void __launch_bounds__(kShortThreads, kCtasPerSm)
attn_stream_short_kernel(const __grid_constant__ AttnArgs a, const StreamItem* __restrict__ items, int n_sub, int total_units,
                         const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    stream_roles<BF16, D, CL>(a, smem, items, n_sub, total_units, nullptr, nullptr, map_k, map_v);
    __syncthreads();
    if (ctl_of<D>(smem)->abort_flag) tc5::settle();
    if constexpr (CL > 1) {
        tc5::cluster_arrive();                                    // the other CTAs have read what they need of this one's shared memory
        tc5::cluster_wait();
    }
}

template <bool BF16, int D>
cudaError_t launch_short(const hat_plan* plan, const AttnArgs& args, const CUtensorMap& mk, const CUtensorMap& mv, cudaStream_t stream) {
    using G_ = Geo<D>;
    constexpr int smem = 1024 + G_::SLOTS * G_::SLOT + G_::Q + G_::X + (int)sizeof(Ctl<G_::SLOTS>);
    const int cl = plan->short_cluster, units = (int)plan->short_items.size() * plan->num_kv_heads * plan->verify_subtiles;
    auto kern = cl == 1 ? attn_stream_short_kernel<BF16, D, 1> : cl == 2 ? attn_stream_short_kernel<BF16, D, 2>
                : cl == 4 ? attn_stream_short_kernel<BF16, D, 4> : attn_stream_short_kernel<BF16, D, 8>;
    cudaError_t e = smem_attr_once(reinterpret_cast<const void*>(kern), smem);
    if (e != cudaSuccess) return e;
    return launch_pdl_clusters(cl, kern, dim3((unsigned)(units * cl)), dim3(kShortThreads), smem, stream, args, plan->dev.short_items,
                               plan->verify_subtiles, units, mk, mv);
}

template <bool BF16, int D>
cudaError_t launch_one(const hat_plan* plan, const AttnArgs& args, const CUtensorMap& mk, const CUtensorMap& mv, cudaStream_t stream) {
    using G_ = Geo<D>;
    constexpr int smem = 1024 + G_::SLOTS * G_::SLOT + G_::Q + G_::X + (int)sizeof(Ctl<G_::SLOTS>);
    static_assert(smem <= 115712, "two CTAs share an SM");
    auto kern = attn_stream_kernel<BF16, D>;
    cudaError_t e = smem_attr_once(reinterpret_cast<const void*>(kern), smem);
    if (e != cudaSuccess) return e;
    const int units = (int)plan->stream_items.size() * plan->num_kv_heads * plan->verify_subtiles;
    return launch_pdl(kern, dim3((unsigned)std::min(units, kCtasPerSm * plan->num_sms)), dim3(kThreads), smem, stream, args,
                      plan->dev.stream_items, plan->verify_subtiles, units, plan->dev.status + 5, plan->dev.piece_counters, mk, mv);
}

}  // namespace

bool stream_layout_supported(int dtype, int head_dim, int num_pages, int H, int64_t stride_page, int64_t stride_token,
                             int64_t stride_head) {
    CUtensorMap m;
    // the encoder checks alignment and ranges only; any 16-byte aligned address will do for the probe
    return tma_encode_page_map(&m, dtype == HAT_DTYPE_BF16, reinterpret_cast<const void*>(uintptr_t(1) << 30), head_dim,
                               num_pages, H, stride_page, stride_token, stride_head);
}

cudaError_t launch_attn_stream(const hat_plan* plan, const AttnArgs& args, cudaStream_t stream) {
    const bool bf16 = plan->dtype == HAT_DTYPE_BF16;
    const CUtensorMap *mk = nullptr, *mv = nullptr;
    if (!plan_page_maps(plan, args.cache, &mk, &mv)) return cudaErrorInvalidValue;
    auto go = [&](auto b, auto d) -> cudaError_t {
        constexpr bool B = decltype(b)::value;
        constexpr int D = decltype(d)::value;
        return plan->short_cluster > 0 ? launch_short<B, D>(plan, args, *mk, *mv, stream) : launch_one<B, D>(plan, args, *mk, *mv, stream);
    };
    using I128 = std::integral_constant<int, 128>;
    using I64 = std::integral_constant<int, 64>;
    if (plan->head_dim == 128) return bf16 ? go(std::true_type{}, I128{}) : go(std::false_type{}, I128{});
    return bf16 ? go(std::true_type{}, I64{}) : go(std::false_type{}, I64{});
}

}  // namespace hat
