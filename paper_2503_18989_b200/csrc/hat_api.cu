// C ABI of the library: status strings, host-side validation and scheduling (the plan), and the
// entry points that enqueue the kernels.  Declarations and argument contracts are in include/hat.h.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>
#include <limits>
#include <queue>

#include "hat_internal.h"
#include "tma_desc.h"

namespace hat {

static thread_local int g_last_cuda_error = 0;
static std::atomic<int64_t> g_launches{0};

void count_launch(int n) { g_launches.fetch_add(n, std::memory_order_relaxed); }
void set_last_cuda_error(int e) { g_last_cuda_error = e; }

cudaError_t smem_attr_once(const void* kernel, int bytes) {
    struct Done { const void* kernel; int device; };
    static std::mutex mu;
    static std::vector<Done> done;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    for (const Done& d : done)
        if (d.kernel == kernel && d.device == dev) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) done.push_back(Done{kernel, dev});
    return e;
}

bool plan_pool_maps(const hat_plan* plan, const CacheView& c, const CUtensorMap** mk, const CUtensorMap** mv) {
    MapCache& m = const_cast<hat_plan*>(plan)->maps;
    if (!m.have_kv || m.k != c.k_pool || m.v != c.v_pool || m.stride_page != c.stride_page ||
        m.stride_token != c.stride_token || m.stride_head != c.stride_head) {
        const bool bf16 = plan->dtype == HAT_DTYPE_BF16;
        m.have_kv = false;
        if (!tma_encode_pool_map(&m.mk, bf16, c.k_pool, plan->head_dim, plan->num_pages, plan->num_kv_heads, c.stride_page,
                                 c.stride_token, c.stride_head) ||
            !tma_encode_pool_map(&m.mv, bf16, c.v_pool, plan->head_dim, plan->num_pages, plan->num_kv_heads, c.stride_page,
                                 c.stride_token, c.stride_head))
            return false;
        m.k = c.k_pool; m.v = c.v_pool;
        m.stride_page = c.stride_page; m.stride_token = c.stride_token; m.stride_head = c.stride_head;
        m.have_kv = true;
    }
    *mk = &m.mk; *mv = &m.mv;
    return true;
}

bool plan_page_maps(const hat_plan* plan, const CacheView& c, const CUtensorMap** mk, const CUtensorMap** mv) {
    MapCache& m = const_cast<hat_plan*>(plan)->maps;
    if (!m.have_page || m.page_k != c.k_pool || m.page_v != c.v_pool || m.page_strides[0] != c.stride_page ||
        m.page_strides[1] != c.stride_token || m.page_strides[2] != c.stride_head) {
        const bool bf16 = plan->dtype == HAT_DTYPE_BF16;
        m.have_page = false;
        if (!tma_encode_page_map(&m.mpk, bf16, c.k_pool, plan->head_dim, plan->num_pages, plan->num_kv_heads, c.stride_page,
                                 c.stride_token, c.stride_head) ||
            !tma_encode_page_map(&m.mpv, bf16, c.v_pool, plan->head_dim, plan->num_pages, plan->num_kv_heads, c.stride_page,
                                 c.stride_token, c.stride_head))
            return false;
        m.page_k = c.k_pool; m.page_v = c.v_pool;
        m.page_strides[0] = c.stride_page; m.page_strides[1] = c.stride_token; m.page_strides[2] = c.stride_head;
        m.have_page = true;
    }
    *mk = &m.mpk; *mv = &m.mpv;
    return true;
}

bool plan_tile_maps(const hat_plan* plan, const CacheView& c, const CUtensorMap** mk, const CUtensorMap** mv, int* fold) {
    MapCache& m = const_cast<hat_plan*>(plan)->maps;
    if (!m.have_tile || m.tile_k != c.k_pool || m.tile_v != c.v_pool || m.tile_strides[0] != c.stride_page ||
        m.tile_strides[1] != c.stride_token || m.tile_strides[2] != c.stride_head) {
        const bool bf16 = plan->dtype == HAT_DTYPE_BF16;
        m.have_tile = false;
        if (!tma_encode_tile_map(&m.mtk, bf16, c.k_pool, plan->head_dim, plan->num_pages, plan->num_kv_heads, c.stride_page,
                                 c.stride_token, c.stride_head, &m.tile_fold) ||
            !tma_encode_tile_map(&m.mtv, bf16, c.v_pool, plan->head_dim, plan->num_pages, plan->num_kv_heads, c.stride_page,
                                 c.stride_token, c.stride_head, &m.tile_fold))
            return false;
        m.tile_k = c.k_pool; m.tile_v = c.v_pool;
        m.tile_strides[0] = c.stride_page; m.tile_strides[1] = c.stride_token; m.tile_strides[2] = c.stride_head;
        m.have_tile = true;
    }
    *mk = &m.mtk; *mv = &m.mtv; *fold = m.tile_fold;
    return true;
}

bool plan_new_maps(const hat_plan* plan, const void* k_new, const void* v_new, const CUtensorMap** mk, const CUtensorMap** mv,
                   const CUtensorMap** mv_half) {
    MapCache& m = const_cast<hat_plan*>(plan)->maps;
    if (k_new && (!m.have_new || m.k_new != k_new || m.v_new != v_new)) {
        const bool bf16 = plan->dtype == HAT_DTYPE_BF16;
        const int T = plan->total_rows, H = plan->num_kv_heads, d = plan->head_dim;
        m.have_new = false;
        if (!tma_encode_new_map(&m.mkn, bf16, k_new, T, H, d, 8, d / 64) || !tma_encode_new_map(&m.mvn, bf16, v_new, T, H, d, 8, d / 64) ||
            !tma_encode_new_map(&m.mvn_half, bf16, v_new, T, H, d, kPageSize, 1))
            return false;
        m.k_new = k_new; m.v_new = v_new;
        m.have_new = true;
    }
    *mk = k_new ? &m.mkn : &m.mq;
    *mv = k_new ? &m.mvn : &m.mq;
    *mv_half = k_new ? &m.mvn_half : &m.mq;
    return true;
}

const CUtensorMap* plan_q_map(const hat_plan* plan, const void* q) {
    MapCache& m = const_cast<hat_plan*>(plan)->maps;
    if (!m.have_q || m.q != q) {
        m.have_q = false;
        if (!tma_encode_q_map(&m.mq, plan->dtype == HAT_DTYPE_BF16, q, plan->total_rows, plan->num_heads, plan->head_dim)) return nullptr;
        m.q = q;
        m.have_q = true;
    }
    return &m.mq;
}

static int cuda_fail(cudaError_t e) {
    g_last_cuda_error = (int)e;
    return HAT_ERR_CUDA;
}

static int env_int(const char* name, int dflt) {
    const char* s = std::getenv(name);
    if (!s || !*s) return dflt;
    char* end = nullptr;
    long v = std::strtol(s, &end, 10);
    return (end && *end == 0) ? (int)v : dflt;
}

static inline int round_up(int x, int m) { return (x + m - 1) / m * m; }
static inline int ceil_div(int x, int m) { return (x + m - 1) / m; }

static int check_cache_geometry(const hat_cache_desc* c) {
    if (!c) return HAT_ERR_INVALID_ARG;
    if (c->num_pages < 0) return HAT_ERR_INVALID_ARG;
    if (c->dtype != HAT_DTYPE_FP16 && c->dtype != HAT_DTYPE_BF16) return HAT_ERR_UNSUPPORTED;
    if (c->page_size != kPageSize) return HAT_ERR_UNSUPPORTED;
    if (c->head_dim != 64 && c->head_dim != 128) return HAT_ERR_UNSUPPORTED;
    if (c->num_kv_heads <= 0) return HAT_ERR_INVALID_ARG;
    if (c->stride_page <= 0 || c->stride_token <= 0 || c->stride_head <= 0) return HAT_ERR_INVALID_ARG;
    if (c->stride_page % 8 || c->stride_token % 8 || c->stride_head % 8) return HAT_ERR_UNSUPPORTED;
    return HAT_OK;
}

static bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

// Cut the key range [0, kv_end) of one tile into pieces of `split_len` keys (the last piece takes the
// remainder) and emit one work item per piece.
static void emit_tile(hat_plan* p, std::vector<WorkItem>& items, int req, int row0, int rows_valid,
                      int kv_end, int split_len) {
    int nsplit = (split_len > 0) ? ceil_div(kv_end, split_len) : 1;
    if (nsplit <= 1) {
        items.push_back(WorkItem{req, row0, 0, kv_end, -1, p->prefix_len[req], p->chunk_len[req], p->cu_chunk[req]});
        return;
    }
    int64_t base = p->part_rows;
    for (int s = 0; s < nsplit; ++s) {
        int b = s * split_len, e = std::min(kv_end, b + split_len);
        items.push_back(WorkItem{req, row0, b, e, (int32_t)(base + (int64_t)s * rows_valid), p->prefix_len[req], p->chunk_len[req], p->cu_chunk[req]});
    }
    int row_base = p->cu_chunk[req] + row0;
    for (int i = 0; i < rows_valid; ++i)
        p->merge_rows.push_back(MergeRow{row_base + i, (int32_t)(base + i), rows_valid, nsplit});
    p->part_rows += (int64_t)nsplit * rows_valid;
    p->info.max_splits = std::max(p->info.max_splits, nsplit);
}

static int split_len_for(int kv_end, int wanted, int granule) {
    // at most kMaxSplits pieces per tile
    int least = round_up(ceil_div(kv_end, kMaxSplits), granule);
    return std::max(wanted, least);
}

// Whether the two halves of every cut tile are merged inside the one-CTA tile kernel, by clusters of two CTAs: every tile is
// cut in two, has at most 128 rows, and the pieces are one round of the CTAs.  (Side by side with another grid on one
// counter, HAT_SIDE_SMS, a unit has no CTA of its own.)  With 64 columns the merge behind is short, and with few CTAs it is the
// cheaper one: prompts of 2048 in chunks of 256, launch / clusters, 32 heads fp16 140 / 118 us, bf16 147 / 127, but 8 heads 2 to 5 % more.
static bool pieces_meet_in_clusters(const hat_plan* p, int num_sms, int64_t units, bool all_in_two, bool all_narrow) {
    return (p->head_dim == 128 || units >= num_sms / 2) && all_in_two && all_narrow && units <= num_sms / 2 * 2 && env_int("HAT_SIDE_SMS", 0) <= 0;
}

// ns that a unit takes a CTA of the one-CTA tile kernel: its 128-key steps, two query tiles or one, and what does not depend on the keys (the
// Q tiles, refilling the rings, the rows).  Fitted to 1, 2 and 3 rounds of equal units, 256 to 3072 keys.
static int64_t tile_unit_ns(const hat_plan* p, int keys, int rows) {
    const bool bf16 = p->dtype == HAT_DTYPE_BF16, d128 = p->head_dim == 128;
    const int wide = d128 ? (bf16 ? 3100 : 2400) : (bf16 ? 2480 : 2000), narrow = d128 ? (bf16 ? 1780 : 1450) : (bf16 ? 1350 : 1020);
    return (int64_t)ceil_div(keys, 128) * (rows > 128 ? wide : narrow) + (d128 && rows > 128 ? 6000 : 4000);
}

// When the last of n units ends that CTAs draw in order.
template <typename F>
static int64_t last_end(int ctas, int n, F&& ns_of) {
    std::vector<int64_t> at(ctas, 0);                            // a heap: when each CTA is free, the first one in front
    int64_t last = 0;
    for (int i = 0; i < n; ++i) {
        const int64_t t = at[0] + ns_of(i);
        int k = 0;
        for (int c = 1; c < ctas; c = 2 * k + 1) {
            c += c + 1 < ctas && at[c + 1] < at[c];
            if (at[c] >= t) break;
            at[k] = at[c];
            k = c;
        }
        at[k] = t;
        last = std::max(last, t);
    }
    return last;
}

// Key-range length for the tile-class requests of a batch that is too small to fill the persistent tcgen05 kernel.
// Every candidate length is priced with a small model of the one-CTA kernel (also for batches of the pair kernel, whose 74 pairs
// take 2350 to 2720 cycles a step: the model is only a rough guide there), in SM clock cycles measured on B200: a 128-key
// step of a 256-row unit (two query tiles) or of a unit of at most 128 rows (two chains share it), the fixed cost of a
// unit (its Q tiles, refilling the rings, storing its rows), and the merge pass (its launch plus reading every partial
// row).  Units go to the CTAs longest first, as the kernel draws them.  Returns 0 for "leave every request whole".
// `tile_rows` says how many rows a unit may have; given 0, both forms are priced and it is set to the cheaper one's: units of
// 128 rows take about as long per row and key, and twice as many units need half as many key ranges, that is less to merge or
// nothing, and two ranges are merged by clusters (one request of 256 rows x 32 heads, fp16, us with units of 256 / 128 rows: prefix
// 0 11.4 / 8.7, 512 18.0 / 12.5, 1280 20.7 / 15.5, 4000 40.6 / 32.3; 512 rows at 1000 31.6 / 23.3; but two of 200 rows x 40
// heads at 500, where 128-row units need a second round, 21.9 / 25.5).
static int pick_prefill_split(const hat_plan* p, int num_sms, int* tile_rows, int key_granule, bool clusters) {
    constexpr int64_t kStepWide = 4000, kStepNarrow = 2200, kUnit = 10000, kMergeLaunch = 5700, kMergeCluster = 2500;
    constexpr int64_t kMergeBytesPerCycle = 3000;
    struct Tile { int keys, rows; };
    std::vector<Tile> tiles;
    int max_keys = 0;
    auto cut_rows = [&](int unit_rows) {
        tiles.clear();
        for (int r = 0; r < p->num_requests; ++r) {
            const int C = p->chunk_len[r];
            if (C <= 16) continue;
            for (int row0 = 0; row0 < C; row0 += unit_rows) {
                const int rows = std::min(unit_rows, C - row0);
                tiles.push_back(Tile{p->prefix_len[r] + row0 + rows, rows});
                max_keys = std::max(max_keys, tiles.back().keys);
            }
        }
    };
    const int H = p->num_heads;
    std::vector<int64_t> units;
    auto price = [&](int len, int64_t least) -> int64_t {      // exact only below `least`
        units.clear();
        int64_t part_rows = 0, work = 0;
        bool in_two = clusters, narrow = true;
        for (const Tile& t : tiles) {
            const int sl = len > 0 ? split_len_for(t.keys, len, key_granule) : t.keys;
            const int n = ceil_div(t.keys, sl);
            if (n > 1) part_rows += (int64_t)n * t.rows;
            in_two &= n == 2; narrow &= t.rows <= 128;
            for (int s = 0; s < n; ++s) {
                const int keys = std::min(t.keys, (s + 1) * sl) - s * sl;
                units.push_back(ceil_div(keys, 128) * (t.rows > 128 ? kStepWide : kStepNarrow) + kUnit);
                work += units.back();
            }
        }
        const int64_t merge = pieces_meet_in_clusters(p, num_sms, (int64_t)units.size() * H, in_two, narrow) ? kMergeCluster
                              : part_rows > 0 ? kMergeLaunch + part_rows * H * (p->head_dim + 1) * 4 / kMergeBytesPerCycle : 0;
        std::sort(units.begin(), units.end(), std::greater<int64_t>());
        if ((int64_t)units.size() * H <= num_sms) return units[0] + merge;
        if (work * H / num_sms + merge >= least) return least;
        std::priority_queue<int64_t, std::vector<int64_t>, std::greater<int64_t>> sms;
        for (int i = 0; i < num_sms; ++i) sms.push(0);
        int64_t makespan = 0;
        for (int h = 0; h < H; ++h) {
            for (int64_t u : units) {
                const int64_t t = sms.top() + u;
                sms.pop();
                sms.push(t);
                makespan = std::max(makespan, t);
            }
        }
        return makespan + merge;
    };
    int best = 0, best_rows = *tile_rows;
    int64_t best_cost = std::numeric_limits<int64_t>::max();
    for (int unit_rows : {256, 128}) {
        if (*tile_rows != 0 && unit_rows != *tile_rows) continue;
        cut_rows(unit_rows);
        for (int len = 0; len < max_keys; len += (len == 0 ? 256 : len < 1024 ? 128 : len < 4096 ? 512 : 2048)) {
            const int64_t c = price(len, best_cost);
            if (c < best_cost) { best_cost = c; best = len; best_rows = unit_rows; }
        }
    }
    *tile_rows = best_rows;
    return best;
}

// Key-range length for the streaming-class requests.  The kernel is persistent (two CTAs per SM, units of one piece x one
// head drawn longest first) and as long as HBM is the limit whole requests are best, however uneven: what remains when the
// short ones are done still has enough bytes in flight.  A cut costs: the partial rows, a fence and a count per piece and the
// merge (measured: 12 requests x 32 heads 46 us whole, 50 us in 512-key ranges; 30 requests 151 / 160 us in 768-key ranges).
// So requests are cut only when the longest one alone would take longer than HBM needs for the batch, and then into as
// many pieces as the CTAs can take in one round, or in one more round than the whole requests need (16 requests x 8 K/V heads
// x 2 slabs: 124 us whole, 95 us in 400 units, 93 us in 576, 89 us in 1000, 99 us in 1900).
static int pick_verify_split_slabs(const hat_plan* p, int num_sms, double* price_us);
static int pick_verify_split(const hat_plan* p, int num_sms, double* slabs_price) {
    if (p->verify_subtiles > 1) return pick_verify_split_slabs(p, num_sms, slabs_price);
    constexpr int kWhole = 1 << 24, kLeast = 96;       // shorter pieces than 6 pages only add to the merge
    const double tp = 0.25 * p->head_dim / 128;   // us per page of a CTA that has the SM's share of HBM to itself
    const double tb = p->head_dim * 64 / 6.45e6;                               // us per page (K and V) at the measured HBM rate
    constexpr double kCut = 3.0;                       // us
    const int64_t heads = (int64_t)p->num_kv_heads * p->verify_subtiles;
    const int64_t slots = 2 * (int64_t)num_sms;
    int64_t pages = 0, whole_units = 0;
    int longest = 0;
    for (int r = 0; r < p->num_requests; ++r) {
        if (p->chunk_len[r] < 1 || p->chunk_len[r] > 16) continue;
        const int n = p->prefix_len[r] + p->chunk_len[r];
        pages += ceil_div(n, kPageSize) + 1;
        longest = std::max(longest, n);
        ++whole_units;
    }
    pages *= heads; whole_units *= heads;
    auto time_of = [&](int keys) { return std::max((ceil_div(keys, kPageSize) + 1) * tp, pages * tb); };
    if (time_of(longest) <= pages * tb + kCut) return kWhole;
    const int64_t most = 2 * whole_units <= slots ? slots : whole_units + slots;
    auto units_at = [&](int len) {
        int64_t n = 0;
        for (int r = 0; r < p->num_requests; ++r)
            if (p->chunk_len[r] >= 1 && p->chunk_len[r] <= 16) {
                const int keys = p->prefix_len[r] + p->chunk_len[r];
                n += ceil_div(keys, split_len_for(keys, len, kPageSize));
            }
        return n * heads;
    };
    int lo = kLeast / kPageSize, hi = std::max(lo, ceil_div(longest, kPageSize));
    while (lo < hi) {
        const int mid = (lo + hi) / 2;
        if (units_at(mid * kPageSize) <= most) hi = mid; else lo = mid + 1;
    }
    return time_of(lo * kPageSize) + kCut < time_of(longest) ? lo * kPageSize : kWhole;
}

// The same for batches with more than one slab of 16 pairs a K/V head.  There mma.sync is the limit, not HBM: a page takes a slab
// about the same time however many CTAs run, so what counts is how evenly the units fill the CTAs.  Every candidate
// length (the longest request in 1, 1.5, 2 ... 8 pieces) is priced by placing its units, longest first, on the CTAs; all heads of a piece are
// alike, so as many as divide evenly are placed as one.  Measured, us, rule above / this, bf16: 16 requests of 1300 to 7800 tokens x 8 K/V
// heads x 16..32 pairs 92.4 / 86.3, 10 x 16 heads 119.7 / 91.2, 12 of up to 2048 tokens 33.1 / 27.4, 16 x 8 heads x 8..64 pairs 129.2 /
// 103.7, 8 x 8 heads 51.9 / 52.8.
static int pick_verify_split_slabs(const hat_plan* p, int num_sms, double* price_us) {
    const double page = 0.26 * p->head_dim / 128, unit = 0.8, cut = 3.0;       // us: a page, a unit, a piece of a cut request
    const int group = p->num_heads / p->num_kv_heads;
    int alike = 1;
    for (int g = 2; g <= 8; ++g) if (p->num_kv_heads % g == 0) alike = g;
    const int copies = p->num_kv_heads / alike, slots = std::max(1, 2 * num_sms / alike);
    int longest = 0;
    for (int r = 0; r < p->num_requests; ++r)
        if (p->chunk_len[r] >= 1 && p->chunk_len[r] <= 16) longest = std::max(longest, p->prefix_len[r] + p->chunk_len[r]);
    std::vector<double> times, load;
    auto price = [&](int len) {
        times.clear();
        for (int r = 0; r < p->num_requests; ++r) {
            const int C = p->chunk_len[r];
            if (C < 1 || C > 16) continue;
            const int keys = p->prefix_len[r] + C, n = ceil_div(keys, split_len_for(keys, len, kPageSize));
            const int pages = ceil_div(p->prefix_len[r], kPageSize) + 1;
            times.insert(times.end(), (size_t)n * copies * ceil_div(C * group, 16), (double)pages / n * page + unit + (n > 1 ? cut : 0.0));
        }
        std::sort(times.begin(), times.end(), std::greater<double>());
        load.assign(slots, 0.0);                                       // a heap, least loaded first
        double most = 0.0;
        for (double t : times) {
            std::pop_heap(load.begin(), load.end(), std::greater<double>());
            load.back() += t;
            most = std::max(most, load.back());
            std::push_heap(load.begin(), load.end(), std::greater<double>());
        }
        return most;
    };
    int best = 1 << 24;
    double least = price(best);
    for (int halves = 3; halves <= 16; ++halves) {
        const int len = std::max(96, round_up(ceil_div(2 * longest, halves), kPageSize));
        const double t = price(len);
        if (t < 0.98 * least) { least = t; best = len; }
        if (len == 96) break;
    }
    *price_us = least;
    return best;
}

// Whether every unit of the streaming class gets a CTA of its own (the short form of the streaming kernel), and in how many pieces a request is
// cut then: 1, 2, 4 or 8, the CTAs of a cluster; 0: the persistent kernel takes the pieces planned above.  HAT_VERIFY_CLUSTER overrides.
// A page takes a CTA 0.20 us (bf16; fp16 0.17; 64 columns 0.75 of that; 15 % more with two CTAs on an SM), start, hand-over and rows about 5, the exchange within a cluster
// 1.4 to 2.4.  The persistent kernel needs HBM's time and 7 us or more, 12 at least (fence, count and merge of the pieces), or what the placing of
// its slabs said and 5.  It keeps what it may do as fast: batches whose longest request is much longer than the others, which it cuts unevenly.
// Measured, us, persistent / short, bf16: one request x 32 heads 200 tokens 9.2 / 7.0, 700 11.2 / 8.9, 3000 15.8 / 14.2, 8000 30.5 /
// 27.8; x 8 heads of 4 700 12.8 / 7.8, 3000 20.1 / 11.8; two of 500 to 2000 x 32 15.0 / 14.2; 9 x 32 41.1 / 38.8; 64 columns: 700 x 8 9.3 / 6.0; where
// it is not taken: 3 of up to 4096 x 32 32.2 / 33.8, one of 3000 x 40 16.3 / 18.2, 7 of up to 8192 x 8 heads of 4 39.6 / 62.8.
static int pick_short_cluster(const hat_plan* p, int num_sms, double slabs_price) {
    const bool d128 = p->head_dim == 128;
    int64_t units = 0, pages = 0;
    int longest = 0;
    for (int r = 0; r < p->num_requests; ++r) {
        if (p->chunk_len[r] < 1 || p->chunk_len[r] > 16) continue;
        const int n = ceil_div(p->prefix_len[r], kPageSize) + 1;
        units += (int64_t)p->num_kv_heads * p->verify_subtiles;
        pages += (int64_t)n * p->num_kv_heads;
        longest = std::max(longest, n);
    }
    if (units == 0) return 0;
    const int forced = env_int("HAT_VERIFY_CLUSTER", -1);
    if (forced == 0) return 0;
    if ((forced == 1 || forced == 2 || forced == 4 || forced == 8) && units * forced <= 65535) return forced;
    const double page = (p->dtype == HAT_DTYPE_BF16 ? 0.203 : 0.168) * (d128 ? 1.0 : 0.75), hbm = (double)pages * p->head_dim * 64 / 6.45e6;
    const double exchange[4] = {0.0, d128 ? 1.4 : 0.8, d128 ? 2.1 : 1.0, d128 ? 2.4 : 1.1};
    int best = 0;
    double least = p->verify_subtiles > 1 ? slabs_price + 5.0 : std::max(hbm + 7.0, d128 ? 12.0 : 10.0);
    // With prompt chunks behind, whose CTAs take the SMs the drafts leave, cut requests may be priced up to a quarter higher: the model knows the
    // drafts alone.  Of 24 such batches that this decides, short / persistent, geometric means: step 0.93, drafts' rows final 0.93 (at most 1.08
    // and 1.04; 6 chunks and 3 drafts x 8 heads of 4 51.8 / 58.4 and 18.4 / 22.5 us).  Uncut ones keep the plain price: with lengths
    // far apart a CTA each is later (10 requests x 40 heads, up to 5545 tokens, drafts 86 / 72, step 99 / 92).
    const double above = p->info.num_prefill_requests > 0 ? 1.25 : 1.0;
    const bool whole = (int64_t)p->stream_items.size() * p->num_kv_heads * p->verify_subtiles == units && p->verify_subtiles == 1;
    for (int i = 0; i < 4; ++i) {
        const int64_t ctas = units << i;
        // clusters of 4 and 8 do not fill every SM of a GPC: a second round would follow
        if (ctas > 2 * (int64_t)num_sms || (i > 1 && ctas > (int64_t)num_sms * 256 / 148)) break;
        const bool two = ctas > num_sms;
        const double t = std::max(hbm + 6.5, (d128 ? 5.0 : 4.0) + page * (two ? 1.15 : 1.0) * ceil_div(longest, 1 << i) + exchange[i] + (two ? 1.2 : 0.0));
        const double beat = best > 0 ? least : least * (i < 3 ? 0.97 : 1.0) * (i > 0 ? above : 1.0);
        // requests that the persistent kernel would not cut are never slower with a CTA each
        if ((hbm < 60.0 && t < beat) || (whole && i == 0)) { least = t; best = 1 << i; }
    }
    return best;
}

// Whether the chunk's rows are appended by a kernel in front of the one-CTA tile kernel instead of inside it.  Inside, the append costs
// no launch and no second read, but the instructions for it crowd the kernel's loops out of the instruction cache and its producer
// works on units with chunk pages longer; in front, it costs a launch and the bytes once more.  So in front where CTAs have
// several units each and a unit is short work: 64 columns, or on average at most one query tile.  Measured, us inside / in front, fp16, 32
// heads: 30 chunks of 32 to 128 rows at up to 1024 114 / 93, 64 columns 84 / 68; 30 of 64 to 512 at up to 4096 401 / 419, 64 columns
// 311 / 307; 8 heads, 64 columns 23.0 / 23.5.  The CTA-pair kernel, whose loops are smaller, appends inside (30 chunks, bf16, 433 / 441).
static bool append_is_apart(const hat_plan* p, int num_sms, int tile_rows) {
    int64_t tiles = 0, rows = 0;
    for (int r = 0; r < p->num_requests; ++r)
        if (p->chunk_len[r] > 16) { tiles += ceil_div(p->chunk_len[r], tile_rows); rows += p->chunk_len[r]; }
    return tiles * p->num_heads > 2 * (int64_t)num_sms && (p->head_dim == 64 || rows <= 128 * tiles);
}

// tile_kernel: 0 = mma.sync, 1 = tcgen05 with two query tiles per CTA, 3 = tcgen05 by pairs of CTAs (cta_group::2) with a
// ring of three score buffers; both tcgen05 kernels take 256-row units
static void schedule(hat_plan* p, int num_sms, int tile_kernel, bool whole) {
    const bool use_tc5 = tile_kernel != 0;
    const int H = p->num_heads;
    const int R = p->num_requests;
    hat_plan_info& info = p->info;

    const int verify_max_rows = 16;
    // tile kernel: tcgen05 with 256-row tiles (two 128-row MMA tiles) and 128-key steps, or mma.sync with 4 warps x 16 rows and 64-key steps
    int tile_rows = use_tc5 ? 256 : 64;
    const int key_granule = use_tc5 ? 128 : 64;
    info.prefill_kernel = tile_kernel;

    // ---- streaming (verify-class) requests: key ranges of one length.
    // A CTA of the streaming kernels serves one K/V head and a slab of (row, query head of the group) pairs.
    const int group = H / p->num_kv_heads;
    int max_verify_rows = 0;
    for (int r = 0; r < R; ++r) {
        int C = p->chunk_len[r];
        if (C >= 1 && C <= verify_max_rows) {
            info.num_verify_requests++;
            max_verify_rows = std::max(max_verify_rows, C);
        } else if (C > verify_max_rows) {
            info.num_prefill_requests++;
        }
    }
    const bool stream_tma = info.stream_kernel != 0;
    p->verify_subtiles = std::max(1, ceil_div(max_verify_rows * group, 16));
    int vsplit = env_int("HAT_VERIFY_SPLIT_LEN", 0);
    double slabs_price = 1e9;
    if (whole) vsplit = 1 << 24;
    else if (vsplit <= 0) vsplit = pick_verify_split(p, num_sms, &slabs_price);
    vsplit = std::max(kPageSize, round_up(vsplit, kPageSize));
    info.verify_split_len = vsplit;

    // ---- tile (prefill-class) requests: cut keys only when there are too few tiles to cover the SMs
    int64_t tiles = 0, tile_keys = 0;
    for (int r = 0; r < R; ++r) {
        int C = p->chunk_len[r];
        if (C <= verify_max_rows) continue;
        for (int row0 = 0; row0 < C; row0 += tile_rows) {
            tiles++;
            tile_keys += p->prefix_len[r] + std::min(C, row0 + tile_rows);
        }
    }
    int psplit = whole ? 0 : env_int("HAT_PREFILL_SPLIT_LEN", -1);
    int want_rows = tile_kernel == 1 && !whole ? env_int("HAT_PREFILL_TILE_ROWS", 0) : tile_rows;   // 0: whichever is cheaper
    if (want_rows != 128 && want_rows != 0) want_rows = tile_rows;
    if (psplit < 0) {
        psplit = 0;
        const int64_t want_ctas = (int64_t)num_sms * 2;
        if (tiles > 0 && tiles * H < want_ctas && use_tc5) {
            psplit = pick_prefill_split(p, num_sms, &want_rows, key_granule, tile_kernel == 1);
        } else if (tiles > 0 && tiles * H < want_ctas) {
            // aim for want_ctas pieces of equal length, not shorter than 256 keys
            const int pieces = ceil_div((int)want_ctas, H);
            psplit = std::max(256, round_up((int)((tile_keys + pieces - 1) / pieces), key_granule));
        }
    }
    if (psplit > 0) psplit = round_up(psplit, key_granule);
    info.prefill_split_len = psplit;
    if (want_rows > 0) tile_rows = want_rows;
    info.prefill_tile_rows = tile_rows;

    int stream_merged = 0;                  // rows the streaming kernel merges itself
    // streaming-class requests first: their merge rows form the head of merge_rows, so that they can be merged (and
    // announced through the plan's event) before the tile kernel runs
    for (int r = 0; r < R; ++r) {
        const int C = p->chunk_len[r], P = p->prefix_len[r];
        if (C <= 0 || C > verify_max_rows) continue;
        const int kv_end = P + C;
        const int sl = split_len_for(kv_end, vsplit, kPageSize);
        if (!stream_tma) { emit_tile(p, p->verify_items, r, 0, C, kv_end, sl); continue; }
        // the TMA kernel: as many pieces as ranges of that length, of (nearly) equal size
        const int pieces = ceil_div(kv_end, sl), pages = ceil_div(P, kPageSize) + 1;
        const int32_t part0 = (int32_t)p->part_rows;
        for (int s = 0; s < pieces; ++s)
            p->stream_items.push_back(StreamItem{r, p->cu_chunk[r], C, P, (int)((int64_t)pages * s / pieces), (int)((int64_t)pages * (s + 1) / pieces),
                                                 pieces > 1 ? part0 + s * C : -1, part0, pieces, p->num_piece_counters, 0, 0});
        if (pieces > 1) {
            p->part_rows += (int64_t)pieces * C;
            p->num_piece_counters += p->num_kv_heads * p->verify_subtiles;
            stream_merged += C;
            info.max_splits = std::max(info.max_splits, pieces);
        }
    }
    p->num_verify_merge_rows = (int)p->merge_rows.size();
    p->short_cluster = stream_tma && env_int("HAT_VERIFY_SPLIT_LEN", 0) <= 0 ? pick_short_cluster(p, num_sms, slabs_price) : 0;
    for (int i = 0; i < 4; ++i) if (p->short_cluster == 1 << i) info.stream_kernel = 2 + i;
    if (p->short_cluster > 0)
        for (int r = 0; r < R; ++r) {
            const int C = p->chunk_len[r], P = p->prefix_len[r];
            if (C >= 1 && C <= verify_max_rows) p->short_items.push_back(StreamItem{r, p->cu_chunk[r], C, P, 0, ceil_div(P, kPageSize) + 1, -1, 0, 1, 0, 0, 0});
        }
    int cluster_merged = 0;                 // rows the one-CTA tile kernel merges itself
    auto each_tile = [&](auto&& f) {
        for (int r = 0; r < R; ++r) {
            const int C = p->chunk_len[r];
            if (C <= verify_max_rows) continue;
            for (int row0 = 0; row0 < C; row0 += tile_rows) {
                const int rows_valid = std::min(tile_rows, C - row0), kv_end = p->prefix_len[r] + row0 + rows_valid;
                f(r, row0, rows_valid, kv_end, psplit > 0 ? split_len_for(kv_end, psplit, key_granule) : 0);
            }
        }
    };
    bool in_two = tile_kernel == 1, narrow = true;
    int64_t pieces = 0;
    each_tile([&](int, int, int rows, int kv_end, int sl) {
        in_two &= sl > 0 && ceil_div(kv_end, sl) == 2;
        narrow &= rows <= 128;
        pieces += 2;
    });
    p->tile_clusters = pieces > 0 && pieces_meet_in_clusters(p, num_sms, pieces * H, in_two, narrow);
    p->append_apart = tile_kernel == 1 && append_is_apart(p, num_sms, tile_rows);
    each_tile([&](int r, int row0, int rows, int kv_end, int sl) {
        if (!p->tile_clusters) { emit_tile(p, p->prefill_items, r, row0, rows, kv_end, sl); return; }
        // one piece behind the other: the CTAs of a cluster
        for (int b = 0; b < kv_end; b += sl)
            p->prefill_items.push_back(WorkItem{r, row0, b, std::min(kv_end, b + sl), -1, p->prefix_len[r], p->chunk_len[r], p->cu_chunk[r]});
        cluster_merged += rows;
        info.max_splits = std::max(info.max_splits, 2);
    });
    // longest pieces first so the tail of the grid is made of short ones
    auto longer = [](const WorkItem& a, const WorkItem& b) {
        return (a.kv_end - a.kv_begin) > (b.kv_end - b.kv_begin);
    };
    std::stable_sort(p->verify_items.begin(), p->verify_items.end(), longer);
    std::stable_sort(p->stream_items.begin(), p->stream_items.end(),
                     [](const StreamItem& a, const StreamItem& b) { return a.page1 - a.page0 > b.page1 - b.page0; });
    if (!p->tile_clusters) std::stable_sort(p->prefill_items.begin(), p->prefill_items.end(), longer);

    // Units of the persistent tcgen05 kernels, in the order the CTAs draw them: requests by their longest item first;
    // inside a request head by head, and for each head all items of the request one after the other, so that the row
    // blocks of one chunk (which read the same K/V of that head) run at the same time on neighbouring CTAs and meet in L2.
    p->tile_units.clear();
    p->num_pair_units = 0;
    if (use_tc5) {
        std::vector<int> first_of_req(R, -1);
        std::vector<std::vector<int>> group;
        for (int i = 0; i < (int)p->prefill_items.size(); ++i) {
            const int r = p->prefill_items[i].req;
            if (first_of_req[r] < 0) { first_of_req[r] = (int)group.size(); group.emplace_back(); }
            group[first_of_req[r]].push_back(i);
        }
        // With the CTA-pair kernel in use, units of more than 128 rows come first (they are its); units that would leave
        // half of a pair idle follow and go to the one-CTA kernel.
        auto rows_of = [&](int i) { return std::min(tile_rows, p->chunk_len[p->prefill_items[i].req] - p->prefill_items[i].row0); };
        for (int pass = 0; pass < (tile_kernel == 3 ? 2 : 1); ++pass) {
            for (const std::vector<int>& g : group)      // items are sorted longest first, so groups are too
                for (int h = 0; h < H; ++h)
                    for (int i : g) {
                        if (tile_kernel == 3 && ((rows_of(i) > 128 || p->pair_takes_all) != (pass == 0))) continue;
                        p->tile_units.push_back((uint32_t)i | ((uint32_t)h << 16));
                    }
            if (pass == 0) p->num_pair_units = tile_kernel == 3 ? (int)p->tile_units.size() : 0;
        }
        // Where CTAs have few units each, the batch ends when the CTA with the most work does: then the longest units first, if that ends
        // sooner than request by request (odd chunks, 6 x 40 heads, with rotation and drafts 134 -> 128 us a step; 2 of up to 600 rows x 32 heads fp16 64 -> 59).  With
        // many units a CTA the blocks of a chunk keep together (20 chunks of up to 600 rows x 40 heads bf16 469 / 517).
        const int n = (int)p->tile_units.size();
        if (tile_kernel == 1 && !p->tile_clusters && n > num_sms && n <= 4 * num_sms) {
            std::vector<int64_t> ns;
            std::vector<int> by_time;
            for (int i = 0; i < (int)p->prefill_items.size(); ++i) {
                ns.push_back(tile_unit_ns(p, p->prefill_items[i].kv_end - p->prefill_items[i].kv_begin, rows_of(i)));
                by_time.push_back(i);
            }
            std::stable_sort(by_time.begin(), by_time.end(), [&](int a, int b) { return ns[a] > ns[b]; });
            // looked at with a quarter of the heads on a quarter of the CTAs, where that comes out even: 4 us of planning instead of 17
            const int part = H % 4 == 0 && num_sms % 4 == 0 ? 4 : 1, heads = H / part;
            std::vector<int64_t> by_request;
            for (uint32_t u : p->tile_units)
                if ((int)(u >> 16) < heads) by_request.push_back(ns[u & 0xffff]);
            const int64_t now = last_end(num_sms / part, n / part, [&](int k) { return by_request[k]; });
            if (100 * last_end(num_sms / part, n / part, [&](int k) { return ns[by_time[k / heads]]; }) < 98 * now)
                for (int k = 0; k < n; ++k) p->tile_units[k] = (uint32_t)by_time[k / H] | ((uint32_t)(k % H) << 16);
        }
    }

    info.num_verify_items = (int32_t)(p->verify_items.size() + p->stream_items.size());
    info.num_prefill_items = (int32_t)p->prefill_items.size();
    info.num_merge_rows = (int32_t)p->merge_rows.size() + stream_merged + cluster_merged;
    const int64_t d = p->head_dim;
    int64_t part_out_bytes = p->part_rows * H * d * 4;
    part_out_bytes = (part_out_bytes + 255) / 256 * 256;
    info.workspace_bytes = p->part_rows ? part_out_bytes + ((p->part_rows * H * 4 + 255) / 256 * 256) : 0;
}

int upload_plans(hat_plan* const* plans, size_t count, PlanRes* res) {
    // the arrays of all plans, each at a 256-byte boundary, go over in one copy
    struct Offsets { size_t cu, pl, cl, bt, rr, vi, si, sh, pi, mr, tu, tm, st, table; };
    std::vector<Offsets> at(count);
    std::vector<UploadPart> parts;
    size_t bytes = 0, most_status = 0;
    // status word; (unit counter, finished CTAs) of the tile kernel, of a second tile grid, of the streaming kernel; spare;
    // finished pieces of the requests the streaming kernel merges
    for (size_t i = 0; i < count; ++i) {
        plans[i]->num_status_words = 8 + plans[i]->num_piece_counters;
        most_status = std::max(most_status, (size_t)plans[i]->num_status_words);
    }
    const std::vector<int32_t> status(most_status, 0);
    auto place = [&](const void* src, size_t n) {
        const size_t off = (bytes + 255) / 256 * 256;
        parts.push_back(UploadPart{src, n, off});
        bytes = off + std::max<size_t>(n, 16);
        return off;
    };
    auto add = [&](const auto& v) { return place(v.data(), v.size() * sizeof(v[0])); };
    for (size_t i = 0; i < count; ++i) {
        const hat_plan* p = plans[i];
        at[i] = Offsets{add(p->cu_chunk), add(p->prefix_len), add(p->chunk_len), add(p->block_table), add(p->row_req), add(p->verify_items),
                        add(p->stream_items), add(p->short_items), add(p->prefill_items), add(p->merge_rows), add(p->tile_units), add(p->tree_mask),
                        place(status.data(), p->num_status_words * sizeof(int32_t)), 0};
    }
    // behind the arrays: room for the (cos, sin) table of rotation and projection, filled on the device when first used
    size_t total = bytes;
    for (size_t i = 0; i < count; ++i) {
        at[i].table = (total + 255) / 256 * 256;
        total = at[i].table + (plans[i]->is_part ? 0 : std::max<size_t>((size_t)plans[i]->total_rows * (plans[i]->head_dim / 2) * sizeof(float2), 16));
    }
    int device = -1;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return cuda_fail(e);
    e = plan_res_acquire(device, total, res);
    if (e != cudaSuccess) return cuda_fail(e);
    e = plan_res_upload(*res, parts.data(), parts.size(), bytes);
    if (e != cudaSuccess) return cuda_fail(e);
    char* base = static_cast<char*>(res->blob);
    for (size_t i = 0; i < count; ++i) {
        hat_plan* p = plans[i];
        const Offsets& o = at[i];
        p->device = device;
        p->rope_table = p->is_part ? nullptr : reinterpret_cast<float2*>(base + o.table);
        DevicePlan& d = p->dev;
        d.cu_chunk = reinterpret_cast<const int32_t*>(base + o.cu);
        d.prefix_len = reinterpret_cast<const int32_t*>(base + o.pl);
        d.chunk_len = reinterpret_cast<const int32_t*>(base + o.cl);
        d.block_table = reinterpret_cast<const int32_t*>(base + o.bt);
        d.row_req = reinterpret_cast<const int32_t*>(base + o.rr);
        d.verify_items = reinterpret_cast<const WorkItem*>(base + o.vi);
        d.stream_items = reinterpret_cast<const StreamItem*>(base + o.si);
        d.short_items = reinterpret_cast<const StreamItem*>(base + o.sh);
        d.prefill_items = reinterpret_cast<const WorkItem*>(base + o.pi);
        d.merge_rows = reinterpret_cast<const MergeRow*>(base + o.mr);
        d.tile_units = reinterpret_cast<const uint32_t*>(base + o.tu);
        d.status = reinterpret_cast<int32_t*>(base + o.st);
        d.piece_counters = d.status + 8;
        d.max_pages = p->max_pages;
        d.tree_mask = p->tree_mask.empty() ? nullptr : reinterpret_cast<const uint32_t*>(base + o.tm);
        d.num_heads = p->num_heads;
        d.num_kv_heads = p->num_kv_heads;
        d.group = p->num_heads / p->num_kv_heads;
        d.total_rows = p->total_rows;
        d.tile_rows = p->info.prefill_tile_rows;
        d.num_pages = p->num_pages;
    }
    return HAT_OK;
}

static int check_call(const hat_cache_desc* cache, const hat_plan* plan) {
    if (!cache || !plan) return HAT_ERR_INVALID_ARG;
    if (plan->host_only) return HAT_ERR_INVALID_ARG;
    int st = check_cache_geometry(cache);
    if (st != HAT_OK) return st;
    if (cache->dtype != plan->dtype || cache->num_pages != plan->num_pages ||
        cache->num_kv_heads != plan->num_kv_heads || cache->head_dim != plan->head_dim)
        return HAT_ERR_INVALID_ARG;
    if (!cache->k_pool || !cache->v_pool) return HAT_ERR_INVALID_ARG;
    if (!aligned(cache->k_pool, 16) || !aligned(cache->v_pool, 16)) return HAT_ERR_INVALID_ARG;
    return HAT_OK;
}

static CacheView view_of(const hat_cache_desc* c) {
    return CacheView{c->k_pool, c->v_pool, c->stride_page, c->stride_token, c->stride_head};
}

int create_plan(const hat_cache_desc* cache, const hat_batch_desc* batch, bool part, bool whole, hat_plan** out) {
    if (!out) return HAT_ERR_INVALID_ARG;
    *out = nullptr;
    if (!cache || !batch) return HAT_ERR_INVALID_ARG;
    int st = check_cache_geometry(cache);
    if (st != HAT_OK) return st;
    const int R = batch->num_requests;
    if (R < 0 || batch->max_pages < 0 || batch->num_q_heads <= 0) return HAT_ERR_INVALID_ARG;
    if (batch->num_q_heads % cache->num_kv_heads != 0) return HAT_ERR_UNSUPPORTED;
    if (!batch->cu_chunk) return HAT_ERR_INVALID_ARG;
    if (R > 0 && (!batch->prefix_len || !batch->chunk_len)) return HAT_ERR_INVALID_ARG;
    if (batch->cu_chunk[0] != 0) return HAT_ERR_INVALID_ARG;

    // shapes
    int64_t total = 0;
    for (int r = 0; r < R; ++r) {
        if (batch->prefix_len[r] < 0 || batch->chunk_len[r] < 0) return HAT_ERR_INVALID_ARG;
        total += batch->chunk_len[r];
        if (batch->cu_chunk[r + 1] != total) return HAT_ERR_INVALID_ARG;
        if ((int64_t)batch->prefix_len[r] + batch->chunk_len[r] > (int64_t)INT32_MAX / 2) return HAT_ERR_TOO_LARGE;
    }
    if (total > INT32_MAX / 2) return HAT_ERR_TOO_LARGE;

    // block tables: long enough, inside the pool, and no page written by two requests
    std::vector<uint8_t> written(cache->num_pages > 0 ? cache->num_pages : 0, 0);
    for (int r = 0; r < R; ++r) {
        const int C = batch->chunk_len[r];
        if (C == 0) continue;
        const int N = batch->prefix_len[r] + C;
        const int need = (N + kPageSize - 1) / kPageSize;
        if (need > batch->max_pages) return HAT_ERR_OUT_OF_RANGE;
        if (!batch->block_table) return HAT_ERR_INVALID_ARG;
        const int32_t* row = batch->block_table + (int64_t)r * batch->max_pages;
        for (int j = 0; j < need; ++j)
            if (row[j] < 0 || row[j] >= cache->num_pages) return HAT_ERR_OUT_OF_RANGE;
        for (int j = batch->prefix_len[r] / kPageSize; j < need; ++j) {
            if (written[row[j]]) return HAT_ERR_OUT_OF_RANGE;
            written[row[j]] = 1;
        }
    }

    // a page that one request writes and another one (or the same one, twice in its table) reads as prefix: then the whole
    // append has to come first; otherwise a kernel may take the chunk's rows from k_new / v_new
    bool append_first = false;
    for (int r = 0; r < R && !append_first; ++r) {
        if (batch->chunk_len[r] == 0) continue;
        const int32_t* row = batch->block_table + (int64_t)r * batch->max_pages;
        for (int j = 0; j < batch->prefix_len[r] / kPageSize; ++j)
            if (written[row[j]]) { append_first = true; break; }
    }

    hat_plan* p = new (std::nothrow) hat_plan();
    if (!p) return HAT_ERR_INVALID_ARG;
    struct Owner {
        hat_plan* p;
        ~Owner() { if (p) hat_plan_destroy(p); }
    } owner{p};                                              // until the plan is handed out
    p->dtype = cache->dtype;
    p->num_pages = cache->num_pages;
    p->num_heads = batch->num_q_heads;
    p->num_kv_heads = cache->num_kv_heads;
    p->head_dim = cache->head_dim;
    p->max_pages = batch->max_pages;
    p->num_requests = R;
    p->total_rows = (int32_t)total;
    p->host_only = (batch->flags & HAT_PLAN_HOST_ONLY) != 0;
    p->device = -1;
    p->part_rows = 0;
    p->timing = nullptr;
    p->append_first = append_first;
    p->num_piece_counters = 0;
    p->short_cluster = 0;
    p->num_verify_merge_rows = 0;
    p->tile_clusters = false;
    p->append_apart = false;
    p->parts_made = false;
    p->is_part = part;
    p->captured = p->loose = p->loose_many = false;
    p->loose_stream = nullptr;
    p->rope_table = nullptr;
    p->rope_theta = 0.f;
    p->table_in_graph = false;
    p->table_stream = nullptr;
    p->last_stream = nullptr;
    p->has_last = false;
    p->side_sms = 0;
    p->aux_stream = nullptr;
    p->ev_fork = p->ev_join = nullptr;
    p->wait_cycles = 2000000000LL;
    p->withhold_next = 0;
    std::memset(&p->info, 0, sizeof p->info);
    std::memset(&p->dev, 0, sizeof p->dev);
    p->cu_chunk.assign(batch->cu_chunk, batch->cu_chunk + R + 1);
    p->prefix_len.assign(batch->prefix_len, batch->prefix_len + R);
    p->chunk_len.assign(batch->chunk_len, batch->chunk_len + R);
    if (batch->block_table && batch->max_pages > 0)
        p->block_table.assign(batch->block_table, batch->block_table + (int64_t)R * batch->max_pages);
    if (batch->tree_mask) p->tree_mask.assign(batch->tree_mask, batch->tree_mask + total);
    p->row_req.resize(total);
    for (int r = 0; r < R; ++r)
        for (int t = p->cu_chunk[r]; t < p->cu_chunk[r + 1]; ++t) p->row_req[t] = r;

    p->info.num_requests = R;
    p->info.total_rows = (int32_t)total;
    const int64_t d = p->head_dim, H = p->num_heads;
    for (int r = 0; r < R; ++r) {
        const int64_t C = p->chunk_len[r], P = p->prefix_len[r];
        if (C == 0) continue;
        p->info.attn_flops += 4 * d * H * (C * P + C * (C + 1) / 2);
        p->info.kv_read_bytes += 2 * (P + C) * p->num_kv_heads * d * 2;
    }

    int num_sms = 148;
    if (!p->host_only) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return cuda_fail(e);
    }
    // the tcgen05 tile kernels need a pool layout a TMA descriptor can express (the CTA-pair one also head_dim 128)
    bool use_tc5 = true;
    if (const char* k = std::getenv("HAT_PREFILL_KERNEL"))
        if (std::strcmp(k, "mma") == 0) use_tc5 = false;
    if (use_tc5 && !p->host_only)
        use_tc5 = tc5_layout_supported(p->dtype, p->head_dim, p->num_pages, p->num_kv_heads, cache->stride_page,
                                       cache->stride_token, cache->stride_head);
    p->num_sms = num_sms;
    // Which tcgen05 tile kernel: the CTA-pair kernel (cta_group::2) shares every K/V tile between the two 128-row halves
    // of a 256-row unit and is the faster one for long units; short ones, whose start and rows count for more, and batches that do
    // not fill the pairs are faster on the one-CTA kernel, with units of 128 rows and halves merged by clusters where they are few.
    // HAT_PREFILL_KERNEL = tc5 | pair | mixed (of bf16 batches, wide units to pairs, whatever their length) | mma overrides.
    int tile_kernel = use_tc5 ? 1 : 0;
    int64_t wide_tiles = 0, wide_keys = 0;
    if (use_tc5 && p->head_dim == 128 && p->dtype == HAT_DTYPE_BF16) {
        for (int r = 0; r < R; ++r) {
            const int C = p->chunk_len[r];
            if (C <= 16) continue;
            for (int row0 = 0; row0 < C; row0 += 256)
                if (C - row0 > 128) { ++wide_tiles; wide_keys += p->prefix_len[r] + std::min(C, row0 + 256); }
        }
        // bf16 (its units of more than 128 rows; narrower ones of the same batch run on single CTAs behind them): a step of 128 keys and a
        // unit take a pair 1.45 and 7 us, a CTA 3.3 and 7.5, so pairs pay from some 2200 keys on where they are evenly loaded and surely from 3000, measured (one CTA / pairs, us, 32 heads,
        // means of 3 batches): 4 chunks of 512 at 4000 217 / 211, 8 at 3000 351 / 310, 8 at up to 8000 404 / 392, 12 of 256 to 512 at 2000 to 8000 583 / 536; 40 heads 4 at 4000 331 / 270,
        // 16 at 4000 1116 / 1041; below: 8 at up to 1000 93 / 108, 8 of 200 to 600 at up to 4000 287 / 319,
        // 30 of 256 to 512 at up to 4000 784 / 821; few units: one chunk of 256 at 1000 19.5 / 29.0, 4 of 512 at 4000 x 8 heads 66 / 75.
        // fp16, whose CTAs multiply half as much for the same exponentials, is left to single CTAs: 4 of 512 at 4000 163 / 185, 16 653 / 778, 8 at up to 8000 290 / 329, 12 of 256 to 512
        // 431 / 483, 40 heads 16 at 4000 832 / 968; pairs gain only where the units of single CTAs end unevenly (4 of 512 at 4000 x 40 heads 242 / 237).
        const bool many = wide_tiles * p->num_heads >= 3 * (int64_t)num_sms / 2;
        if (many && wide_keys / wide_tiles >= 3000) tile_kernel = 3;
    }
    p->pair_takes_all = false;
    if (const char* k = std::getenv("HAT_PREFILL_KERNEL")) {
        if (use_tc5 && p->head_dim == 128 && std::strcmp(k, "pair") == 0) { tile_kernel = 3; p->pair_takes_all = true; }
        else if (use_tc5 && std::strcmp(k, "mixed") == 0 && wide_tiles > 0) tile_kernel = 3;
        else if (use_tc5 && std::strcmp(k, "tc5") == 0) tile_kernel = 1;
    }
    // the streaming kernel takes its pages by TMA when a descriptor can be built for the pool layout
    bool stream_tma = true;
    if (const char* k = std::getenv("HAT_STREAM_KERNEL"))
        if (std::strcmp(k, "mma") == 0) stream_tma = false;
    if (stream_tma && !p->host_only)
        stream_tma = stream_layout_supported(p->dtype, p->head_dim, p->num_pages, p->num_kv_heads, cache->stride_page,
                                             cache->stride_token, cache->stride_head);
    p->info.stream_kernel = stream_tma ? 1 : 0;
    schedule(p, num_sms, tile_kernel, whole);
    p->info.num_pair_units = p->num_pair_units;
    // launch-geometry limits: work items index gridDim.y (65535), partial rows and units are 32-bit
    const int64_t verify_count = (int64_t)(p->verify_items.size() + p->stream_items.size());
    if (verify_count > 65535 || verify_count * p->num_kv_heads * p->verify_subtiles > INT32_MAX / 2 || p->prefill_items.size() > 65535 || p->num_heads > 65535 ||
        p->part_rows > INT32_MAX / 2 || (int64_t)p->prefill_items.size() * p->num_heads > INT32_MAX / 2)
        return HAT_ERR_TOO_LARGE;

    if (!p->host_only) {
        if (part) { *out = p; owner.p = nullptr; return HAT_OK; }   // uploaded with the others
        st = upload_plans(&p, 1, &p->res);
        if (st != HAT_OK) return st;
        // Optional throughput mode for a mixed batch on the tcgen05 path (HAT_SIDE_SMS = n > 0): see the launch
        // sequence.  Off by default: it finishes the whole step sooner but the decode-phase rows later.  The side
        // stream has the highest priority so that the tile CTAs are placed before the streaming kernel's many small
        // CTAs fill the SMs.
        if (verify_count > 0 && !p->prefill_items.empty() && p->info.prefill_kernel == 1) {
            int side = env_int("HAT_SIDE_SMS", 0);
            side = std::max(0, std::min(side, p->num_sms - 8));
            if (side > 0) {
                int lo = 0, hi = 0;
                cudaError_t ee = cudaDeviceGetStreamPriorityRange(&lo, &hi);
                if (ee == cudaSuccess) ee = cudaStreamCreateWithPriority(&p->aux_stream, cudaStreamNonBlocking, hi);
                if (ee == cudaSuccess) ee = cudaEventCreateWithFlags(&p->ev_fork, cudaEventDisableTiming);
                if (ee == cudaSuccess) ee = cudaEventCreateWithFlags(&p->ev_join, cudaEventDisableTiming);
                if (ee != cudaSuccess) return cuda_fail(ee);
                p->side_sms = side;
            }
        }
    }
    *out = p;
    owner.p = nullptr;
    return HAT_OK;
}

cudaError_t plan_begin(hat_plan* p, cudaStream_t s) {
    if (p->loose && !p->loose_many && p->loose_stream == s) p->loose = false;      // ev_done, recorded on s by plan_end, covers it
    return p->has_last && p->last_stream != s ? cudaStreamWaitEvent(s, p->res.ev_done, 0) : cudaSuccess;
}

void plan_end(hat_plan* p, cudaStream_t s) {
    if (cudaEventRecord(p->res.ev_done, s) == cudaSuccess) { p->last_stream = s; p->has_last = true; }
    else p->loose = p->loose_many = true;
}

// One attention step; the final rows go to `out` (fp32) or, when out16 is given, to out16 in the cache's 16-bit type.
int run_attention(const hat_cache_desc* cache, const hat_plan* plan, const void* q, const void* k_new,
                         const void* v_new, float* out, void* out16, float* lse, float sm_scale, void* workspace,
                         size_t workspace_bytes, cudaStream_t s, bool check_alignment) {
    int st = check_call(cache, plan);
    if (st != HAT_OK) return st;
    if ((k_new == nullptr) != (v_new == nullptr)) return HAT_ERR_INVALID_ARG;
    if (plan->total_rows == 0) return HAT_OK;
    const void* dst = out16 ? out16 : static_cast<const void*>(out);
    if (!q || !dst || !lse) return HAT_ERR_INVALID_ARG;
    if (check_alignment && (!aligned(q, 16) || !aligned(dst, 16) || !aligned(lse, 16))) return HAT_ERR_INVALID_ARG;
    if (k_new && (!aligned(k_new, 16) || !aligned(v_new, 16))) return HAT_ERR_INVALID_ARG;
    const size_t need = (size_t)plan->info.workspace_bytes;
    if (need > 0) {
        if (!workspace || !aligned(workspace, 256)) return HAT_ERR_INVALID_ARG;
        if (workspace_bytes < need) return HAT_ERR_WORKSPACE_TOO_SMALL;
    }
    if (!(sm_scale > 0.f) || !std::isfinite(sm_scale)) sm_scale = 1.0f / std::sqrt((float)plan->head_dim);

    cudaError_t e;
    // The plan's device state (unit counter, status word) serves one call at a time: a call on another stream than the
    // previous one is ordered behind it.
    // A call that is being captured into a graph cannot wait for (or be waited for through) an event of the world outside
    // the capture: there the caller orders the capturing stream behind the plan's earlier work before the capture begins.
    hat_plan* mplan = const_cast<hat_plan*>(plan);
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if ((e = cudaStreamIsCapturing(s, &cap)) != cudaSuccess) return cuda_fail(e);
    const bool capturing = cap != cudaStreamCaptureStatusNone;
    if (capturing) mplan->captured = true;
    else if ((e = plan_begin(mplan, s)) != cudaSuccess) return cuda_fail(e);
    struct Done {
        hat_plan* p; cudaStream_t s; bool record;
        ~Done() { if (record) plan_end(p, s); }
    } done{mplan, s, !capturing};
    // optional event recorder: a start and an end event per slot (append, tile, streaming, merge)
    Timing* tm = plan->timing;
    int call = -1;
    if (tm && tm->next < tm->max_calls) call = tm->next++;
    auto mark = [&](int slot, int end) {
        if (call >= 0) cudaEventRecord(tm->events[((size_t)call * HAT_TIMING_SLOTS + slot) * 2 + end], s);
        if (call >= 0 && end) tm->launched[(size_t)call * HAT_TIMING_SLOTS + slot] = 1;
    };
    // the attention kernels append on the way, each class its own requests' rows, unless pages are shared between a writer and
    // a reader, a class runs on the mma.sync kernels, or a kernel in front is cheaper
    const bool has_verify = plan->info.num_verify_items > 0;
    const bool fused = k_new && !plan->append_first && !plan->append_apart && (!has_verify || plan->info.stream_kernel != 0) &&
                       (plan->prefill_items.empty() || plan->info.prefill_kernel != 0);
    if (k_new && !fused) {
        mark(0, 0);
        e = launch_kv_append(plan, view_of(cache), cache->k_pool, cache->v_pool, k_new, v_new, s);
        if (e != cudaSuccess) return cuda_fail(e);
        mark(0, 1);
    }
    AttnArgs a;
    a.plan = plan->dev;
    a.cache = view_of(cache);
    a.q = q;
    a.k_new = fused ? k_new : nullptr;
    a.v_new = fused ? v_new : nullptr;
    a.k_dst = cache->k_pool;
    a.v_dst = cache->v_pool;
    a.out = out;
    a.out16 = out16;
    a.out16_bf16 = plan->dtype == HAT_DTYPE_BF16 ? 1 : 0;
    a.lse = lse;
    a.part_out = static_cast<float*>(workspace);
    const int64_t H = plan->num_heads, d = plan->head_dim;
    const size_t part_out_bytes = ((size_t)plan->part_rows * H * d * 4 + 255) / 256 * 256;
    a.part_lse = need ? reinterpret_cast<float*>(static_cast<char*>(workspace) + part_out_bytes) : nullptr;
    a.part_rows = plan->part_rows;
    a.scale_log2 = sm_scale * 1.4426950408889634f;
    a.wait_cycles = plan->wait_cycles;
    a.withhold = plan->withhold_next;
    a.tail_reset = 0;
    a.static_first = 0;
    a.overlap = 0;
    const_cast<hat_plan*>(plan)->withhold_next = 0;

    // Decode-phase (draft verification) requests first: their rows are final, and announced through the plan's event,
    // before the prompt chunks of the same batch are computed, so that they are not held back by them.
    const int n_vm = plan->num_verify_merge_rows, n_m = (int)plan->merge_rows.size();
    // Mixed batch: the tile kernel starts at once on all but side_sms SMs (own stream), the streaming kernel takes the
    // rest, and when it is done a second tile grid joins on the SMs it frees; both grids draw from one unit counter.
    const bool side = plan->side_sms > 0;
    if (side) {
        if ((e = cudaMemsetAsync(plan->dev.status + 1, 0, sizeof(int32_t), s)) != cudaSuccess) return cuda_fail(e);
        if ((e = cudaEventRecord(plan->ev_fork, s)) != cudaSuccess) return cuda_fail(e);
        if ((e = cudaStreamWaitEvent(plan->aux_stream, plan->ev_fork, 0)) != cudaSuccess) return cuda_fail(e);
        mark(1, 0);
        e = launch_attn_tc5(plan, a, plan->aux_stream, plan->num_sms - plan->side_sms, /*reset_counter=*/false);
        if (e == cudaSuccess) e = cudaEventRecord(plan->ev_join, plan->aux_stream);
        if (e != cudaSuccess) return cuda_fail(e);
    }
    if (has_verify) {
        mark(2, 0);
        e = plan->info.stream_kernel != 0 ? launch_attn_stream(plan, a, s)
                                          : launch_attn_mma(plan, a, /*verify_class=*/true, s);
        if (e == cudaSuccess && n_vm > 0) e = launch_merge(plan, a, 0, n_vm, s);
        if (e != cudaSuccess) return cuda_fail(e);
        mark(2, 1);
    }
    // a batch without such rows has nothing to announce (an event that was never recorded counts as occurred); of the parts of a
    // batch the last one that has some announces (the others have no event)
    if (has_verify && plan->res.ev_verify && (e = cudaEventRecord(plan->res.ev_verify, s)) != cudaSuccess) return cuda_fail(e);
    // The tile kernels depend on nothing the streaming kernel does: they take the SMs as it leaves them.  (Not under the timing
    // recorder, which wants the kernels one after the other.)
    a.overlap = has_verify && plan->info.stream_kernel != 0 && !side && call < 0 ? 1 : 0;
    if (side) {
        e = launch_attn_tc5(plan, a, s, plan->side_sms, /*reset_counter=*/false);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(s, plan->ev_join, 0);
        if (e != cudaSuccess) return cuda_fail(e);
        mark(1, 1);
    } else if (!plan->prefill_items.empty()) {
        mark(1, 0);
        if (plan->info.prefill_kernel == 3) {
            // long units of more than 128 rows on CTA pairs, the others (if any) on single CTAs that take the SMs as the pairs leave them
            e = launch_attn_pair(plan, a, s, plan->num_pair_units);
            if (e == cudaSuccess) e = launch_attn_tc5(plan, a, s, 0, true, plan->num_pair_units, -1, /*counter_word=*/3, /*overlap=*/true);
        } else {
            e = plan->info.prefill_kernel == 1 ? launch_attn_tc5(plan, a, s)
                                               : launch_attn_mma(plan, a, /*verify_class=*/false, s);
        }
        if (e != cudaSuccess) return cuda_fail(e);
        mark(1, 1);
    }
    if (n_m > n_vm) {
        mark(3, 0);
        e = launch_merge(plan, a, n_vm, n_m - n_vm, s);
        if (e != cudaSuccess) return cuda_fail(e);
        mark(3, 1);
    }
    return HAT_OK;
}

}  // namespace hat

using namespace hat;

extern "C" {

const char* hat_status_string(int status) {
    switch (status) {
        case HAT_OK: return "ok";
        case HAT_ERR_INVALID_ARG: return "invalid argument";
        case HAT_ERR_UNSUPPORTED: return "unsupported configuration";
        case HAT_ERR_OUT_OF_RANGE: return "index out of range";
        case HAT_ERR_WORKSPACE_TOO_SMALL: return "workspace too small";
        case HAT_ERR_CUDA: return "CUDA error";
        case HAT_ERR_DEVICE_TIMEOUT: return "device-side wait timed out";
        case HAT_ERR_TOO_LARGE: return "size exceeds a fixed maximum";
        case HAT_ERR_DEVICE_BOUNDS: return "device-side index check failed (debug build)";
        default: return "unknown status";
    }
}

int hat_version(void) { return HAT_VERSION; }
int hat_last_cuda_error(void) { return g_last_cuda_error; }
int64_t hat_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

int64_t hat_device_alloc_count(void) { return plan_res_allocs(); }

int hat_plan_create(const hat_cache_desc* cache, const hat_batch_desc* batch, hat_plan** out) {
    return guarded([&] { return create_plan(cache, batch, /*part=*/false, /*whole=*/false, out); });
}

int hat_plan_get_info(const hat_plan* plan, hat_plan_info* out) {
    if (!plan || !out) return HAT_ERR_INVALID_ARG;
    *out = plan->info;
    return HAT_OK;
}

int hat_plan_workspace_bytes(const hat_plan* plan, size_t* out) {
    if (!plan || !out) return HAT_ERR_INVALID_ARG;
    *out = (size_t)plan->info.workspace_bytes;
    return HAT_OK;
}

int hat_plan_destroy(hat_plan* plan) {
    if (!plan) return HAT_OK;
    int st = HAT_OK;
    if (plan->timing) {
        for (cudaEvent_t ev : plan->timing->events) cudaEventDestroy(ev);
        delete plan->timing;
    }
    if (!plan->parts.empty()) {
        bool covered = true;                                 // by the parts' common ev_done
        for (hat_plan* part : plan->parts) {
            plan->part_res.in_use |= part->has_last;
            covered &= !part->captured && !part->loose;
            delete part;
        }
        const cudaError_t e = plan_res_release(plan->part_res, covered);
        if (e != cudaSuccess) st = cuda_fail(e);
    }
    if (plan->ev_fork) cudaEventDestroy(plan->ev_fork);
    if (plan->ev_join) cudaEventDestroy(plan->ev_join);
    if (plan->aux_stream) cudaStreamDestroy(plan->aux_stream);
    if (!plan->host_only) {
        // handed on to a later plan unless a graph may replay a call, or work that ev_done does not cover may still run
        plan->res.in_use = plan->has_last;
        const cudaError_t e = plan_res_release(plan->res, !plan->captured && !plan->loose);
        if (e != cudaSuccess) st = cuda_fail(e);
    }
    delete plan;
    return st;
}

int hat_release_cached(void) {
    return guarded([] {
        const cudaError_t e = plan_res_trim();
        return e == cudaSuccess ? HAT_OK : cuda_fail(e);
    });
}

int hat_kv_append(const hat_cache_desc* cache, const hat_plan* plan, const void* k_new, const void* v_new,
                  void* stream) {
    int st = check_call(cache, plan);
    if (st != HAT_OK) return st;
    if (plan->total_rows == 0) return HAT_OK;
    if (!k_new || !v_new || !aligned(k_new, 16) || !aligned(v_new, 16)) return HAT_ERR_INVALID_ARG;
    plan_note_call(const_cast<hat_plan*>(plan), static_cast<cudaStream_t>(stream));
    cudaError_t e = launch_kv_append(plan, view_of(cache), cache->k_pool, cache->v_pool, k_new, v_new,
                                     static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? HAT_OK : cuda_fail(e);
}

int hat_kv_append_rope(const hat_cache_desc* cache, const hat_plan* plan, const void* k_new, const void* v_new,
                       float theta, int interleaved, void* stream) {
    int st = check_call(cache, plan);
    if (st != HAT_OK) return st;
    if (!(theta > 1.f) || !std::isfinite(theta)) return HAT_ERR_INVALID_ARG;
    if (plan->total_rows == 0) return HAT_OK;
    if (!k_new || !v_new || !aligned(k_new, 16) || !aligned(v_new, 16)) return HAT_ERR_INVALID_ARG;
    const CacheView view = view_of(cache);
    plan_note_call(const_cast<hat_plan*>(plan), static_cast<cudaStream_t>(stream));
    cudaError_t e = launch_rope(plan, plan->num_kv_heads, theta, interleaved != 0, k_new, nullptr, &view, cache->k_pool,
                                cache->v_pool, v_new, static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? HAT_OK : cuda_fail(e);
}

int hat_rope_q(const hat_plan* plan, const void* q, void* q_out, float theta, int interleaved, void* stream) {
    if (!plan || plan->host_only) return HAT_ERR_INVALID_ARG;
    if (!(theta > 1.f) || !std::isfinite(theta)) return HAT_ERR_INVALID_ARG;
    if (plan->total_rows == 0) return HAT_OK;
    if (!q || !q_out || !aligned(q, 16) || !aligned(q_out, 16)) return HAT_ERR_INVALID_ARG;
    plan_note_call(const_cast<hat_plan*>(plan), static_cast<cudaStream_t>(stream));
    cudaError_t e = launch_rope(plan, plan->num_heads, theta, interleaved != 0, q, q_out, nullptr, nullptr, nullptr, nullptr,
                                static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? HAT_OK : cuda_fail(e);
}

int hat_qkv_rope_append(const hat_cache_desc* cache, const hat_plan* plan, const void* x, int hidden, const void* w_qkv,
                        void* q_out, float theta, int interleaved, void* stream) {
    int st = check_call(cache, plan);
    if (st != HAT_OK) return st;
    if (theta > 0.f && (!(theta > 1.f) || !std::isfinite(theta))) return HAT_ERR_INVALID_ARG;
    if (hidden <= 0) return HAT_ERR_INVALID_ARG;
    if (hidden % 64 != 0 || (plan->head_dim != 64 && plan->head_dim != 128)) return HAT_ERR_UNSUPPORTED;
    if (plan->total_rows == 0) return HAT_OK;
    if (!x || !w_qkv || !q_out || !aligned(x, 16) || !aligned(w_qkv, 16) || !aligned(q_out, 16)) return HAT_ERR_INVALID_ARG;
    plan_note_call(const_cast<hat_plan*>(plan), static_cast<cudaStream_t>(stream));
    return guarded([&] {
        const cudaError_t e = launch_qkv_gemm(plan, view_of(cache), cache->k_pool, cache->v_pool, x, hidden, w_qkv, q_out, theta,
                                              interleaved != 0, static_cast<cudaStream_t>(stream));
        return e == cudaSuccess ? HAT_OK : cuda_fail(e);
    });
}

int hat_chunk_attention(const hat_cache_desc* cache, const hat_plan* plan, const void* q, const void* k_new,
                        const void* v_new, float* out, float* lse, float sm_scale, void* workspace,
                        size_t workspace_bytes, void* stream) {
    if (!out && plan && plan->total_rows > 0) return HAT_ERR_INVALID_ARG;
    return guarded([&] { return run_attention(cache, plan, q, k_new, v_new, out, nullptr, lse, sm_scale, workspace, workspace_bytes, static_cast<cudaStream_t>(stream)); });
}

int hat_chunk_attention_out16(const hat_cache_desc* cache, const hat_plan* plan, const void* q, const void* k_new,
                              const void* v_new, void* out16, float* lse, float sm_scale, void* workspace,
                              size_t workspace_bytes, void* stream) {
    if (!out16 && plan && plan->total_rows > 0) return HAT_ERR_INVALID_ARG;
    return guarded([&] { return run_attention(cache, plan, q, k_new, v_new, nullptr, out16, lse, sm_scale, workspace, workspace_bytes, static_cast<cudaStream_t>(stream)); });
}

int hat_plan_verify_event(const hat_plan* plan, void** event_out) {
    if (!plan || !event_out || plan->host_only) return HAT_ERR_INVALID_ARG;
    *event_out = plan->res.ev_verify;
    return HAT_OK;
}

int hat_plan_wait_verify(const hat_plan* plan) {
    if (!plan || plan->host_only || !plan->res.ev_verify) return HAT_ERR_INVALID_ARG;
    cudaError_t e = cudaEventSynchronize(plan->res.ev_verify);
    return e == cudaSuccess ? HAT_OK : cuda_fail(e);
}

int hat_plan_enable_timing(hat_plan* plan, int max_calls) {
    if (!plan || plan->host_only || max_calls <= 0 || max_calls > (1 << 20)) return HAT_ERR_INVALID_ARG;
    if (plan->timing) {
        for (cudaEvent_t ev : plan->timing->events) cudaEventDestroy(ev);
        delete plan->timing;
        plan->timing = nullptr;
    }
    Timing* tm = new (std::nothrow) Timing();
    if (!tm) return HAT_ERR_INVALID_ARG;
    if (guarded([&] {
            tm->events.resize((size_t)max_calls * HAT_TIMING_SLOTS * 2);
            tm->launched.assign((size_t)max_calls * HAT_TIMING_SLOTS, 0);
            return HAT_OK;
        }) != HAT_OK) {
        delete tm;
        return HAT_ERR_INVALID_ARG;
    }
    for (size_t i = 0; i < tm->events.size(); ++i) {
        cudaError_t e = cudaEventCreate(&tm->events[i]);
        if (e != cudaSuccess) {
            for (size_t j = 0; j < i; ++j) cudaEventDestroy(tm->events[j]);
            delete tm;
            return cuda_fail(e);
        }
    }
    tm->max_calls = max_calls;
    plan->timing = tm;
    return HAT_OK;
}

int hat_plan_read_timing(hat_plan* plan, float* ms, int capacity_calls, int* num_calls) {
    if (!plan || !ms || !num_calls || capacity_calls < 0 || !plan->timing) return HAT_ERR_INVALID_ARG;
    Timing* tm = plan->timing;
    const int n = std::min(tm->next, capacity_calls);
    for (int c = 0; c < n; ++c) {
        for (int sl = 0; sl < HAT_TIMING_SLOTS; ++sl) {
            float t = 0.f;
            if (tm->launched[(size_t)c * HAT_TIMING_SLOTS + sl]) {
                cudaEvent_t e0 = tm->events[((size_t)c * HAT_TIMING_SLOTS + sl) * 2];
                cudaEvent_t e1 = tm->events[((size_t)c * HAT_TIMING_SLOTS + sl) * 2 + 1];
                cudaError_t e = cudaEventSynchronize(e1);
                if (e == cudaSuccess) e = cudaEventElapsedTime(&t, e0, e1);
                if (e != cudaSuccess) return cuda_fail(e);
            }
            ms[(size_t)c * HAT_TIMING_SLOTS + sl] = t;
        }
    }
    *num_calls = n;
    tm->next = 0;
    std::fill(tm->launched.begin(), tm->launched.end(), 0);
    return HAT_OK;
}

int hat_plan_staging_bytes(const hat_plan* plan, size_t* out) {
    if (!plan || !out) return HAT_ERR_INVALID_ARG;
    const size_t T = plan->total_rows, H = plan->num_heads, Hkv = plan->num_kv_heads, d = plan->head_dim;
    const size_t q16 = (T * H * d * 2 + 255) / 256 * 256;
    const size_t kv16 = (T * Hkv * d * 2 + 255) / 256 * 256;
    const size_t out32 = (T * H * d * 4 + 255) / 256 * 256;
    const size_t lse32 = (T * H * 4 + 255) / 256 * 256;
    *out = q16 + 2 * kv16 + out32 + lse32;
    return HAT_OK;
}

int hat_chunk_attention_host(const hat_cache_desc* cache, const hat_plan* plan, const void* q_host,
                             const void* k_new_host, const void* v_new_host, float* out_host, float* lse_host,
                             float sm_scale, void* staging, size_t staging_bytes, void* workspace,
                             size_t workspace_bytes, void* stream) {
    int st = check_call(cache, plan);
    if (st != HAT_OK) return st;
    if (plan->total_rows == 0) return HAT_OK;
    if (!q_host || !k_new_host || !v_new_host || !out_host || !lse_host) return HAT_ERR_INVALID_ARG;
    size_t need = 0;
    hat_plan_staging_bytes(plan, &need);
    if (!staging || !aligned(staging, 256)) return HAT_ERR_INVALID_ARG;
    if (staging_bytes < need) return HAT_ERR_WORKSPACE_TOO_SMALL;
    if (plan->info.workspace_bytes > 0) {
        if (!workspace || !aligned(workspace, 256)) return HAT_ERR_INVALID_ARG;
        if (workspace_bytes < (size_t)plan->info.workspace_bytes) return HAT_ERR_WORKSPACE_TOO_SMALL;
    }
    const size_t T = plan->total_rows, H = plan->num_heads, Hkv = plan->num_kv_heads, d = plan->head_dim;
    const size_t act_bytes = T * H * d * 2, kv_bytes = T * Hkv * d * 2, out_bytes = T * H * d * 4;
    const size_t q16 = (act_bytes + 255) / 256 * 256, kv16 = (kv_bytes + 255) / 256 * 256, out32 = (out_bytes + 255) / 256 * 256;
    char* base = static_cast<char*>(staging);
    void* dq = base;
    void* dk = base + q16;
    void* dv = base + q16 + kv16;
    float* dout = reinterpret_cast<float*>(base + q16 + 2 * kv16);
    float* dlse = reinterpret_cast<float*>(base + q16 + 2 * kv16 + out32);
    cudaError_t e = cudaSuccess;
    st = guarded([&] {
        return host_step(cache, plan, HostBuffers{q_host, k_new_host, v_new_host, out_host, lse_host}, HostBuffers{dq, dk, dv, dout, dlse}, sm_scale,
                         workspace, workspace_bytes, static_cast<cudaStream_t>(stream), &e);
    });
    return st == HAT_ERR_CUDA && e != cudaSuccess ? cuda_fail(e) : st;
}

int hat_last_device_status(const hat_plan* plan, void* stream, int* out) {
    if (!plan || !out || plan->host_only) return HAT_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int32_t word = 0;
    // behind the plan's latest call, whose counters are among the words that are cleared
    cudaError_t e = plan->has_last && plan->last_stream != s ? cudaStreamWaitEvent(s, plan->res.ev_done, 0) : cudaSuccess;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&word, plan->dev.status, sizeof word, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(plan->dev.status, 0, plan->num_status_words * sizeof word, s);     // status, counters
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(e);
    for (const hat_plan* part : plan->parts) {
        int st = HAT_OK;
        const int rc = hat_last_device_status(part, stream, &st);
        if (rc != HAT_OK) return rc;
        if (st != HAT_OK) word |= st == HAT_ERR_DEVICE_TIMEOUT ? 1 : 2;
    }
    *out = word == 0 ? HAT_OK : (word & 1) ? HAT_ERR_DEVICE_TIMEOUT : HAT_ERR_DEVICE_BOUNDS;
    return HAT_OK;
}

int hat_plan_set_wait_limit(hat_plan* plan, long long cycles, int withhold_next_call) {
    if (!plan || cycles < 0) return HAT_ERR_INVALID_ARG;
    plan->wait_cycles = cycles > 0 ? cycles : 2000000000LL;
    plan->withhold_next = withhold_next_call ? 1 : 0;
    return HAT_OK;
}

}  // extern "C"
