// The step for callers whose activations live in host memory: copies in, append and attention, copies back.
//
// Bound: the PCIe link (53 GB/s each way).  Copying everything in, computing and copying everything back leaves the link
// idle in one direction all the time and in both while the kernels run (636 rows x 32 heads: 294 + 95 + 190 us).  So a batch
// with enough rows is split into parts, contiguous requests with plans of their own: part by part the rows come in on a
// stream of the plan's, are computed on the caller's stream and go back on a third one.  The caller's stream waits for the
// last copy back.  636 rows: 603 us in one part, 508 us in
// five (the link moves 44 to 77 GB/s in both directions together at such sizes).
#include <algorithm>

#include "hat_internal.h"

namespace hat {
namespace {

// A part carries at least about this many bytes in (45 us of the link: its copies' gaps and its kernels' launches cost 10; 15.7
// MB in parts of 8 / 5 / 3.5 / 2.5 / 1.8 / 0.8 MB: 556 / 542 / 531 / 530 / 559 / 575 us), and there are at most kMaxParts.
constexpr size_t kPartBytes = size_t(5) << 19;
constexpr int kMaxParts = 8;

// Splits the batch into contiguous requests; false: one part would do.
bool split_requests(const hat_plan* p, std::vector<int>& first) {
    const size_t row_bytes = ((size_t)p->num_heads + 2 * (size_t)p->num_kv_heads) * p->head_dim * 2;
    const size_t total = row_bytes * p->total_rows;
    const size_t target = std::max(kPartBytes, (total + kMaxParts - 1) / kMaxParts);
    first.assign(1, 0);
    size_t have = 0, left = total;
    for (int r = 0; r < p->num_requests; ++r) {
        const size_t n = row_bytes * p->chunk_len[r];
        // a new part where the current one is full enough and what follows still makes one
        if (have > 0 && have + n / 2 >= target && left >= target / 2) { first.push_back(r); have = 0; }
        have += n;
        left -= n;
    }
    return first.size() > 1;
}

// Makes and uploads the plans; false: they are not all there.
bool plan_parts(hat_plan* p, const hat_cache_desc* cache, std::vector<int>& first) {
    first.push_back(p->num_requests);
    std::vector<int32_t> cu;
    p->parts.reserve(first.size());
    p->part_row.reserve(first.size());
    for (size_t i = 0; i + 1 < first.size(); ++i) {
        const int r0 = first[i], n = first[i + 1] - r0;
        cu.resize(n + 1);
        for (int r = 0; r <= n; ++r) cu[r] = p->cu_chunk[r0 + r] - p->cu_chunk[r0];
        hat_batch_desc b = {};
        b.num_requests = n;
        b.num_q_heads = p->num_heads;
        b.max_pages = p->max_pages;
        b.cu_chunk = cu.data();
        b.prefix_len = p->prefix_len.data() + r0;
        b.chunk_len = p->chunk_len.data() + r0;
        b.block_table = p->block_table.empty() ? nullptr : p->block_table.data() + (size_t)r0 * p->max_pages;
        b.tree_mask = p->tree_mask.empty() ? nullptr : p->tree_mask.data() + p->cu_chunk[r0];
        hat_plan* part = nullptr;
        // a part alone may want more key ranges than the whole batch: not more workspace than the caller has
        int st = create_plan(cache, &b, /*part=*/true, /*whole=*/false, &part);
        if (st == HAT_OK && part->info.workspace_bytes > p->info.workspace_bytes) {
            delete part;
            st = create_plan(cache, &b, /*part=*/true, /*whole=*/true, &part);
        }
        if (st != HAT_OK) return false;
        p->parts.push_back(part);
        p->part_row.push_back(p->cu_chunk[r0]);
    }
    return upload_plans(p->parts.data(), p->parts.size(), &p->part_res) == HAT_OK;
}

void make_parts(hat_plan* p, const hat_cache_desc* cache) {
    std::vector<int> first;
    p->parts_made = true;
    bool several = false, ok = false;
    guarded([&] { several = split_requests(p, first); return HAT_OK; });
    if (!several) return;
    guarded([&] { ok = plan_parts(p, cache, first); return HAT_OK; });
    hat_plan* last = nullptr;                                // of the parts with drafts: announces those of the whole batch
    for (hat_plan* part : p->parts) {
        part->res.ev_done = p->part_res.ev_done;
        if (part->info.num_verify_items > 0) last = part;
        if (!ok) delete part;
    }
    if (ok && last) last->res.ev_verify = p->res.ev_verify;
    if (!ok) {
        p->parts.clear();
        p->part_row.clear();
        plan_res_free(p->part_res);
    }
}

}  // namespace

int host_step(const hat_cache_desc* cache, const hat_plan* plan, const HostBuffers& h, const HostBuffers& dev, float sm_scale, void* workspace,
              size_t workspace_bytes, cudaStream_t s, cudaError_t* err) {
    hat_plan* p = const_cast<hat_plan*>(plan);
    cudaError_t& e = *err;
    const size_t H = p->num_heads, Hkv = p->num_kv_heads, d = p->head_dim;
    const size_t q_row = H * d * 2, kv_row = Hkv * d * 2, out_row = H * d * 4, lse_row = H * 4;
    auto at = [](const void* base, size_t bytes) { return static_cast<char*>(const_cast<void*>(base)) + bytes; };
    auto copy_in = [&](size_t row, size_t rows, cudaStream_t st) {
        e = cudaMemcpyAsync(at(dev.k, row * kv_row), at(h.k, row * kv_row), rows * kv_row, cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(at(dev.v, row * kv_row), at(h.v, row * kv_row), rows * kv_row, cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(at(dev.q, row * q_row), at(h.q, row * q_row), rows * q_row, cudaMemcpyHostToDevice, st);
        return e == cudaSuccess;
    };
    auto copy_out = [&](size_t row, size_t rows, cudaStream_t st) {
        e = cudaMemcpyAsync(at(h.out, row * out_row), at(dev.out, row * out_row), rows * out_row, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(at(h.lse, row * lse_row), at(dev.lse, row * lse_row), rows * lse_row, cudaMemcpyDeviceToHost, st);
        return e == cudaSuccess;
    };
    auto attend = [&](const hat_plan* pl, size_t row) {
        return run_attention(cache, pl, at(dev.q, row * q_row), at(dev.k, row * kv_row), at(dev.v, row * kv_row),
                             reinterpret_cast<float*>(at(dev.out, row * out_row)), nullptr, reinterpret_cast<float*>(at(dev.lse, row * lse_row)),
                             sm_scale, workspace, workspace_bytes, s, /*check_alignment=*/false);
    };

    // One part: also where the parts' order or the plan's own state matters (pages shared between requests, the timing
    // recorder, the self test of the waits) and inside a stream capture.
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if ((e = cudaStreamIsCapturing(s, &cap)) != cudaSuccess) return HAT_ERR_CUDA;
    const bool plain = cap != cudaStreamCaptureStatusNone || p->append_first || p->timing || p->withhold_next;
    if (!plain && !p->parts_made) make_parts(p, cache);      // where it fails the batch goes as one part
    if (plain || p->parts.empty()) {
        if (!copy_in(0, p->total_rows, s)) return HAT_ERR_CUDA;
        const int st = attend(plan, 0);
        if (st != HAT_OK) return st;
        return copy_out(0, p->total_rows, s) ? HAT_OK : HAT_ERR_CUDA;
    }

    if ((e = plan_res_copy_streams(p->res)) != cudaSuccess) return HAT_ERR_CUDA;
    const cudaStream_t in = p->res.copy_in, out = p->res.copy_out;
    const cudaEvent_t ev = p->res.ev_copy;      // recorded and waited for at once, so that one serves every edge
    auto edge = [&](cudaStream_t from, cudaStream_t to) {
        e = cudaEventRecord(ev, from);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(to, ev, 0);
        return e == cudaSuccess;
    };
    if (!edge(s, in) || !edge(s, out)) return HAT_ERR_CUDA;
    // The parts' kernels run behind the plan's previous call and its next one behind them, like those of a call in one part;
    // the copies in (to the caller's staging memory) need not wait for that.
    if ((e = plan_begin(p, s)) != cudaSuccess) return HAT_ERR_CUDA;
    struct Done {
        hat_plan* p; cudaStream_t s;
        void now() { if (p) plan_end(p, s); p = nullptr; }
        ~Done() { now(); }
    } done{p, s};
    const size_t n = p->parts.size();
    for (size_t i = 0; i < n; ++i) {
        hat_plan* part = p->parts[i];
        part->wait_cycles = p->wait_cycles;
        if (part->total_rows > 0) {
            if (!copy_in(p->part_row[i], part->total_rows, in) || !edge(in, s)) return HAT_ERR_CUDA;
            const int st = attend(part, p->part_row[i]);
            if (st != HAT_OK) return st;
        }
        // one part behind: a copy back to pageable memory blocks the host, which should have enqueued the next part by then
        if (i > 0 && !copy_out(p->part_row[i - 1], p->parts[i - 1]->total_rows, out)) return HAT_ERR_CUDA;
        if (!edge(s, out)) return HAT_ERR_CUDA;
    }
    done.now();                                              // before the last copies back: they are no one's business but the caller's
    if (!copy_out(p->part_row[n - 1], p->parts[n - 1]->total_rows, out) || !edge(out, s)) return HAT_ERR_CUDA;
    return HAT_OK;
}

}  // namespace hat
