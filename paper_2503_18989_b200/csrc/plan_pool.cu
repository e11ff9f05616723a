// What destroyed plans hand on to later ones: device memory and events; and the pinned buffer plans are uploaded from.
//
// A serving loop makes one plan per inference step.  With a few GB of pools on the device a cudaMalloc / cudaFree pair
// costs 360 + 270 us of host time (measured beside 6 GB, 12 requests), both synchronise the device, and a pageable
// cudaMemcpy on the legacy stream waits for the previous step's kernels: together more than the eight layers of the
// step take on the GPU.  The pool turns that into a search of a short list and one small asynchronous copy.
//
// Bounds: at most kMaxIdle entries and kMaxIdleBytes of device memory wait in the list, per process; the oldest that are no
// longer in use make room for what is given back, and hat_release_cached() frees the rest.  Entries are handed on whole under one
// lock; an entry whose last owner's kernels may still run is taken (or freed for room) only after that owner's ev_done has occurred.
#include <algorithm>
#include <atomic>
#include <cstring>
#include <mutex>
#include <vector>

#include "hat_internal.h"

namespace hat {
namespace {

constexpr size_t kMaxIdle = 64;
constexpr size_t kMaxIdleBytes = size_t(64) << 20;
std::atomic<int64_t> g_allocs{0};

// what a plan that needs n bytes is given where nothing waits for it: a power of two, 64 KiB at least
size_t block_size(size_t n) {
    size_t b = size_t(64) << 10;
    while (b < n) b *= 2;
    return b;
}

struct Pool {
    std::mutex mu;
    std::vector<PlanRes> idle;        // room for kMaxIdle from the start: giving back allocates nothing
    // uploads: one at a time, complete before the next, so that one pinned buffer serves all plans
    std::mutex up_mu;
    std::vector<std::pair<int, cudaStream_t>> up_streams;   // per device
    void* up_buf = nullptr;
    size_t up_bytes = 0;
};
Pool& pool() {
    static Pool* p = [] { Pool* q = new Pool(); q->idle.reserve(kMaxIdle); return q; }();   // never destroyed: plans may outlive static destructors
    return *p;
}

size_t idle_bytes(const std::vector<PlanRes>& v) {
    size_t n = 0;
    for (const PlanRes& r : v) n += r.blob_bytes;
    return n;
}

}  // namespace

cudaError_t plan_res_free(PlanRes& r) {
    cudaError_t e = cudaSuccess;
    if (r.ev_verify) cudaEventDestroy(r.ev_verify);
    if (r.ev_done) cudaEventDestroy(r.ev_done);
    if (r.ev_table) cudaEventDestroy(r.ev_table);
    if (r.ev_copy) cudaEventDestroy(r.ev_copy);
    if (r.copy_in) cudaStreamDestroy(r.copy_in);
    if (r.copy_out) cudaStreamDestroy(r.copy_out);
    if (r.blob) e = cudaFree(r.blob);              // waits for the device, so kernels that still use the plan finish first
    r = PlanRes{};
    return e;
}

cudaError_t plan_res_acquire(int device, size_t blob_bytes, PlanRes* out) {
    Pool& p = pool();
    {
        std::unique_lock<std::mutex> lock(p.mu);
        int ready = -1, oldest = -1;
        for (int i = 0; i < (int)p.idle.size(); ++i) {          // in the order they were given back
            PlanRes& r = p.idle[i];
            // not for a plan that would need much less: the large ones would all end up with small plans
            if (r.device != device || r.blob_bytes < blob_bytes || r.blob_bytes / 8 > block_size(blob_bytes)) continue;
            if (oldest < 0) oldest = i;
            if (!r.in_use || cudaEventQuery(r.ev_done) == cudaSuccess) { ready = i; break; }
        }
        // kMaxIdle steps in flight: wait for the oldest instead of growing further
        const bool wait = ready < 0 && oldest >= 0 && p.idle.size() >= kMaxIdle;
        if (ready < 0 && wait) ready = oldest;
        if (ready >= 0) {
            *out = p.idle[ready];
            p.idle.erase(p.idle.begin() + ready);
            lock.unlock();
            cudaGetLastError();                                  // cudaErrorNotReady of a query is no error
            if (wait) {
                const cudaError_t e = cudaEventSynchronize(out->ev_done);
                if (e != cudaSuccess) { plan_res_free(*out); return e; }
            }
            out->in_use = false;
            return cudaSuccess;
        }
        cudaGetLastError();
    }
    PlanRes r;
    r.device = device;
    r.blob_bytes = block_size(blob_bytes);
    g_allocs.fetch_add(1, std::memory_order_relaxed);
    cudaError_t e = cudaMalloc(&r.blob, r.blob_bytes);
    if (e == cudaErrorMemoryAllocation) {                        // give back what waits in the list and try once more
        cudaGetLastError();
        plan_res_trim();
        e = cudaMalloc(&r.blob, r.blob_bytes);
    }
    if (e != cudaSuccess) r.blob = nullptr;
    for (cudaEvent_t* ev : {&r.ev_verify, &r.ev_done, &r.ev_table})
        if (e == cudaSuccess && (e = cudaEventCreateWithFlags(ev, cudaEventDisableTiming)) != cudaSuccess) *ev = nullptr;
    if (e != cudaSuccess) { plan_res_free(r); return e; }
    *out = r;
    return cudaSuccess;
}

cudaError_t plan_res_copy_streams(PlanRes& r) {
    cudaError_t e = cudaSuccess;
    for (cudaStream_t* s : {&r.copy_in, &r.copy_out})
        if (!*s && e == cudaSuccess && (e = cudaStreamCreateWithFlags(s, cudaStreamNonBlocking)) != cudaSuccess) *s = nullptr;
    if (!r.ev_copy && e == cudaSuccess && (e = cudaEventCreateWithFlags(&r.ev_copy, cudaEventDisableTiming)) != cudaSuccess) r.ev_copy = nullptr;
    return e;
}

cudaError_t plan_res_release(PlanRes& r, bool reusable) {
    if (!r.blob || !reusable || r.blob_bytes > kMaxIdleBytes) return plan_res_free(r);
    Pool& p = pool();
    PlanRes gone[kMaxIdle];
    size_t num_gone = 0;
    {
        std::lock_guard<std::mutex> lock(p.mu);
        size_t bytes = idle_bytes(p.idle);
        bool queried = false;
        for (size_t i = 0; i < p.idle.size() && (p.idle.size() >= kMaxIdle || bytes + r.blob_bytes > kMaxIdleBytes);) {
            PlanRes& old = p.idle[i];
            if (old.in_use) {
                queried = true;
                if (cudaEventQuery(old.ev_done) != cudaSuccess) { ++i; continue; }
            }
            bytes -= old.blob_bytes;
            gone[num_gone++] = old;
            p.idle.erase(p.idle.begin() + i);
        }
        if (queried) cudaGetLastError();                         // cudaErrorNotReady of a query is no error
        if (p.idle.size() < kMaxIdle && bytes + r.blob_bytes <= kMaxIdleBytes) {
            p.idle.push_back(r);
            r = PlanRes{};
        }
    }
    cudaError_t first = plan_res_free(r);                        // nothing, if it waits in the list
    for (size_t i = 0; i < num_gone; ++i) {
        const cudaError_t e = plan_res_free(gone[i]);
        if (first == cudaSuccess) first = e;
    }
    return first;
}

int64_t plan_res_allocs() { return g_allocs.load(std::memory_order_relaxed); }

cudaError_t plan_res_upload(PlanRes& r, const UploadPart* parts, size_t num_parts, size_t bytes) {
    Pool& p = pool();
    std::lock_guard<std::mutex> lock(p.up_mu);
    cudaStream_t s = nullptr;
    for (auto& d : p.up_streams)
        if (d.first == r.device) s = d.second;
    cudaError_t e = cudaSuccess;
    if (!s) {
        if ((e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking)) != cudaSuccess) return e;
        p.up_streams.emplace_back(r.device, s);
    }
    if (p.up_bytes < bytes) {
        if (p.up_buf) cudaFreeHost(p.up_buf);
        p.up_bytes = std::max(bytes, size_t(1) << 20);
        if ((e = cudaMallocHost(&p.up_buf, p.up_bytes)) != cudaSuccess) { p.up_buf = nullptr; p.up_bytes = 0; return e; }
    }
    for (size_t i = 0; i < num_parts; ++i)
        if (parts[i].bytes) std::memcpy(static_cast<char*>(p.up_buf) + parts[i].off, parts[i].src, parts[i].bytes);
    // a stream of its own: the copy does not queue behind the caller's kernels, and the plan is complete on return
    e = cudaMemcpyAsync(r.blob, p.up_buf, bytes, cudaMemcpyHostToDevice, s);
    return e == cudaSuccess ? cudaStreamSynchronize(s) : e;
}

cudaError_t plan_res_trim() {
    Pool& p = pool();
    std::vector<PlanRes> gone;
    gone.reserve(kMaxIdle);                                      // what the list has afterwards
    {
        std::lock_guard<std::mutex> lock(p.mu);
        gone.swap(p.idle);
    }
    {
        std::lock_guard<std::mutex> lock(p.up_mu);
        if (p.up_buf) cudaFreeHost(p.up_buf);
        p.up_buf = nullptr;
        p.up_bytes = 0;
    }
    cudaError_t first = cudaSuccess;
    int back = 0;
    cudaGetDevice(&back);
    for (PlanRes& r : gone) {
        cudaSetDevice(r.device);
        const cudaError_t e = plan_res_free(r);
        if (first == cudaSuccess) first = e;
    }
    if (!gone.empty()) cudaSetDevice(back);
    return first;
}

void plan_note_call(hat_plan* p, cudaStream_t s) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) == cudaSuccess && cap != cudaStreamCaptureStatusNone) { p->captured = true; return; }
    if (p->loose && p->loose_stream != s) p->loose_many = true;
    p->loose = true;
    p->loose_stream = s;
}

}  // namespace hat
