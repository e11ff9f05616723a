// What destroyed plans hand on to later ones: device memory, the pinned buffer it is filled from, and events.
//
// A serving loop makes one plan per inference step.  With a few GB of pools on the device a cudaMalloc / cudaFree pair
// costs 360 + 270 us of host time (measured beside 6 GB, 12 requests), both synchronise the device, and a pageable
// cudaMemcpy on the legacy stream waits for the previous step's kernels: together more than the eight layers of the
// step take on the GPU.  The pool turns that into a search of a short list and one small asynchronous copy.
//
// Bounds: at most kMaxIdle entries and kMaxIdleBytes of device memory wait in the list, per process; what does not fit
// is freed, and hat_release_cached() frees the rest.  Entries are handed on whole under one lock; an entry whose last
// owner's kernels may still run is taken only after that owner's ev_done has occurred.
#include <cstring>
#include <mutex>
#include <vector>

#include "hat_internal.h"

namespace hat {
namespace {

constexpr size_t kMaxIdle = 16;
constexpr size_t kMaxIdleBytes = size_t(64) << 20;

struct Pool {
    std::mutex mu;
    std::vector<PlanRes> idle;
    std::vector<std::pair<int, cudaStream_t>> upload;   // per device: the stream uploads run on
};
Pool& pool() {
    static Pool* p = new Pool();      // never destroyed: plans may outlive static destructors
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
    if (r.blob) e = cudaFree(r.blob);              // waits for the device, so kernels that still use the plan finish first
    if (r.pinned) cudaFreeHost(r.pinned);
    r = PlanRes{};
    return e;
}

cudaError_t plan_res_acquire(int device, size_t blob_bytes, size_t pinned_bytes, PlanRes* out) {
    Pool& p = pool();
    {
        std::unique_lock<std::mutex> lock(p.mu);
        int ready = -1, oldest = -1;
        for (int i = 0; i < (int)p.idle.size(); ++i) {          // in the order they were given back
            PlanRes& r = p.idle[i];
            // not for a plan that needs a small part of it only: the large ones would all end up with small plans
            if (r.device != device || r.blob_bytes < blob_bytes || r.pinned_bytes < pinned_bytes || r.blob_bytes / 8 > blob_bytes) continue;
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
    auto up = [](size_t n) { size_t m = size_t(64) << 10; while (m < n) m *= 2; return m; };
    r.blob_bytes = up(blob_bytes);
    r.pinned_bytes = up(pinned_bytes);
    cudaError_t e = cudaMalloc(&r.blob, r.blob_bytes);
    if (e == cudaErrorMemoryAllocation) {                        // give back what waits in the list and try once more
        cudaGetLastError();
        plan_res_trim();
        e = cudaMalloc(&r.blob, r.blob_bytes);
    }
    if (e != cudaSuccess) r.blob = nullptr;
    if (e == cudaSuccess && (e = cudaMallocHost(&r.pinned, r.pinned_bytes)) != cudaSuccess) r.pinned = nullptr;
    for (cudaEvent_t* ev : {&r.ev_verify, &r.ev_done, &r.ev_table})
        if (e == cudaSuccess && (e = cudaEventCreateWithFlags(ev, cudaEventDisableTiming)) != cudaSuccess) *ev = nullptr;
    if (e != cudaSuccess) { plan_res_free(r); return e; }
    *out = r;
    return cudaSuccess;
}

cudaError_t plan_res_release(PlanRes& r, bool reusable) {
    if (!r.blob) return plan_res_free(r);
    if (reusable) {
        Pool& p = pool();
        std::lock_guard<std::mutex> lock(p.mu);
        if (p.idle.size() < kMaxIdle && idle_bytes(p.idle) + r.blob_bytes <= kMaxIdleBytes) {
            p.idle.push_back(r);
            r = PlanRes{};
            return cudaSuccess;
        }
    }
    return plan_res_free(r);
}

cudaError_t plan_res_upload(PlanRes& r, size_t bytes) {
    Pool& p = pool();
    cudaStream_t s = nullptr;
    {
        std::lock_guard<std::mutex> lock(p.mu);
        for (auto& d : p.upload)
            if (d.first == r.device) s = d.second;
        if (!s) {
            const cudaError_t e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
            if (e != cudaSuccess) return e;
            p.upload.emplace_back(r.device, s);
        }
    }
    // a stream of its own: the copy does not queue behind the caller's kernels, and the plan is complete on return
    cudaError_t e = cudaMemcpyAsync(r.blob, r.pinned, bytes, cudaMemcpyHostToDevice, s);
    return e == cudaSuccess ? cudaStreamSynchronize(s) : e;
}

cudaError_t plan_res_trim() {
    Pool& p = pool();
    std::vector<PlanRes> gone;
    {
        std::lock_guard<std::mutex> lock(p.mu);
        gone.swap(p.idle);
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
