// Rotary position encoding fused into the KV append, and the same rotation for the query rows.
//
// The decoder layers of the paper's models (Vicuna-7B/13B, Sec. 4.1) rotate query and key rows by their token position
// before the attention of Sec. 2.1, and the cache stores the rotated keys.  Row i of request r has position
// p = prefix_len[r] + i; pair c of a head (c = 0 .. d/2 - 1) turns by p * theta^(-2c/d).  Pairs are (x[c], x[c + d/2])
// or, interleaved, (x[2c], x[2c + 1]).  The angle is formed and reduced to [-pi, pi] in double (at position 8000 an fp32
// angle is already off by more than the 16-bit result resolves), sine, cosine and the rotation run in fp32, and the
// result is rounded to the 16-bit type once.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <cmath>

#include "hat_internal.h"
#include "tc5_ptx.cuh"

namespace hat {
namespace {

constexpr int kHeads = 4;      // heads per thread

template <bool BF16>
__device__ __forceinline__ float2 unpack2(uint32_t w) {
    if constexpr (BF16) return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
    else {
        const __half2 h = *reinterpret_cast<const __half2*>(&w);
        return __half22float2(h);
    }
}

// (cos, sin) of every row and pair: trig[t][c], position of row t = prefix_len[r] + (t - cu_chunk[r])
__global__ void __launch_bounds__(256) rope_table_kernel(DevicePlan plan, int half, const __grid_constant__ InvFreq fr,
                                                         float2* __restrict__ trig) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)plan.total_rows * half) return;
    const int t = (int)(idx / half), c = (int)(idx - (int64_t)t * half);
    const int r = plan.row_req[t];
    const int p = plan.prefix_len[r] + (t - plan.cu_chunk[r]);
    float s, co;
    rope_sincos(p, fr.f[c], &s, &co);
    trig[idx] = make_float2(co, s);
}

// One thread: for one packed row, one 16-byte vector of the low half of a head and its partner in the high half (or,
// interleaved, two neighbouring vectors) = 8 pairs, for kHeads heads: the 8 cosines and sines depend on the row and the pair
// only.  They come from the plan's table (TABLE), which the first call with a base fills and every layer of the step shares, or
// are computed here.  `to_cache`: rows are K rows and go to their slot of the pool, with the matching V vectors copied as they
// come; otherwise rows are written to `dst` at their packed position (query rows).
//
// Bound: HBM, once the angles (reduced in double) come from the table; before, they were most of the time.  All loads of a
// thread (16 vectors in the append) are in flight before the first rotation.  1518 rows x 40 heads, bf16, two
// calls: 28 us and a gap without the table, 15 us with it.
template <bool BF16, bool TABLE>
__global__ void __launch_bounds__(256)
rope_kernel(DevicePlan plan, int heads, int d, const __grid_constant__ InvFreq fr, const float2* __restrict__ trig, int interleaved,
            const uint4* src, uint4* dst, int to_cache, int64_t stride_page, int64_t stride_token,
            int64_t stride_head, uint4* __restrict__ k_pool, uint4* __restrict__ v_pool, const uint4* __restrict__ v_new, int64_t total) {
    tc5::pdl_launch_dependents();
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool in = idx < total;
    const int vec_per_head = d / 8, pairs_vec = vec_per_head / 2;        // vectors per head, vector pairs per head
    const int groups = (heads + kHeads - 1) / kHeads;
    const int t = in ? (int)(idx / ((int64_t)groups * pairs_vec)) : 0;
    const int within = in ? (int)(idx - (int64_t)t * groups * pairs_vec) : 0;
    const int hg = within / pairs_vec, pv = within - hg * pairs_vec;
    const int r = plan.row_req[t];
    const int p = plan.prefix_len[r] + (t - plan.cu_chunk[r]);
    int64_t pool_base = 0;
    if (to_cache) {
        const int page = plan.block_table[(int64_t)r * plan.max_pages + p / kPageSize];
        pool_base = ((int64_t)page * stride_page + (int64_t)(p % kPageSize) * stride_token) / 8;
    }
    tc5::pdl_wait();                                                     // up to here only the plan's own arrays were read
    if (!in) return;

    const int va = interleaved ? 2 * pv : pv;                            // the two vectors this thread owns in a head
    const int vb = interleaved ? 2 * pv + 1 : pv + pairs_vec;
    const int h0 = hg * kHeads;
    uint4 a[kHeads], b[kHeads], xa[kHeads], xb[kHeads];
#pragma unroll
    for (int i = 0; i < kHeads; ++i)
        if (h0 + i < heads) {
            const int64_t row_vec = ((int64_t)t * heads + h0 + i) * vec_per_head;
            a[i] = src[row_vec + va]; b[i] = src[row_vec + vb];          // (dst may be src)
            if (to_cache) { xa[i] = __ldg(v_new + row_vec + va); xb[i] = __ldg(v_new + row_vec + vb); }
        }
    float sn[8], cs[8];                                                  // pair 8 pv + k of every head
    if constexpr (TABLE) {
        const float4* tr = reinterpret_cast<const float4*>(trig + (int64_t)t * (d / 2) + 8 * pv);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float4 x = tr[k];                                      // two (cos, sin)
            cs[2 * k] = x.x; sn[2 * k] = x.y; cs[2 * k + 1] = x.z; sn[2 * k + 1] = x.w;
        }
    } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) rope_sincos(p, fr.f[8 * pv + k], &sn[k], &cs[k]);
    }
#pragma unroll
    for (int i = 0; i < kHeads; ++i) {
        if (h0 + i >= heads) break;
        uint32_t* aw = reinterpret_cast<uint32_t*>(&a[i]);
        uint32_t* bw = reinterpret_cast<uint32_t*>(&b[i]);
        if (interleaved) {
            // each 32-bit word is one pair: words of a are pairs 8 pv .. +3, words of b pairs 8 pv + 4 .. +7
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float2 x = unpack2<BF16>(aw[k]), y = unpack2<BF16>(bw[k]);
                aw[k] = pack_out16(x.x * cs[k] - x.y * sn[k], x.y * cs[k] + x.x * sn[k], BF16);
                bw[k] = pack_out16(y.x * cs[k + 4] - y.y * sn[k + 4], y.y * cs[k + 4] + y.x * sn[k + 4], BF16);
            }
        } else {
            // element e of a pairs with element e of b: pair 8 pv + e
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float2 x = unpack2<BF16>(aw[k]), y = unpack2<BF16>(bw[k]);
                aw[k] = pack_out16(x.x * cs[2 * k] - y.x * sn[2 * k], x.y * cs[2 * k + 1] - y.y * sn[2 * k + 1], BF16);
                bw[k] = pack_out16(y.x * cs[2 * k] + x.x * sn[2 * k], y.y * cs[2 * k + 1] + x.y * sn[2 * k + 1], BF16);
            }
        }
        if (to_cache) {
            const int64_t base = pool_base + (int64_t)(h0 + i) * stride_head / 8;
            k_pool[base + va] = a[i];
            k_pool[base + vb] = b[i];
            v_pool[base + va] = xa[i];
            v_pool[base + vb] = xb[i];
        } else {
            const int64_t row_vec = ((int64_t)t * heads + h0 + i) * vec_per_head;
            dst[row_vec + va] = a[i];
            dst[row_vec + vb] = b[i];
        }
    }
}

}  // namespace

static InvFreq inv_freq(float theta, int d) {
    InvFreq fr;
    for (int c = 0; c < 64; ++c) fr.f[c] = c < d / 2 ? std::pow((double)theta, -2.0 * c / d) : 0.0;
    return fr;
}

// The table depends on the plan's positions and on the base only: every layer of a step uses the one its first call filled.
cudaError_t plan_rope_table(const hat_plan* plan, float theta, cudaStream_t stream, bool replace, const float2** table) {
    hat_plan* mp = const_cast<hat_plan*>(plan);
    const int half = plan->head_dim / 2;
    *table = nullptr;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(stream, &cap);
    if (e != cudaSuccess) return e;
    auto fill = [&]() {
        const int64_t total = (int64_t)plan->total_rows * half;
        rope_table_kernel<<<(unsigned)((total + 255) / 256), 256, 0, stream>>>(plan->dev, half, inv_freq(theta, plan->head_dim), mp->rope_table);
        count_launch();
        return cudaGetLastError();
    };
    if (cap != cudaStreamCaptureStatusNone) {
        // Inside a stream capture nothing runs now: the fill becomes part of the captured graph, ahead of the call that needs it,
        // and every replay refills the table at a time the plan does not know of.
        if (!replace) return cudaSuccess;
        if ((e = fill()) != cudaSuccess) return e;
        mp->table_in_graph = true;
    } else if (mp->table_in_graph || mp->rope_theta != theta) {
        // (a table that a replay may have refilled since is not trusted)
        if (mp->rope_theta > 0.f || mp->table_in_graph) {
            if (!replace) return cudaSuccess;
            // a call with the previous base may still be reading the table that is about to be replaced (rare: one model
            // has one base)
            if (mp->rope_theta > 0.f && mp->rope_theta != theta && (e = cudaDeviceSynchronize()) != cudaSuccess) return e;
        }
        if ((e = fill()) != cudaSuccess) return e;
        if ((e = cudaEventRecord(mp->res.ev_table, stream)) != cudaSuccess) return e;
        mp->rope_theta = theta;
        mp->table_stream = stream;
    } else if (mp->table_stream != stream) {
        if ((e = cudaStreamWaitEvent(stream, mp->res.ev_table, 0)) != cudaSuccess) return e;
    }
    *table = mp->rope_table;
    return cudaSuccess;
}

cudaError_t launch_rope(const hat_plan* plan, int heads, float theta, int interleaved, const void* src, void* dst,
                        const CacheView* cache, void* k_pool, void* v_pool, const void* v_new, cudaStream_t stream) {
    const int d = plan->head_dim;
    const int64_t total = (int64_t)plan->total_rows * ((heads + kHeads - 1) / kHeads) * (d / 16);
    if (total == 0) return cudaSuccess;
    // a plan whose table holds another base: compute the angles in the kernel instead of replacing it call by call
    const float2* trig = nullptr;
    cudaError_t e = plan_rope_table(plan, theta, stream, /*replace=*/false, &trig);
    if (e != cudaSuccess) return e;
    const int to_cache = cache != nullptr;
    const int64_t sp = to_cache ? cache->stride_page : 0, st = to_cache ? cache->stride_token : 0,
                  sh = to_cache ? cache->stride_head : 0;
    const bool bf16 = plan->dtype == HAT_DTYPE_BF16;
    auto kern = trig ? (bf16 ? rope_kernel<true, true> : rope_kernel<false, true>) : (bf16 ? rope_kernel<true, false> : rope_kernel<false, false>);
    return launch_pdl(kern, dim3((unsigned)((total + 255) / 256)), dim3(256), 0, stream, plan->dev, heads, d, trig ? InvFreq{} : inv_freq(theta, d),
                      trig, interleaved, static_cast<const uint4*>(src), static_cast<uint4*>(dst), to_cache, sp, st, sh,
                      static_cast<uint4*>(k_pool), static_cast<uint4*>(v_pool), static_cast<const uint4*>(v_new), total);
}

}  // namespace hat
