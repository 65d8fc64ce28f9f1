// Shared device helpers and the context structure of the adapter-over-cache trainer.
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cstdint>
#include <cstdio>
#include <map>
#include <mutex>
#include <string>
#include <utility>

#include "pac.h"

namespace pac {

typedef __nv_bfloat16 bf16;

__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(bf16 x) { return __bfloat162float(x); }

// Device-side status words (one small array per context).
// ST_SKIPPED_STEPS: optimizer updates that were left out because ST_TIMEOUT was already set when they ran.
enum { ST_CLAMPED_IDS = 0, ST_TIMEOUT = 1, ST_SKIPPED_STEPS = 2, ST_WORDS = 4 };
__device__ __forceinline__ bool status_timed_out(const unsigned* status) {
    return status && *reinterpret_cast<const volatile unsigned*>(status + ST_TIMEOUT) != 0u;
}

// Programmatic dependent launch: a kernel launched with the programmatic-serialization
// attribute may start while its predecessor in the stream is still running; pdl_wait() blocks
// until the predecessor grid has completed and its writes are visible, pdl_trigger() lets the
// successor start launching.  Without the attribute both are no-ops.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Sample id of batch row b, clamped into [0, N) so that no kernel can read outside
// the cache even if a device-resident id is bad; clamps are counted.
__device__ __forceinline__ long long safe_id(const int* __restrict__ ids, int b, long long N, unsigned* status) {
    long long id = ids[b];
    if (id < 0 || id >= N) {
        if (status) atomicAdd(&status[ST_CLAMPED_IDS], 1u);
        id = id < 0 ? 0 : N - 1;
    }
    return id;
}

// A minibatch's ids as a kernel argument (validated on the host): known before anything ahead in the stream has finished, at the price of one
// constant load.  160: the one-launch forward takes a sample per cluster and 148 SMs hold fewer clusters than that.
constexpr int ARG_IDS = 160;
struct ArgIds { int n, v[ARG_IDS]; };       // n == 0: ids in memory

// Dynamic shared memory above 48 KB needs an opt-in per kernel, and the attribute belongs to the
// device the call is made on.  Several contexts (other shapes, other devices) share the kernels, so
// the largest size granted so far is kept per (device, kernel) and never lowered.
inline cudaError_t smem_opt_in(const void* kernel, size_t bytes) {
    static std::mutex mu;
    static std::map<std::pair<int, const void*>, size_t> granted;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    size_t& g = granted[std::make_pair(dev, kernel)];
    if (bytes <= g) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) g = bytes;
    return e;
}

__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi) {
    uint32_t d;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}
// (x, y) = h + m + l exactly, each term a bf16 pair.
__device__ __forceinline__ void split3_pair(float x, float y, uint32_t& h, uint32_t& m, uint32_t& l) {
    h = bf16_pair(x, y);
    x -= __uint_as_float(h << 16); y -= __uint_as_float(h & 0xffff0000u);
    m = bf16_pair(x, y);
    x -= __uint_as_float(m << 16); y -= __uint_as_float(m & 0xffff0000u);
    l = bf16_pair(x, y);
}

// bf16 terms of W_down for the tensor-core products, [L][2][d][r] in the master's order: hi = bf16(W), lo = bf16(W - hi), together about 16
// mantissa bits.
struct WdShadow {
    bf16* p;
    // x into the terms of one element, `dr` apart.
    __device__ __forceinline__ void put(long long at, long long dr, float x) const {
        const bf16 a = __float2bfloat16(x);
        p[at] = a; p[at + dr] = __float2bfloat16(x - __bfloat162float(a));
    }
    __device__ __forceinline__ void put4(long long at, long long dr, const float (&x)[4]) const {
        bf16 v[2][4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            v[0][e] = __float2bfloat16(x[e]);
            v[1][e] = __float2bfloat16(x[e] - __bfloat162float(v[0][e]));
        }
        *reinterpret_cast<uint2*>(p + at) = *reinterpret_cast<const uint2*>(v[0]);
        *reinterpret_cast<uint2*>(p + at + dr) = *reinterpret_cast<const uint2*>(v[1]);
    }
};
// Layer of element i of the W_down block (dr = d r elements each): a 32-bit division where the block's size allows it.
__device__ __forceinline__ int wd_layer(long long i, long long lam, unsigned dr) {
    return lam <= 0x7fffffffLL ? (int)((unsigned)i / dr) : (int)(i / dr);
}

struct Dims {
    long long N;   // samples in the cache
    int L, S, d;   // layers, tokens, hidden width
    int r;         // adapter width
    int C;         // classes or vocabulary
};

// Offsets of the flat fp32 parameter vector:
// W_down[L][d][r] | lambda[L] | W_up[r][d] | W_head[d][C] | b_head[C]
// With transformer-body adapters the per-layer body blocks follow, layer after layer:
// ... | body[0] | body[1] | ... | body[L-1],  body[l] = g1 | b1 | Wq | Wk | Wv | Wo | g2 | b2 | W1 | c1 | W2 | c2
struct ParamLayout {
    long long w_down, lam, w_up, w_head, b_head, total;
    long long body, body_per;        // first body block and floats per block (body_per == 0: point-wise adapters)
    int br, bf;                      // adapter width and FFN width of the body blocks
    __host__ __device__ static ParamLayout make(int L, int d, int r, int C, bool cls) {
        ParamLayout p;
        p.w_down = 0;
        p.lam = (long long)L * d * r;
        p.w_up = p.lam + L;
        p.w_head = p.w_up + (long long)r * d;
        p.b_head = p.w_head + (cls ? (long long)d * C : 0);
        p.total = p.b_head + (cls ? C : 0);
        p.body = p.total; p.body_per = 0; p.br = r; p.bf = 0;
        return p;
    }
    // decoupled weight decay: the weight matrices, not lambda, biases or LayerNorm parameters
    __host__ __device__ bool decays(long long i) const {
        if (i < lam) return true;
        if (i < body) return i >= w_up && i < b_head;
        const long long off = (i - body) % body_per, rr = (long long)br * br, rf = (long long)br * bf;
        const long long wq = 2LL * br, g2 = wq + 4 * rr, w1 = g2 + 2LL * br, c1 = w1 + rf, w2 = c1 + bf, c2 = w2 + rf;
        return (off >= wq && off < g2) || (off >= w1 && off < c1) || (off >= w2 && off < c2);
    }
};

}  // namespace pac
