// Block-wise absmax INT8 quantisation and dequantisation (paper Section IV-D, Eq. 1-2):
//   c = 127 / absmax(block),  code = round(c * x)  (ties to even),  dequant = code / c,
// every block of `block` consecutive elements on its own; an all-zero block has c = 0.
// All arithmetic in fp32 with explicitly rounded operations, so the integer codes are the same
// on every implementation that follows the equations in fp32.  Both kernels stream: 5 bytes per
// element (4 read + 1 written, or the reverse).
#pragma once
#include "pac_common.cuh"

namespace pac {

// One warp per quantisation block (block <= QUANT_WARP_MAX), several blocks per CTA.
constexpr int QUANT_WARP_MAX = 4096;

__global__ void __launch_bounds__(256) quantize_absmax_warp_kernel(const float* __restrict__ x, long long n, int block,
                                                                   long long n_blocks, signed char* __restrict__ q,
                                                                   float* __restrict__ c) {
    const int lane = threadIdx.x & 31;
    const long long wid = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long j = wid; j < n_blocks; j += nw) {
        const long long i0 = j * block;
        const int len = (int)((n - i0) < block ? (n - i0) : block);
        float amax = 0.f;
        for (int i = lane; i < len; i += 32) amax = fmaxf(amax, fabsf(x[i0 + i]));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
        const float cj = amax > 0.f ? __fdiv_rn(127.f, amax) : 0.f;
        if (lane == 0) c[j] = cj;
        for (int i = lane; i < len; i += 32)                        // second read comes from L1/L2
            q[i0 + i] = (signed char)__float2int_rn(__fmul_rn(cj, x[i0 + i]));
    }
}

// One CTA per quantisation block (large blocks).
__global__ void __launch_bounds__(256) quantize_absmax_cta_kernel(const float* __restrict__ x, long long n, int block,
                                                                  signed char* __restrict__ q, float* __restrict__ c) {
    __shared__ float red[8];
    __shared__ float c_sh;
    const long long j = blockIdx.x, i0 = j * block;
    const int len = (int)((n - i0) < block ? (n - i0) : block);
    float amax = 0.f;
    for (int i = threadIdx.x; i < len; i += blockDim.x) amax = fmaxf(amax, fabsf(x[i0 + i]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = amax;
    __syncthreads();
    if (threadIdx.x == 0) {
        float m = 0.f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = fmaxf(m, red[w]);
        c_sh = m > 0.f ? __fdiv_rn(127.f, m) : 0.f;
        c[j] = c_sh;
    }
    __syncthreads();
    const float cj = c_sh;
    for (int i = threadIdx.x; i < len; i += blockDim.x) q[i0 + i] = (signed char)__float2int_rn(__fmul_rn(cj, x[i0 + i]));
}

__device__ __forceinline__ float absmax4(float4 v) { return fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))); }
// round(c x) as the low byte of c x + 1.5 * 2^23 (the sum is rounded to an integer, ties to even; |c x| <= 127.00001), without the
// quarter-rate conversion; products out of range (not finite) take the conversion.
__device__ __forceinline__ uint32_t quant_bits(float x, float cj) {
    const float v = __fmul_rn(cj, x);
    uint32_t b = __float_as_uint(__fadd_rn(v, 12582912.f));
    if (!(fabsf(v) <= 128.f)) b = (uint32_t)__float2int_rn(v);
    return b;
}
__device__ __forceinline__ uint32_t quant_pack4(float a, float b, float c, float d, float cj) {
    const uint32_t lo = __byte_perm(quant_bits(a, cj), quant_bits(b, cj), 0x0040), hi = __byte_perm(quant_bits(c, cj), quant_bits(d, cj), 0x0040);
    return __byte_perm(lo, hi, 0x5410);
}
// 32 bytes in one access (p 32-byte aligned).
__device__ __forceinline__ void ld_global_32(const float* p, float (&v)[8]) {
    asm volatile("ld.global.nc.L1::no_allocate.L2::evict_first.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]) : "l"(p));
}
__device__ __forceinline__ void st_global_32f(float* p, const float (&v)[8]) {
    asm volatile("st.global.L1::no_allocate.L2::evict_first.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]) : "memory");
}

// What is read or written once and larger (values) gives way in L2 to the codes, which the reader of both directions then finds there:
// 4096 x 11008 values at block 64, both directions 78.6 -> 68.7 us.
// Block = 16, 32, ... 512: a lane owns 16 consecutive values (two 32-byte loads, one 16-byte store), block / 16 lanes share a block
// and one division.  Any n: the last group is handled value by value.  Bound by HBM; with one 16-byte load per thread in flight
// and a division per four values the same blocks took 0.66 of the copy bandwidth.
__global__ void __launch_bounds__(256) quantize_absmax_subwarp_kernel(const float* __restrict__ x, long long n, int lanes_log2,
                                                                      signed char* __restrict__ q, float* __restrict__ c) {
    const long long groups = (n + 15) >> 4, pad = (groups + 31) & ~31LL, stride = (long long)gridDim.x * blockDim.x;
    for (long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x; g < pad; g += stride) {      // whole warps stay together for the shuffles
        const long long i = g << 4;
        float v[2][8] = {};
        if (i + 16 <= n) {
            ld_global_32(x + i, v[0]);
            ld_global_32(x + i + 8, v[1]);
        } else {
#pragma unroll
            for (int e = 0; e < 16; ++e) if (i + e < n) v[e >> 3][e & 7] = x[i + e];
        }
        float amax = 0.f;
#pragma unroll
        for (int e = 0; e < 16; ++e) amax = fmaxf(amax, fabsf(v[e >> 3][e & 7]));
        for (int o = 1; o < (1 << lanes_log2); o <<= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
        const float cj = amax > 0.f ? __fdiv_rn(127.f, amax) : 0.f;
        uint32_t w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float* p = &v[e >> 1][(e & 1) * 4];
            w[e] = quant_pack4(p[0], p[1], p[2], p[3], cj);
        }
        if (i + 16 <= n) {
            *reinterpret_cast<uint4*>(q + i) = make_uint4(w[0], w[1], w[2], w[3]);
        } else {
#pragma unroll
            for (int e = 0; e < 16; ++e) if (i + e < n) q[i + e] = (signed char)(w[e >> 2] >> (8 * (e & 3)));
        }
        if ((g & ((1 << lanes_log2) - 1)) == 0 && i < n) c[g >> lanes_log2] = cj;
    }
}

// Block a multiple of 4 up to 128 PER (any remainder of n): 8 / PER blocks per warp at a time, eight 16-byte loads per lane in flight.
// (One block at a time left a lane one load for blocks of 100: both directions of 2^26 values 282 us; so 158 with the reader below.)
template <int PER>
__global__ void __launch_bounds__(256) quantize_absmax_warp4_kernel(const float* __restrict__ x, long long n, int block, long long n_blocks,
                                                                    signed char* __restrict__ q, float* __restrict__ c) {
    constexpr int NB = 8 / PER;
    const int lane = threadIdx.x & 31;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long j = (((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * NB; j < n_blocks; j += nw * NB) {
        float4 v[NB][PER];
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const long long i0 = (j + b) * block;
            const int len = (int)(n - i0 < block ? (n - i0 > 0 ? n - i0 : 0) : block);
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                const int e = (k * 32 + lane) * 4;
                v[b][k] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (e + 4 <= len) v[b][k] = __ldcs(reinterpret_cast<const float4*>(x + i0 + e));
                else if (e < len) {
                    v[b][k].x = x[i0 + e];
                    if (e + 1 < len) v[b][k].y = x[i0 + e + 1];
                    if (e + 2 < len) v[b][k].z = x[i0 + e + 2];
                }
            }
        }
        float amax[NB];
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            amax[b] = 0.f;
#pragma unroll
            for (int k = 0; k < PER; ++k) amax[b] = fmaxf(amax[b], absmax4(v[b][k]));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int b = 0; b < NB; ++b) amax[b] = fmaxf(amax[b], __shfl_xor_sync(0xffffffffu, amax[b], o));
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const long long i0 = (j + b) * block;
            const int len = (int)(n - i0 < block ? (n - i0 > 0 ? n - i0 : 0) : block);
            const float cj = amax[b] > 0.f ? __fdiv_rn(127.f, amax[b]) : 0.f;
            if (lane == 0 && len > 0) c[j + b] = cj;
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                const int e = (k * 32 + lane) * 4;
                if (e >= len) continue;
                const uint32_t w = quant_pack4(v[b][k].x, v[b][k].y, v[b][k].z, v[b][k].w, cj);
                if (e + 4 <= len) *reinterpret_cast<uint32_t*>(q + i0 + e) = w;
                else
                    for (int t = 0; e + t < len; ++t) q[i0 + e + t] = (signed char)(w >> (8 * t));
            }
        }
    }
}

// Single pass, one CTA of 256 threads per block, block = 1024 * K (2 <= K <= 4), any n.
template <int K>
__global__ void __launch_bounds__(256) quantize_absmax_cta_reg_kernel(const float* __restrict__ x, long long n,
                                                                      signed char* __restrict__ q, float* __restrict__ c) {
    __shared__ float red[8];
    __shared__ float c_sh;
    const long long base = (long long)blockIdx.x * (1024 * K);
    float4 v[K];
    float amax = 0.f;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const long long i = base + (k * 256 + threadIdx.x) * 4;
        v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i + 4 <= n) v[k] = __ldcs(reinterpret_cast<const float4*>(x + i));
        else if (i < n) {
            v[k].x = x[i];
            if (i + 1 < n) v[k].y = x[i + 1];
            if (i + 2 < n) v[k].z = x[i + 2];
        }
        amax = fmaxf(amax, absmax4(v[k]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = amax;
    __syncthreads();
    if (threadIdx.x == 0) {
        float m = 0.f;
        for (int w = 0; w < 8; ++w) m = fmaxf(m, red[w]);
        c_sh = m > 0.f ? __fdiv_rn(127.f, m) : 0.f;
        c[blockIdx.x] = c_sh;
    }
    __syncthreads();
    const float cj = c_sh;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const long long i = base + (k * 256 + threadIdx.x) * 4;
        const uint32_t w = quant_pack4(v[k].x, v[k].y, v[k].z, v[k].w, cj);
        if (i + 4 <= n) *reinterpret_cast<uint32_t*>(q + i) = w;
        else
            for (int b = 0; i + b < n; ++b) q[i + b] = (signed char)(w >> (8 * b));
    }
}

// code / c, correctly rounded: with rc = RN(1 / c), y = RN(code rc) and the exact remainder e = code - y c, RN(y + e rc) is the
// rounded quotient (Markstein's theorem; confirmed for all 2^23 significands of c and all codes).  Outside 2^-100 .. 2^100 (and for
// c = 0 or not a number) the scale is left to the division.
struct DequantScale {
    float c, rc;
    bool plain;
    __device__ __forceinline__ explicit DequantScale(float c_) : c(c_) {
        plain = !(c_ >= 0x1p-100f && c_ <= 0x1p100f);
        rc = plain ? 0.f : __fdiv_rn(1.f, c_);
    }
    __device__ __forceinline__ float operator()(float code) const {
        const float y = __fmul_rn(code, rc);
        return __fmaf_rn(__fmaf_rn(-y, c, code), rc, y);
    }
    __device__ __forceinline__ float slow(float code) const { return c != 0.f ? __fdiv_rn(code, c) : 0.f; }
};
// Byte k of w as a float: 2^23 + (code + 128), less 2^23 + 128.
__device__ __forceinline__ float code_float(uint32_t w_plus, int k) {
    return __uint_as_float(__byte_perm(w_plus, 0x4B000000u, 0x7440 | k)) - 8388736.f;
}
__device__ __forceinline__ void dequant4(uint32_t w, const DequantScale& s, float* o) {
    w ^= 0x80808080u;
#pragma unroll
    for (int k = 0; k < 4; ++k) o[k] = s(code_float(w, k));
    if (s.plain)
#pragma unroll
        for (int k = 0; k < 4; ++k) o[k] = s.slow(code_float(w, k));
}

// Sixteen codes of one block per thread (block a multiple of 16): a 16-byte load, one reciprocal, two 32-byte stores.  Any n.
// `shift` >= 0: block / 16 = 2^shift.  Bound by HBM; a correctly rounded division per code took 0.44 of the copy bandwidth.
__global__ void __launch_bounds__(256) dequantize_absmax_16_kernel(const signed char* __restrict__ q, const float* __restrict__ c, long long n,
                                                                   int block16, int shift, float* __restrict__ out) {
    const long long groups = (n + 15) >> 4, stride = (long long)gridDim.x * blockDim.x;
    for (long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x; g < groups; g += stride) {
        const long long i = g << 4;
        const DequantScale s(__ldg(c + (shift >= 0 ? g >> shift : g / block16)));
        if (i + 16 <= n) {
            const uint4 w = __ldg(reinterpret_cast<const uint4*>(q + i));
            float a[8], b[8];
            dequant4(w.x, s, a); dequant4(w.y, s, a + 4); dequant4(w.z, s, b); dequant4(w.w, s, b + 4);
            st_global_32f(out + i, a);
            st_global_32f(out + i + 8, b);
        } else {
            for (int e = 0; i + e < n; ++e) out[i + e] = s.slow((float)q[i + e]);
        }
    }
}

// The same where sixteen codes may lie in two blocks (block a multiple of 4 from 16 on, n < 2^33): each four codes in one, the first four's found by
// a multiplication: group index (below 2^31) times ceil(2^(31 + s) / block4), 2^(s - 1) < block4 <= 2^s, shifted right by 31 + s (Granlund and Montgomery, PLDI 1994).
__global__ void __launch_bounds__(256) dequantize_absmax_16_any_kernel(const signed char* __restrict__ q, const float* __restrict__ c, long long n, long long n_blocks,
                                                                       uint32_t block4, uint32_t magic, int shift, float* __restrict__ out) {
    const long long groups = (n + 15) >> 4, stride = (long long)gridDim.x * blockDim.x;
    for (long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x; g < groups; g += stride) {
        const long long i = g << 4;
        const uint32_t i4 = (uint32_t)(g << 2), j = __umulhi(i4, magic) >> shift, edge = (j + 1) * block4;      // edge: first four codes of the next block
        const float c0 = __ldg(c + j), c1 = i4 + 4 > edge && j + 1 < n_blocks ? __ldg(c + j + 1) : c0;
        if (i + 16 <= n) {
            const uint4 w = __ldg(reinterpret_cast<const uint4*>(q + i));
            const DequantScale s0(c0), s1 = i4 + 4 > edge ? DequantScale(c1) : s0;
            float a[8], b[8];
            dequant4(w.x, s0, a);
            dequant4(w.y, i4 + 1 < edge ? s0 : s1, a + 4); dequant4(w.z, i4 + 2 < edge ? s0 : s1, b); dequant4(w.w, i4 + 3 < edge ? s0 : s1, b + 4);
            st_global_32f(out + i, a);
            st_global_32f(out + i + 8, b);
        } else {
            for (int e = 0; i + e < n; ++e) out[i + e] = DequantScale(i4 + (e >> 2) < edge ? c0 : c1).slow((float)q[i + e]);
        }
    }
}

// Four codes per thread (block a multiple of 4), four independent groups in flight.  Any n.
__global__ void __launch_bounds__(256) dequantize_absmax_vec_kernel(const signed char* __restrict__ q, const float* __restrict__ c,
                                                                    long long n, int block4, float* __restrict__ out) {
    const long long n4 = n >> 2, stride = (long long)gridDim.x * blockDim.x, t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool narrow = n4 <= 0x7fffffffLL;            // 32-bit index division
    for (long long i0 = t; i0 < n4; i0 += 4 * stride) {
        uint32_t b[4];
        float cj[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const long long i = i0 + k * stride;
            if (i < n4) { b[k] = __ldg(reinterpret_cast<const uint32_t*>(q) + i); cj[k] = __ldg(c + (narrow ? (long long)((uint32_t)i / (uint32_t)block4) : i / block4)); }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const long long i = i0 + k * stride;
            if (i < n4) {
                float o[4];
                dequant4(b[k], DequantScale(cj[k]), o);
                __stcs(reinterpret_cast<float4*>(out) + i, make_float4(o[0], o[1], o[2], o[3]));
            }
        }
    }
    if (t < (n & 3)) {
        const long long i = (n & ~3LL) + t;
        out[i] = DequantScale(c[i / (4LL * block4)]).slow((float)q[i]);
    }
}

__global__ void __launch_bounds__(256) dequantize_absmax_kernel(const signed char* __restrict__ q, const float* __restrict__ c,
                                                                long long n, int block, float* __restrict__ out) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const float cj = c[i / block];
        out[i] = cj != 0.f ? __fdiv_rn((float)q[i], cj) : 0.f;
    }
}

}  // namespace pac
