// Register-tiled fp32 products over rows of the activation cache and over the plain path's row-major
// stacks.  They carry the configurations whose precision rules out reduced-precision operands (fp32
// caches, transformer-body adapters) and the shapes TMA cannot address.
//
//   sgemm_rows_kernel   out[z][m][j]  = sum_k rows(z; m, k) W[z][k][j]      (u_l = h_l W_down^l)
//   sgemm_tn_kernel     out[i][j]     = sum_m A[m][i] B[m][j]               (dW = A^T B over all token rows)
//
// Both are bound by the FP32 pipe (128 FMA per SM and clock).  A thread owns TM x TN outputs; the operands
// of a K step are staged once per CTA in shared memory, fetched into registers while the step before is
// multiplied.  TM x TN = 8 x 4 needs 16 shared-memory wavefronts per 128 FMA instructions of a warp, half of
// what the pipe leaves room for; the 4 x 4 tiles of the generic gemm_simt need as many as there are.
// Every output is summed by one thread in ascending k (per k slice), so results do not depend on timing.
#pragma once
#include "pac_common.cuh"

namespace pac {

// Four consecutive columns of a row (zeros beyond n); `vec`: rows start on a four-element boundary.
__device__ __forceinline__ float4 load_row4(const float* __restrict__ row, int c, int n, bool vec) {
    if (vec && c + 3 < n) return __ldg(reinterpret_cast<const float4*>(row + c));
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (c < n) v.x = __ldg(row + c);
    if (c + 1 < n) v.y = __ldg(row + c + 1);
    if (c + 2 < n) v.z = __ldg(row + c + 2);
    if (c + 3 < n) v.w = __ldg(row + c + 3);
    return v;
}
__device__ __forceinline__ float4 load_row4(const bf16* __restrict__ row, int c, int n, bool vec) {
    if (vec && c + 3 < n) {
        const uint2 q = __ldg(reinterpret_cast<const uint2*>(row + c));
        return make_float4(__uint_as_float(q.x << 16), __uint_as_float(q.x & 0xffff0000u), __uint_as_float(q.y << 16),
                           __uint_as_float(q.y & 0xffff0000u));
    }
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (c < n) v.x = to_f32(row[c]);
    if (c + 1 < n) v.y = to_f32(row[c + 1]);
    if (c + 2 < n) v.z = to_f32(row[c + 2]);
    if (c + 3 < n) v.w = to_f32(row[c + 3]);
    return v;
}

// Row m of the minibatch at layer z, straight from the cache (the gather is the address).
template <typename T>
struct SgCacheRows {
    typedef T elem;
    const T* cache; const int* ids; long long N; int L, S, d;
    bool vec;                                   // d % 4 == 0
    __device__ const T* row(int z, int m) const {
        const int b = m / S, s = m - b * S;
        return cache + ((safe_id(ids, b, N, nullptr) * L + z) * S + s) * (long long)d;
    }
};
// Row m of a row-major fp32 stack.
struct SgRows {
    typedef float elem;
    const float* base; long long zstride; int ld;
    bool vec;                                   // base 16-byte aligned, ld and zstride multiples of 4
    __device__ const float* row(int z, int m) const { return base + z * zstride + (long long)m * ld; }
};

constexpr int SG_KR = 32;                       // K extent of a stage (sgemm_rows_kernel)

// BM x BN outputs per CTA of (BM / TM) * (BN / TN) threads.  A is staged as it lies, [m][k] (stride SG_KR + 4:
// 16-byte rows, and the few rows a warp reads at a time fall into different banks), and read four k at a
// time; W as [k][j].
template <int BM, int BN, int TM, int TN, class AL>
__global__ void __launch_bounds__((BM / TM) * (BN / TN))
sgemm_rows_kernel(int M, int N, int K, AL A, SgRows W, float* __restrict__ out, long long zstride) {
    constexpr int NT = (BM / TM) * (BN / TN), TX = BN / TN;
    constexpr int LA = SG_KR + 4, LB = BN + 4;
    constexpr int QA = BM * SG_KR / 4 / NT, QB = (SG_KR * BN / 4 + NT - 1) / NT;
    static_assert(BM * SG_KR / 4 % NT == 0, "the A tile is dealt out evenly");
    __shared__ __align__(16) float As[BM * LA], Bs[SG_KR * LB];
    const int z = blockIdx.z, m0 = blockIdx.y * BM, j0 = blockIdx.x * BN;
    const int t = threadIdx.x, tx = t % TX, ty = t / TX;
    // this thread's slice of the A tile: rows ar + q * (NT / 8), four columns at ac
    const int ar = t / (SG_KR / 4), ac = (t % (SG_KR / 4)) * 4;
    const typename AL::elem* arow[QA];
    bool alive[QA];
#pragma unroll
    for (int q = 0; q < QA; ++q) {
        const int m = m0 + ar + q * (NT / (SG_KR / 4));
        alive[q] = m < M;
        arow[q] = A.row(z, alive[q] ? m : m0);
    }
    float4 ra[QA], rb[QB];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int q = 0; q < QA; ++q)
            ra[q] = alive[q] ? load_row4(arow[q], k0 + ac, K, A.vec) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int q = 0; q < QB; ++q) {
            const int e = t + q * NT, k = e / (BN / 4), j = (e % (BN / 4)) * 4;
            rb[q] = (e < SG_KR * BN / 4 && k0 + k < K) ? load_row4(W.row(z, k0 + k), j0 + j, N, W.vec) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    float acc[TM][TN] = {};
    fetch(0);
    for (int k0 = 0; k0 < K; k0 += SG_KR) {
#pragma unroll
        for (int q = 0; q < QA; ++q) *reinterpret_cast<float4*>(As + (ar + q * (NT / (SG_KR / 4))) * LA + ac) = ra[q];
#pragma unroll
        for (int q = 0; q < QB; ++q) {
            const int e = t + q * NT;
            if (e < SG_KR * BN / 4) *reinterpret_cast<float4*>(Bs + (e / (BN / 4)) * LB + (e % (BN / 4)) * 4) = rb[q];
        }
        __syncthreads();
        if (k0 + SG_KR < K) fetch(k0 + SG_KR);
#pragma unroll
        for (int k = 0; k < SG_KR; k += 4) {
            float b[4][TN];
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                if constexpr (TN == 4) {
                    const float4 v = *reinterpret_cast<const float4*>(Bs + (k + kk) * LB + tx * 4);
                    b[kk][0] = v.x; b[kk][1] = v.y; b[kk][2] = v.z; b[kk][3] = v.w;
                } else {
#pragma unroll
                    for (int n = 0; n < TN; ++n) b[kk][n] = Bs[(k + kk) * LB + tx * TN + n];
                }
            }
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                const float4 a = *reinterpret_cast<const float4*>(As + (ty + i * (BM / TM)) * LA + k);
#pragma unroll
                for (int n = 0; n < TN; ++n) {
                    acc[i][n] = fmaf(a.x, b[0][n], acc[i][n]);
                    acc[i][n] = fmaf(a.y, b[1][n], acc[i][n]);
                    acc[i][n] = fmaf(a.z, b[2][n], acc[i][n]);
                    acc[i][n] = fmaf(a.w, b[3][n], acc[i][n]);
                }
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int m = m0 + ty + i * (BM / TM);
        if (m >= M) continue;
        float* o = out + z * zstride + (long long)m * N;
#pragma unroll
        for (int n = 0; n < TN; ++n) {
            const int j = j0 + tx * TN + n;
            if (j < N) o[j] = acc[i][n];
        }
    }
}

// ---------------------------------------------------------------------------
// A^T B over all rows.  A launch covers several products per layer (jobs) and all layers; a CTA owns one
// tile of one product and one slice of the rows.  With more than one slice the partial sums of slice s go
// to out + s * part_stride and are added up in slice order by whoever reads them.
// ---------------------------------------------------------------------------
constexpr int TN_MAX_JOBS = 6;
constexpr int TN_KR = 32;                       // token rows per stage
template <class AL>
struct TnJobs {
    AL A[TN_MAX_JOBS];
    SgRows B[TN_MAX_JOBS];
    int mi[TN_MAX_JOBS], nj[TN_MAX_JOBS];       // output extent
    int tiles_j[TN_MAX_JOBS], first[TN_MAX_JOBS + 1];      // tiles along j; first tile of the job
    long long out_off[TN_MAX_JOBS];
    int n = 0;
    int tile_i = 0, tile_j = 0;
    void add(const AL& a, int mi_, const SgRows& b, int nj_, long long off) {
        A[n] = a; B[n] = b; mi[n] = mi_; nj[n] = nj_; out_off[n] = off;
        tiles_j[n] = (nj_ + tile_j - 1) / tile_j;
        if (n == 0) first[0] = 0;
        first[n + 1] = first[n] + tiles_j[n] * ((mi_ + tile_i - 1) / tile_i);
        ++n;
    }
};

template <int BI, int BJ, int TI, int TJ, class AL>
__global__ void __launch_bounds__((BI / TI) * (BJ / TJ))
sgemm_tn_kernel(TnJobs<AL> J, int M, int m_slice, float* __restrict__ out, long long zstride, long long part_stride) {
    constexpr int NT = (BI / TI) * (BJ / TJ), TX = BJ / TJ;
    constexpr int LA = BI + 4, LB = BJ + 4;
    constexpr int QA = (TN_KR * BI / 4 + NT - 1) / NT, QB = (TN_KR * BJ / 4 + NT - 1) / NT;
    __shared__ __align__(16) float As[TN_KR * LA], Bs[TN_KR * LB];
    const int z = blockIdx.y, t = threadIdx.x, tx = t % TX, ty = t / TX;
    int jb = 0;
    while (jb + 1 < J.n && (int)blockIdx.x >= J.first[jb + 1]) ++jb;
    const int tile = blockIdx.x - J.first[jb];
    const int i0 = tile / J.tiles_j[jb] * BI, j0 = tile % J.tiles_j[jb] * BJ;
    const AL A = J.A[jb];
    const SgRows B = J.B[jb];
    const int Mi = J.mi[jb], Nj = J.nj[jb];
    const int mb = blockIdx.z * m_slice, me = min(M, mb + m_slice);
    float4 ra[QA], rb[QB];
    auto fetch = [&](int m0) {
#pragma unroll
        for (int q = 0; q < QA; ++q) {
            const int e = t + q * NT, m = m0 + e / (BI / 4), i = (e % (BI / 4)) * 4;
            ra[q] = (e < TN_KR * BI / 4 && m < me) ? load_row4(A.row(z, m), i0 + i, Mi, A.vec) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int q = 0; q < QB; ++q) {
            const int e = t + q * NT, m = m0 + e / (BJ / 4), j = (e % (BJ / 4)) * 4;
            rb[q] = (e < TN_KR * BJ / 4 && m < me) ? load_row4(B.row(z, m), j0 + j, Nj, B.vec) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    float acc[TI][TJ] = {};
    if (mb < me) fetch(mb);
    for (int m0 = mb; m0 < me; m0 += TN_KR) {
#pragma unroll
        for (int q = 0; q < QA; ++q) {
            const int e = t + q * NT;
            if (e < TN_KR * BI / 4) *reinterpret_cast<float4*>(As + (e / (BI / 4)) * LA + (e % (BI / 4)) * 4) = ra[q];
        }
#pragma unroll
        for (int q = 0; q < QB; ++q) {
            const int e = t + q * NT;
            if (e < TN_KR * BJ / 4) *reinterpret_cast<float4*>(Bs + (e / (BJ / 4)) * LB + (e % (BJ / 4)) * 4) = rb[q];
        }
        __syncthreads();
        if (m0 + TN_KR < me) fetch(m0 + TN_KR);
#pragma unroll 8
        for (int k = 0; k < TN_KR; ++k) {
            float a[TI], b[TJ];
#pragma unroll
            for (int i = 0; i < TI; i += 4) {
                const float4 v = *reinterpret_cast<const float4*>(As + k * LA + ty * 4 + (i / 4) * (BI / TI * 4));
                a[i] = v.x; a[i + 1] = v.y; a[i + 2] = v.z; a[i + 3] = v.w;
            }
            if constexpr (TJ == 4) {
                const float4 v = *reinterpret_cast<const float4*>(Bs + k * LB + tx * 4);
                b[0] = v.x; b[1] = v.y; b[2] = v.z; b[3] = v.w;
            } else {
#pragma unroll
                for (int j = 0; j < TJ; ++j) b[j] = Bs[k * LB + tx * TJ + j];
            }
#pragma unroll
            for (int i = 0; i < TI; ++i)
#pragma unroll
                for (int j = 0; j < TJ; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
    float* o = out + blockIdx.z * part_stride + z * zstride + J.out_off[jb];
#pragma unroll
    for (int i = 0; i < TI; ++i) {
        const int gi = i0 + ty * 4 + (i / 4) * (BI / TI * 4) + (i & 3);
        if (gi >= Mi) continue;
#pragma unroll
        for (int j = 0; j < TJ; ++j) {
            const int gj = j0 + tx * TJ + j;
            if (gj < Nj) o[(long long)gi * Nj + gj] = acc[i][j];
        }
    }
}

// out[i] = sum_s part[s][i] in slice order (n a multiple of 4).  The gradient blocks behind lambda[L] in the flat vector start
// on a 16-byte boundary only when L % 4 == 0: vector loads, scalar stores.
__global__ void __launch_bounds__(256) sum_slices_kernel(const float* __restrict__ part, int slices, long long n, float* __restrict__ out) {
    const long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) * 4;
    if (i >= n) return;
    float4 a = *reinterpret_cast<const float4*>(part + i);
    for (int s = 1; s < slices; ++s) {
        const float4 v = *reinterpret_cast<const float4*>(part + s * n + i);
        a.x += v.x; a.y += v.y; a.z += v.z; a.w += v.w;
    }
    out[i] = a.x; out[i + 1] = a.y; out[i + 2] = a.z; out[i + 3] = a.w;
}

// Slices of the reduction over M rows: enough CTAs for two per multiprocessor, none shorter than 64 rows.
inline int tn_slices(long long tiles, int M, int sms, int most) {
    long long s = (2LL * sms + tiles - 1) / tiles;
    s = s < most ? s : most;
    s = s < M / 64 ? s : M / 64;
    return (int)(s < 1 ? 1 : s);
}

}  // namespace pac
