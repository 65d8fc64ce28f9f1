// Products at fp32 precision on tcgen05, operands converted on the way into shared memory.
//
//   rows   out[z][m][j] = sum_k A(z; m, k) B[z][k][j]        (u_l = h_l W_down^l)
//   tn     out[i][j]    = sum_m A(z; m, i) B[z][m][j]        (dW = A^T B over all token rows)
//
// An fp32 operand enters as the exact sum of three bf16 terms (8 + 8 + 8 mantissa bits; exact for magnitudes from about 2^-110, where the third
// term starts to underflow, to the largest bf16, and see xg_redo for what lies beyond), a bf16 one as it is.  Of the products of terms those
// of relative size 2^-16 and above are formed, six or three; the dropped ones, below 2^-25, are smaller than the rounding of one fp32
// multiplication.  Sums are fp32, in several accumulators (xg_accs).  That is 1365 products per clock and SM against 128 on the FP32 pipe, so the kernel is bound
// by bringing the operands in: A comes straight from the activation cache (the gather is the address; any row length and alignment),
// producer warps fetch it into registers, split it and store the swizzled tiles, one warp issues the MMAs.  Two teams of eight producers take turns, each with
// a stage of its own, so that a team's loads are in flight while the other converts: in one CTA, or in two CTAs of one team each on an SM, whose starts
// and ends then fall under each other's stages (2048 x 768 x 64 x 12 layers, u 38 -> 35 us, on a bf16 cache 34 -> 27; which form a launch takes: xg_rows_plan, xg_slices).
// At 2048 rows, 12 layers, d = 768, r = 64: u 35 us, dW_down 29 us (the FP32-pipe tiles before it, 8 x 4 outputs per thread: 77 and 84 us).
// Loads are what it waits for (a third of the issue slots are used); row addresses are therefore formed once per stage (tn) or once per kernel
// (rows).  Prefetching the stage after next into L2 made the step 8 % slower.
// Every output is summed in a fixed order.
#pragma once
#include "pac_common.cuh"
#include "pac_tensor.cuh"

namespace pac {

// Row m of the minibatch at layer z, straight from the cache.
template <typename T>
struct XgCacheRows {
    typedef T elem;
    static constexpr bool cache_rows = true;
    const T* cache; const int* ids; long long N; int L, S, d;
    bool vec;                                   // rows start on 16-byte boundaries
    __device__ void take_ids(const int* v) { ids = v; }
    __device__ const T* row(int z, int m) const {
        const int b = m / S, s = m - b * S;
        return cache + ((safe_id(ids, b, N, nullptr) * L + z) * S + s) * (long long)d;
    }
};
// Row m of a row-major fp32 stack.
struct XgRows {
    typedef float elem;
    static constexpr bool cache_rows = false;
    const float* base; long long zstride; int ld;
    bool vec;                                   // rows start on 16-byte boundaries
    __device__ void take_ids(const int*) {}
    __device__ const float* row(int z, int m) const { return base + z * zstride + (long long)m * ld; }
};

constexpr int XG_TEAM = 8, XG_TILE = 128, XG_K = 64, XG_MAX_JOBS = 6;
__host__ __device__ constexpr int xg_threads(int teams) { return 32 * (teams * XG_TEAM + 1); }
static_assert(ARG_IDS <= xg_threads(1), "the first block stores the ids, one per thread");
constexpr uint32_t XG_TERM_A = XG_TILE * XG_K * 2, XG_BOX = 64 * 128;

// Products of one launch: several per layer (tn), all layers.
template <class AL>
struct XgJobs {
    AL A[XG_MAX_JOBS];
    XgRows B[XG_MAX_JOBS];
    int mi[XG_MAX_JOBS], nj[XG_MAX_JOBS];       // output extent
    int tiles_j[XG_MAX_JOBS], first[XG_MAX_JOBS + 1];
    long long out_off[XG_MAX_JOBS];
    int n = 0;
    int tile_j = 16;                            // columns per tile, a multiple of 16 up to 128
    int trans = 0;                              // 1: out[j][i]
    void add(const AL& a, int mi_, const XgRows& b, int nj_, long long off) {
        A[n] = a; B[n] = b; mi[n] = mi_; nj[n] = nj_; out_off[n] = off;
        tiles_j[n] = (nj_ + tile_j - 1) / tile_j;
        if (n == 0) first[0] = 0;
        first[n + 1] = first[n] + tiles_j[n] * ((mi_ + XG_TILE - 1) / XG_TILE);
        ++n;
    }
};

// Eight consecutive columns of a row, zeros from n on.
struct XgF8 { float v[8]; };
__device__ __forceinline__ void xg_load(const float* __restrict__ row, int c, int n, bool vec, XgF8& o) {
    if (vec && c + 8 <= n) {
        const float4 a = __ldg(reinterpret_cast<const float4*>(row + c)), b = __ldg(reinterpret_cast<const float4*>(row + c) + 1);
        o.v[0] = a.x; o.v[1] = a.y; o.v[2] = a.z; o.v[3] = a.w; o.v[4] = b.x; o.v[5] = b.y; o.v[6] = b.z; o.v[7] = b.w;
    } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) o.v[e] = c + e < n ? __ldg(row + c + e) : 0.f;
    }
}
__device__ __forceinline__ void xg_load(const bf16* __restrict__ row, int c, int n, bool vec, uint4& o) {
    if (vec && c + 8 <= n) {
        o = __ldg(reinterpret_cast<const uint4*>(row + c));
    } else {
        uint32_t w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const uint32_t lo = c + 2 * e < n ? __ldg(reinterpret_cast<const unsigned short*>(row) + c + 2 * e) : 0;
            const uint32_t hi = c + 2 * e + 1 < n ? __ldg(reinterpret_cast<const unsigned short*>(row) + c + 2 * e + 1) : 0;
            w[e] = lo | (hi << 16);
        }
        o = make_uint4(w[0], w[1], w[2], w[3]);
    }
}
__device__ __forceinline__ void xg_st(uint32_t a, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}
__device__ __forceinline__ void xg_store(uint32_t a, uint32_t term, const uint4& v) { xg_st(a, v.x, v.y, v.z, v.w); (void)term; }
__device__ __forceinline__ void xg_store(uint32_t a, uint32_t term, const XgF8& x) {
    uint32_t h[4], m[4], l[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) split3_pair(x.v[2 * e], x.v[2 * e + 1], h[e], m[e], l[e]);
    xg_st(a, h[0], h[1], h[2], h[3]);
    xg_st(a + term, m[0], m[1], m[2], m[3]);
    xg_st(a + 2 * term, l[0], l[1], l[2], l[3]);
}
template <typename T> struct XgTerms { static constexpr int n = 3; typedef XgF8 reg; };
template <> struct XgTerms<bf16> { static constexpr int n = 1; typedef uint4 reg; };

// Accumulators of a tile.  The tensor core cuts every partial sum to the accumulator's 24 bits instead of rounding it, an error that grows with the
// number of additions and not with its root.  The products of first terms therefore take turns, 16 of the reduction at a time, in accumulators of at most 24
// additions where tensor memory has the columns, and all smaller products have one of their own.  (One for all: against 64 bits u and dW_down were off by
// 3e-6 to 6e-6 at d = 768 and 1024 to 2048 rows; so by 2e-7 to 3e-7, the FP32 pipe by 6e-7.)
constexpr int XG_ACC_STEPS = 24;
inline int xg_accs(int tile_j, int k_steps) {      // beside that of the smaller products
    const int want = (k_steps + XG_ACC_STEPS - 1) / XG_ACC_STEPS, room = 512 / tile_j - 1;
    return want < 1 ? 1 : want < room ? want : room;
}
__host__ __device__ inline uint32_t xg_term_b(int tile_j) { return (uint32_t)((tile_j + 63) / 64) * XG_BOX; }
template <class AL>
inline size_t xg_smem(int tile_j, int teams) { return teams * ((size_t)XgTerms<typename AL::elem>::n * XG_TERM_A + 3 * xg_term_b(tile_j)) + 1024; }

// Outputs (i, j0 + c) for a warp's columns c of a tile, recomputed in fp32 where the sum of split products is not finite: an infinite operand,
// or a finite one beyond the largest bf16, has a first term of infinity and no second one, and a partial sum may overflow on the way.
// dst: the thread's row of sums, `step` apart.
template <bool TN, class AL>
__device__ __noinline__ void xg_redo(AL A, XgRows B, int z, int i, int j0, int c0, int c_step, int nj_tile, int Nj, int kb, int ke, float* dst, long long step) {
#pragma unroll 1
    for (; c0 < nj_tile; c0 += c_step)
#pragma unroll 1
        for (int c = c0; c < c0 + 16 && j0 + c < Nj; ++c) {
            if (fabsf(dst[c * step]) <= 3.402823466e38f) continue;
            float acc = 0.f;
#pragma unroll 4
            for (int k = kb; k < ke; ++k) {
                acc = fmaf(TN ? to_f32(A.row(z, k)[i]) : to_f32(A.row(z, i)[k]), B.row(z, k)[j0 + c], acc);
                if (acc != acc) break;
            }
            dst[c * step] = acc;
        }
}

// The tiles of an incomplete last wave (rows): `whole` tiles are computed by one CTA each, every later one by `parts` CTAs that take k_slice
// of the reduction each, leave their sums in ws and are added up, in order, by the one that finishes last (counted in cnt, which it puts back
// to zero).  At 192 tiles of 12 stages on 148 SMs
// the fp32 step went from 93.8 to 92.0 us (a CTA's start and end, not its stages, are the larger part of what the last wave costs).
struct XgTail { int whole, parts; float* ws; unsigned* cnt; };
// tn: grid (tiles of all jobs, layers, slices of the reduction); rows: (whole + parts * the other tiles).
// tn with more than one slice: the partial sums of slice s go to
// out + s * part_stride and are added up in slice order by whoever reads them.  GB: 8-column groups of B per thread (tile_j = 32 GB at most).
template <bool TN, int GB, int TEAMS, class AL>
__global__ void __launch_bounds__(xg_threads(TEAMS), TEAMS == 1 ? 2 : 1)
xgemm_kernel(const __grid_constant__ XgJobs<AL> J, int K, int k_slice, int accs_most, float* __restrict__ out, long long zstride, long long part_stride, XgTail tail, unsigned* status,
             const __grid_constant__ ArgIds arg, int* __restrict__ ids_out) {
    typedef typename AL::elem T;
    constexpr int TA = XgTerms<T>::n, PRODUCERS = TEAMS * XG_TEAM, THREADS = xg_threads(TEAMS);
    extern __shared__ unsigned char smem_raw[];
    const uint32_t ring = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const int nj_tile = J.tile_j;
    const uint32_t term_b = xg_term_b(nj_tile), stage = TA * XG_TERM_A + 3 * term_b;
    __shared__ __align__(8) unsigned long long bars[5];
    __shared__ uint32_t tmem_base_sh;
    __shared__ int abort_sh;
    const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[2]), accf = smem_u32(&bars[4]);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int z = blockIdx.y, at = blockIdx.x, split = TN ? (int)blockIdx.z : 0, shared_tile = -1;
    if (!TN) {
        if (at >= tail.whole) {
            const int q = at - tail.whole;
            shared_tile = q / tail.parts;
            split = q - shared_tile * tail.parts;
            at = tail.whole + shared_tile;
        }
        const int tiles = J.first[J.n];
        z = at / tiles;
        at -= z * tiles;
    }
    int jb = 0;
    while (jb + 1 < J.n && at >= J.first[jb + 1]) ++jb;
    const int tile = at - J.first[jb];
    const int i0 = tile / J.tiles_j[jb] * XG_TILE, j0 = tile % J.tiles_j[jb] * nj_tile;
    const int Mi = J.mi[jb], Nj = J.nj[jb];
    const int kb = split * k_slice, ke = !TN && shared_tile < 0 ? K : min(K, kb + k_slice), stages = ke > kb ? (ke - kb + XG_K - 1) / XG_K : 0;
    if (threadIdx.x == 0) {
        abort_sh = 0;
        for (int s = 0; s < TEAMS; ++s) { mbar_init(full0 + 8 * s, XG_TEAM); mbar_init(empty0 + 8 * s, 1); }
        mbar_init(accf, 1);
        fence_mbar_init();
    }
    const int accs = min(accs_most, max(1, stages * (XG_K / 16)));      // (a short last slice)
    uint32_t tmem_cols = 32;
    while (tmem_cols < (uint32_t)((accs + 1) * nj_tile)) tmem_cols *= 2;
    if (warp == PRODUCERS) { tmem_alloc(smem_u32(&tmem_base_sh), tmem_cols); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_sh;
    volatile int* abort_flag = &abort_sh;
    pdl_wait();
    pdl_trigger();      // (not before: a successor may rely on everything ahead of this kernel being complete when it starts)
    // the step's ids as an argument: this kernel reads them there and leaves a copy for the ones behind it
    if (!TN && blockIdx.x == 0 && (int)threadIdx.x < arg.n) ids_out[threadIdx.x] = arg.v[threadIdx.x];
    if (warp == PRODUCERS) {
        const uint32_t idesc = instr_desc_bf16(XG_TILE, nj_tile, TN ? 1 : 0, 1);
        // (term of A, term of B), the product of the first terms last
        constexpr int NP = TA == 3 ? 6 : 3;
        constexpr int pa[6] = {1, 0, 2, 0, 1, 0}, pb[6] = {1, 2, 0, 1, 0, 0};
        bool ok = true;
        int turn = 0;                               // accumulator of the stage's first product of first terms
        for (int it = 0; it < stages && ok; ++it) {
            const uint32_t s = TEAMS == 1 ? 0u : it & 1u;
            if (!mbar_wait_uniform(full0 + 8 * s, (TEAMS == 1 ? it : it >> 1) & 1u, abort_flag, status)) { ok = false; break; }
            tc_fence_after();
            if (elect_one()) {
                const uint32_t a = ring + s * stage, b = a + TA * XG_TERM_A;
                const uint64_t ad = TN ? smem_desc_sw128(a, XG_BOX, 1024) : smem_desc_sw128(a, 16, 1024), bd = smem_desc_sw128(b, XG_BOX, 1024);
#pragma unroll 1
                for (int k = 0, at = turn; k < XG_K / 16; ++k) {       // (rolled: a CTA has few stages, its code is fetched from memory)
#pragma unroll
                    for (int p = 0; p < NP; ++p) {
                        const int ta = TA == 3 ? pa[p] : 0, tb = TA == 3 ? pb[p] : 2 - p;
                        const bool first = p == NP - 1;
                        umma_bf16(tmem_base + (uint32_t)((first ? 1 + at : 0) * nj_tile), ad + (uint64_t)((ta * XG_TERM_A) >> 4) + (uint64_t)(k * (TN ? 128 : 2)),
                                  bd + (uint64_t)((tb * term_b) >> 4) + (uint64_t)(k * 128), idesc, (first ? it * (XG_K / 16) + k >= accs : (it | k | p) != 0) ? 1u : 0u);
                    }
                    if (++at == accs) at = 0;
                }
                umma_commit(empty0 + 8 * s);
                if (it + 1 == stages) umma_commit(accf);
            }
            __syncwarp();
            for (turn += XG_K / 16; turn >= accs;) turn -= accs;
        }
    } else {
        const int team = TEAMS == 1 ? 0 : warp >> 3, t = threadIdx.x & 255;
        AL A = J.A[jb];
        if (!TN && arg.n > 0) A.take_ids(arg.v);
        const XgRows B = J.B[jb];
        typename XgTerms<T>::reg ra[4];
        XgF8 rb[GB];
        uint32_t offa[4], offb[GB];
        int cola[4], rowa = 0, rowb[GB], colb[GB];
        const T* pa[4];
        const float* pb[GB];
        const int nb8 = nj_tile >> 3;
        // tn: four threads share a row, so that the row's address is formed once per stage; odd rows take their column groups in another
        // order, which spreads a quarter-warp's stores over all banks.  rows: four fixed rows.
        if (TN) rowa = t >> 2;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int row = TN ? rowa : (t + 256 * i) >> 3, c8 = TN ? (t & 3) + 4 * (i ^ (row & 1)) : t & 7;
            cola[i] = c8 * 8;
            offa[i] = (uint32_t)(c8 >> 3) * XG_BOX + (uint32_t)row * 128u + (uint32_t)(((c8 & 7) ^ (row & 7)) << 4);
            if (!TN) pa[i] = i0 + row < Mi ? A.row(z, i0 + row) : nullptr;
        }
        const long long step_b = (long long)TEAMS * XG_K * B.ld;
#pragma unroll
        for (int i = 0; i < GB; ++i) {
            const int g = t + 256 * i;
            rowb[i] = g / nb8;
            const int c8 = g - rowb[i] * nb8;
            colb[i] = j0 + c8 * 8;
            offb[i] = (uint32_t)(c8 >> 3) * XG_BOX + (uint32_t)rowb[i] * 128u + (uint32_t)(((c8 & 7) ^ (rowb[i] & 7)) << 4);
            pb[i] = B.row(z, kb + team * XG_K + rowb[i]);
            if (rowb[i] >= XG_K) rowb[i] = -1;
        }
        // rows beyond the output or the slice are not read and enter as zeros
        auto fetch = [&](int k0) {
            if (TN) {
                const int m = k0 + rowa;
                const T* row = A.row(z, min(m, ke - 1));
#pragma unroll
                for (int i = 0; i < 4; ++i) xg_load(row, i0 + cola[i], m < ke ? Mi : 0, A.vec, ra[i]);
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i) xg_load(pa[i], k0 + cola[i], pa[i] ? ke : 0, A.vec, ra[i]);
            }
#pragma unroll
            for (int i = 0; i < GB; ++i)
                if (rowb[i] >= 0) {
                    xg_load(pb[i], colb[i], k0 + rowb[i] < ke ? Nj : 0, B.vec, rb[i]);
                    pb[i] += step_b;
                }
        };
        bool ok = true;
        if (team < stages) fetch(kb + team * XG_K);
        for (int it = team; it < stages; it += TEAMS) {
            if (!mbar_wait_uniform(empty0 + 8 * team, ((TEAMS == 1 ? it : it >> 1) & 1u) ^ 1u, abort_flag, status)) { ok = false; break; }
            const uint32_t a = ring + team * stage, b = a + TA * XG_TERM_A;
#pragma unroll
            for (int i = 0; i < 4; ++i) xg_store(a + offa[i], XG_TERM_A, ra[i]);
#pragma unroll
            for (int i = 0; i < GB; ++i)
                if (rowb[i] >= 0) xg_store(b + offb[i], term_b, rb[i]);
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(full0 + 8 * team);
            if (it + TEAMS < stages) fetch(kb + (it + TEAMS) * XG_K);
        }
        if (stages > 0) {
            ok = ok && mbar_wait_warp(accf, 0, abort_flag, status);
            tc_fence_after();
        }
        if (ok) {
            const int q = warp & 3, i = i0 + q * 32 + lane;
            float* o = out + split * part_stride + z * zstride + J.out_off[jb];
            float* ws = tail.ws + ((long long)(shared_tile * tail.parts + split) * XG_TILE + q * 32 + lane) * nj_tile;
            const bool vec = !J.trans && (Nj & 3) == 0 && ((uintptr_t)o & 15) == 0;
            float odd = 0.f;                             // not zero once an element is not finite
            for (int c0 = (warp >> 2) * 16; c0 < nj_tile; c0 += 32 * TEAMS) {
                float v[16] = {};
                if (stages > 0) {
                    const uint32_t at = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)c0;
                    float w[16];
                    tmem_ld16(at, v);                    // the smaller products
                    tmem_ld16(at + (uint32_t)(accs * nj_tile), w);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 16; ++e) v[e] += w[e];
#pragma unroll 1
                    for (int a = accs - 1; a > 0; --a) {
                        tmem_ld16(at + (uint32_t)(a * nj_tile), w);
                        tmem_ld_wait();
#pragma unroll
                        for (int e = 0; e < 16; ++e) v[e] += w[e];
                    }
                }
#pragma unroll
                for (int e = 0; e < 16; ++e) odd = fmaf(v[e], 0.f, odd);
                if (!TN && shared_tile >= 0) {
#pragma unroll
                    for (int e = 0; e < 16; e += 4) *reinterpret_cast<float4*>(ws + c0 + e) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
                    continue;
                }
                if (i >= Mi) continue;
#pragma unroll
                for (int e = 0; e < 16; e += 4) {
                    const int j = j0 + c0 + e;
                    if (vec && j < Nj) {
                        *reinterpret_cast<float4*>(o + (long long)i * Nj + j) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
                    } else {
#pragma unroll
                        for (int x = 0; x < 4; ++x)
                            if (j + x < Nj) o[J.trans ? (long long)(j + x) * Mi + i : (long long)i * Nj + j + x] = v[e + x];
                    }
                }
            }
            if (!(odd == 0.f) && i < Mi) {
                const bool part = !TN && shared_tile >= 0;
                xg_redo<TN>(A, B, z, i, j0, (warp >> 2) * 16, 32 * TEAMS, nj_tile, Nj, kb, ke, part ? ws : J.trans ? o + (long long)j0 * Mi + i : o + (long long)i * Nj + j0, J.trans ? Mi : 1);
            }
        }
    }
    if (!TN && shared_tile >= 0) {
        __shared__ int last;
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) {
            last = atomicAdd(tail.cnt + shared_tile, 1u) == (unsigned)(tail.parts - 1);
            if (last) tail.cnt[shared_tile] = 0u;
            __threadfence();
        }
        __syncthreads();
        if (last) {
            const float* ws = tail.ws + (long long)shared_tile * tail.parts * XG_TILE * nj_tile;
            float* o = out + z * zstride + J.out_off[jb];
            for (int e = threadIdx.x * 4; e < XG_TILE * nj_tile; e += THREADS * 4) {
                float4 a = __ldcg(reinterpret_cast<const float4*>(ws + e));
                for (int k = 1; k < tail.parts; ++k) {
                    const float4 b = __ldcg(reinterpret_cast<const float4*>(ws + (long long)k * XG_TILE * nj_tile + e));
                    a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
                }
                const int i = i0 + e / nj_tile, j = j0 + e % nj_tile;
                const float v[4] = {a.x, a.y, a.z, a.w};
                for (int x = 0; x < 4 && i < Mi; ++x)
                    if (j + x < Nj) o[(long long)i * Nj + j + x] = v[x];
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    drain_after_abort(abort_flag);
    if (warp == PRODUCERS) tmem_dealloc(tmem_base, tmem_cols);
}

// apart: not launched programmatically.  An SM keeps its split of L1 and shared memory until it drains, and between programmatic launches it does not: behind a head kernel of nearly all
// the shared memory a CTA of this kernel ran with 28 KB of L1 instead of 92 (37 -> 41 to 50 us each; 384 tiles of 16 stages at r = 64: evaluation 95.8 us, launched apart 83.1, step
// 202.9 -> 174.2; 480 tiles: 114.4 -> 92.3, 238 -> 197).  Where the head kernel leaves more of it the overlap is worth 1 to 3 us.
template <bool TN, int GB, int TEAMS, class AL>
inline cudaError_t xgemm_launch(const XgJobs<AL>& J, int K, dim3 grid, int k_slice, float* out, long long zstride, long long part_stride, const XgTail& tail, unsigned* status, cudaStream_t stream, const ArgIds& arg, int* ids_out, bool apart) {
    const auto kernel = xgemm_kernel<TN, GB, TEAMS, AL>;
    const size_t smem = xg_smem<AL>(J.tile_j, TEAMS);
    cudaError_t e = smem_opt_in((const void*)kernel, smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    pdl_launch_config(&cfg, attr, grid, dim3(xg_threads(TEAMS)), smem, stream);
    if (apart) cfg.numAttrs = 0;
    const int longest = !TN && tail.whole > 0 ? K : K < k_slice ? K : k_slice;      // a CTA's share of the reduction
    const int accs = xg_accs(J.tile_j, (longest + XG_K - 1) / XG_K * (XG_K / 16));
    return cudaLaunchKernelEx(&cfg, kernel, J, K, k_slice, accs, out, zstride, part_stride, tail, status, arg, ids_out);
}
// Whether the accumulators of two CTAs fit beside each other.
inline bool xg_one_team(int tile_j, int stages) { return (xg_accs(tile_j, stages * (XG_K / 16)) + 1) * tile_j <= 256; }
// Slices of a reduction over K rows and producer teams per CTA: whole waves of CTAs, each about 2 us plus 0.6 us per stage, or 1 us where it has one team and shares its SM (measured), and
// the slices' own traffic.  One team only over the rows of the cache (fp32 step at T5-Base widths 86.2 -> 84.4 us, smallest one 48.4 -> 47.6).  Where its CTAs fill most of the second slots
// their starts and ends fall under each other's stages, which the count does not know: it is then taken up to a quarter above two teams (d = 512, L = 12, 2048 rows, 48 tiles 66.3 us, two
// teams 68.4; d = 576, L = 7, 35 tiles: three steps 106.8, 108.9).  With fewer tiles the count decides (d = 256, L = 12, r = 64, 24 tiles: two teams 48.1 us, one 51.0 at 2048 rows,
// 45.5 / 49.5 at 1600, 40.2 / 41.8 at 1024); of a single stage only one team has work, and its CTA is the lighter one (smallest blocking fp32 step 42.3, two teams 43.8).  The weight products of transformer bodies, whose rows lie in L2, were slower with one team, and tiles beyond 64 columns not reliably faster
// (steps of r = 128 216 -> 200, r = 80 96 -> 105).
struct XgSlices { int n, teams; };
inline XgSlices xg_slices(long long tiles, int K, int sms, int most, int tile_j) {      // tile_j: of products over the rows of the cache, else 0
    const int stages = (K + XG_K - 1) / XG_K;
    int best[3] = {0, 1, 1};
    double best_cost[3] = {0, 1e30, 1e30};
    for (int teams = 2; teams >= 1; --teams)
        for (int s = 1; s <= most && s <= stages; ++s) {
            const int each = (stages + s - 1) / s, slots = teams == 1 ? 2 * sms : sms;
            if (teams == 1 && !(tile_j > 0 && tile_j <= 64 && xg_one_team(tile_j, each))) continue;
            const double waves = (double)((tiles * s + slots - 1) / slots);
            const double cost = waves * (2.0 + (teams == 2 ? 0.6 : each == 1 ? 0.5 : 1.0) * each) + 0.3 * (s - 1);
            if (cost < best_cost[teams]) { best_cost[teams] = cost; best[teams] = s; }
        }
    const bool one = best_cost[1] < best_cost[2] * (5 * tiles * best[1] >= 7LL * sms ? 1.25 : 1.0);
    return one ? XgSlices{best[1], 1} : XgSlices{best[2], 2};
}
template <class AL>
inline cudaError_t xgemm_launch_tn(const XgJobs<AL>& J, int K, int Z, const XgSlices& sl, float* out, long long zstride, long long part_stride, unsigned* status, cudaStream_t stream, bool apart) {
    const int k_slice = ((K + sl.n - 1) / sl.n + XG_K - 1) / XG_K * XG_K;
    const dim3 grid((unsigned)J.first[J.n], (unsigned)Z, (unsigned)sl.n);
    if constexpr (AL::cache_rows)
        if (sl.teams == 1) return xgemm_launch<true, 2, 1>(J, K, grid, k_slice, out, zstride, part_stride, XgTail{}, status, stream, ArgIds{}, nullptr, apart);
    return J.tile_j <= 64 ? xgemm_launch<true, 2, 2>(J, K, grid, k_slice, out, zstride, part_stride, XgTail{}, status, stream, ArgIds{}, nullptr, apart)
                          : xgemm_launch<true, 4, 2>(J, K, grid, k_slice, out, zstride, part_stride, XgTail{}, status, stream, ArgIds{}, nullptr, apart);
}
// How `total` tiles of `stages` stages over the rows of the cache are dealt out (f32: rows of three terms; odd_bf16: bf16 rows that start off a 16-byte boundary, which producers
// load value by value).  A CTA per team from one wave on, except where its stages outweigh what its starts and ends save: a team alone on an SM does not hide its
// loads, so in the first quarter of a second wave two teams to a tile, and the few tiles beyond the first wave shared by all SMs, are faster when reductions are long, and for
// rows loaded value by value from some length on always.  Evaluation at r = 64, one team / two (us), tiles x stages:
//   fp32    160 x 8  32.6 / 38.7   192 x 8  33.1 / 39.9   160 x 12 41.4 / 44.0   160 x 16 51.1 / 48.7   192 x 16 51.7 / 51.9 (24 layers 53.8 / 60.1)   256 x 16 53.3 / 56.0   480 x 16 96.9 / 103.3
//   fp32, r = 16, and off a boundary at r = 64:   160 x 16 45.4 / 40.3, 66.0 / 57.8   192 x 16 45.7 / 43.9, 66.9 / 62.8   256 x 16 47.8 / 49.9, 68.5 / 72.6
//   bf16    160 x 16 37.6 / 43.6   256 x 16 41.4 / 48.8   320 x 16 61.3 / 64.6
//   bf16 off a boundary   160 x 4 27.1 / 31.6   160 x 9 46.9 / 41.7   256 x 9 48.2 / 48.2   160 x 13 68.1 / 51.3   384 x 13 107 / 92   384 x 16 123 / 110
// A tile of the last wave is shared when that takes four or more stages off its CTA (the exchange costs about as much as three).
struct XgRowsPlan { int teams, whole, parts, per; };      // per: stages of a part
inline XgRowsPlan xg_rows_plan(int total, int stages, int tile_j, bool f32, bool odd_bf16, int sms) {
    const bool one = total > sms && xg_one_team(tile_j, stages) && !(odd_bf16 && stages >= 8) && !(f32 && stages > 12 && 4LL * total <= 5LL * sms);
    const int slots = one ? 2 * sms : sms, rest = total % slots;
    XgRowsPlan p{one ? 1 : 2, total, 1, stages};
    if (rest > 0) {
        const int per = (stages + slots / rest - 1) / (slots / rest);
        if (stages - per >= 4) p = XgRowsPlan{p.teams, total - rest, (stages + per - 1) / per, per};
    }
    return p;
}
// ws: 2 sms tiles of 128 x tile_j floats, cnt: 2 sms words of zero.
template <class AL>
inline cudaError_t xgemm_launch_rows(const XgJobs<AL>& J, int K, int Z, int sms, float* out, long long zstride, float* ws, unsigned* cnt, unsigned* status, cudaStream_t stream, const ArgIds& arg, int* ids_out, bool apart) {
    const int total = J.first[J.n] * Z, stages = (K + XG_K - 1) / XG_K;
    const bool f32 = XgTerms<typename AL::elem>::n == 3;
    const XgRowsPlan p = xg_rows_plan(total, stages, J.tile_j, f32, !f32 && !J.A[0].vec, sms);
    const XgTail tail{p.whole, p.parts, ws, cnt};
    const dim3 grid((unsigned)(p.whole + (total - p.whole) * p.parts));
    const int k_slice = p.per * XG_K;
    if (J.tile_j <= 64)
        return p.teams == 1 ? xgemm_launch<false, 2, 1>(J, K, grid, k_slice, out, zstride, 0, tail, status, stream, arg, ids_out, apart) : xgemm_launch<false, 2, 2>(J, K, grid, k_slice, out, zstride, 0, tail, status, stream, arg, ids_out, apart);
    return p.teams == 1 ? xgemm_launch<false, 4, 1>(J, K, grid, k_slice, out, zstride, 0, tail, status, stream, arg, ids_out, apart) : xgemm_launch<false, 4, 2>(J, K, grid, k_slice, out, zstride, 0, tail, status, stream, arg, ids_out, apart);
}

// Columns per tile for an output N wide, tiles of equal width.
inline int xg_tile_j(int N) {
    const int tiles = (N + 127) / 128;
    return ((N + tiles - 1) / tiles + 15) / 16 * 16;
}

}  // namespace pac
