// Transformer-body adapters (Section IV-A), one launch per layer boundary and direction.
//
// The tokens of a sample meet only in the attention, so a layer is cut there: launch i of the forward pass
// runs attention, Wo, LayerNorm 2 and the feed-forward half of layer i - 1 and then merge, LayerNorm 1 and
// q, k, v of layer i; launch l of the backward pass runs dk, dv, LayerNorm 1 and the merge of layer l + 1 and
// then feed-forward, LayerNorm 2, do and dq of layer l.  A CTA owns 16 tokens of one sample from end to end;
// what it needs of the sample's other tokens (k, v; in reverse q, do, P, dS) was written by the launch before.
// The weight gradients A^T B over all rows follow in one launch for all layers (xgemm_kernel).
//
// Products at fp32 precision on the warp-level tensor instructions: 16 tokens are one m16 tile, far below the 128
// rows of a tcgen05 tile, and a CTA's products are short and serial.  Every fp32 operand is the exact sum of three bf16 terms
// (8 + 8 + 8 mantissa bits); of the nine products the six of relative size 2^-16 and above are formed, so the
// dropped ones (below 2^-25) are smaller than the rounding of one fp32 multiplication, and sums are fp32.
// Per SM that is 170 products per clock against 128 on the FP32 pipe, with a tenth of the instructions:
// the same kernels on FMA tiles (8 tokens x 4 columns per thread, weights through a shared-memory ring) took 60 us
// per forward launch instead of 30 at B = 16, S = 128, r = 64, waiting for instructions and shared memory, not for the pipe.
// Weights arrive from L2 in the order of the tile fragments (tb_pack_kernel: a warp reads 512 contiguous bytes per
// 16 x 8 tile) and are split in registers; activations are split once by whoever produces them.
#pragma once
#include "pac_tbody.cuh"
#include "pac_tensor.cuh"

namespace pac {

constexpr int TBF_THREADS = 512, TBF_WARPS = TBF_THREADS / 32, TBF_T = 16, TBF_MAX_R = 192;

// One packed weight matrix: K x N in 16 x 8 tiles, tile (ks, j) at (ks * nt + j) * 128 floats, zero-padded; lane l of a
// tile holds rows 2 (l % 4) + {0, 1, 8, 9} of column l / 4.
struct TbMat { const float* w; int ks, nt; };
__host__ __device__ inline int tb_up16(int x) { return (x + 15) & ~15; }
__host__ __device__ inline int tb_up8(int x) { return (x + 7) & ~7; }

// Offsets (floats) of the packed weights of one layer.
struct TbPack {
    int r, f;
    long long off[8], per_layer;       // Wo, W1, W2, Wqkv | Wqkv^T, W2^T, W1^T, Wo^T
    __host__ __device__ int rows(int m) const { return m == 2 || m == 6 ? f : m == 4 ? 3 * r : r; }                  // K
    __host__ __device__ int cols(int m) const { return m == 1 || m == 5 ? tb_up8(f) : m == 3 ? 3 * tb_up8(r) : tb_up8(r); }
    __host__ __device__ static TbPack make(int r, int f) {
        TbPack p;
        p.r = r; p.f = f;
        long long o = 0;
        for (int m = 0; m < 8; ++m) { p.off[m] = o; o += (long long)tb_up16(p.rows(m)) * p.cols(m); }
        p.per_layer = o;
        return p;
    }
    TbMat mat(const float* base, int m) const { return TbMat{base + off[m], tb_up16(rows(m)) / 16, cols(m) / 8}; }
};

// Lays the weights of every layer out in tile order: grid (blocks, L).
__global__ void __launch_bounds__(256) tb_pack_kernel(const float* __restrict__ body, long long body_per, BodyLayout bl,
                                                      const __grid_constant__ TbPack p, float* __restrict__ packed) {
    const float* w = body + blockIdx.y * body_per;
    float* dst = packed + blockIdx.y * p.per_layer;
    const int r = p.r, f = p.f, r8 = tb_up8(r);
    for (int e = (blockIdx.x * blockDim.x + threadIdx.x) * 4; e < (int)p.per_layer; e += gridDim.x * blockDim.x * 4) {
        int m = 0;
        while (m < 7 && e >= p.off[m + 1]) ++m;
        const int q = e - (int)p.off[m], lane = (q >> 2) & 31, tile = q >> 7, nt = p.cols(m) >> 3;
        const int k0 = (tile / nt) * 16 + 2 * (lane & 3), n = (tile % nt) * 8 + (lane >> 2), K = p.rows(m);
        float v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int k = k0 + (i & 1) + (i >> 1) * 8;
            v[i] = 0.f;
            if (k >= K) continue;
            if (m == 0) { if (n < r) v[i] = w[bl.wo + k * r + n]; }
            else if (m == 1) { if (n < f) v[i] = w[bl.w1 + k * f + n]; }
            else if (m == 2) { if (n < r) v[i] = w[bl.w2 + k * r + n]; }
            else if (m == 3) { const int s = n / r8, c = n - s * r8; if (c < r) v[i] = w[bl.wq + (s * r + k) * r + c]; }
            else if (m == 4) { const int s = k / r, j = k - s * r; if (n < r) v[i] = w[bl.wq + (s * r + n) * r + j]; }
            else if (m == 5) { if (n < f) v[i] = w[bl.w2 + n * r + k]; }
            else if (m == 6) { if (n < r) v[i] = w[bl.w1 + n * f + k]; }
            else if (n < r) v[i] = w[bl.wo + n * r + k];
        }
        *reinterpret_cast<float4*>(dst + e) = make_float4(v[0], v[1], v[2], v[3]);
    }
}

// Saved activations and reverse-pass stacks, all fp32, layer l at l * stride.
struct TbStacks {
    float *x, *xhat1, *n1, *qkv, *o, *xhat2, *n2, *hid, *P, *rstd1, *rstd2, *a;     // qkv: three [M][r] stacks per layer
    float *da, *dx1, *dqkv, *dpre;                                                 // reverse pass, operands of the weight gradients
    float *dob[2], *dS[2];                                                         // do and dS of the layer in flight and the one before
    float* part;                                                                   // [L][CTAs][part_w] column sums per CTA
    long long sMr, sMf, sP, sM;
    int part_w;                                                                    // g1 b1 g2 b2 c2 (r each) | c1 (f) | dlambda
};

struct TbLayerParams {
    TbMat mats[4];                     // of phases 0 .. 3 (see the kernels)
    int tail, head;                    // forward: layer whose attention + feed-forward half runs / layer whose q, k, v are formed (-1: none);
                                       // backward: layer whose dk, dv + merge run / layer whose feed-forward + dq run
    int B, S, r, f, H, hg;             // hg: heads whose score rows are in shared memory at a time
    int tiles;                         // CTAs per sample
    int train;
    int ka, kb, rs, ss;                // row strides in shared memory: wide and narrow operand terms (bf16), fp32 rows, score rows
    TbStacks s;
    const float* u; long long u_stride;
    float* du;                         // backward: [L][M][r], u_stride apart
    const float* lam;
    const float *g1, *b1, *g2, *b2, *c1, *c2;      // parameter vectors: forward g1, b1 of `head`, the rest of `tail`; backward g1 of `tail`, g2 of `head`
    const float* daL;                  // [B][r]
};

// ---------------------------------------------------------------------------
// Three-term operands
// ---------------------------------------------------------------------------
__device__ __forceinline__ void tb_mma(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
struct TbA { uint32_t h[4], m[4], l[4]; };     // 16 x 16 tile, three terms
struct TbB { uint32_t h[2], m[2], l[2]; };     // 16 x 8 tile
// c += A B, small products first.
__device__ __forceinline__ void tb_mma6(float (&c)[4], const TbA& a, const TbB& b) {
    tb_mma(c, a.m, b.m); tb_mma(c, a.h, b.l); tb_mma(c, a.l, b.h);
    tb_mma(c, a.h, b.m); tb_mma(c, a.m, b.h); tb_mma(c, a.h, b.h);
}
__device__ __forceinline__ void tb_split_b(TbB& b, float k0, float k1, float k8, float k9) {
    split3_pair(k0, k1, b.h[0], b.m[0], b.l[0]);
    split3_pair(k8, k9, b.h[1], b.m[1], b.l[1]);
}
// A tile from fp32 rows in shared memory: p points at (row lane / 4, column 2 (lane % 4)) of the tile.
__device__ __forceinline__ void tb_split_a(TbA& a, const float* p, int stride) {
    const float2 v0 = *reinterpret_cast<const float2*>(p), v1 = *reinterpret_cast<const float2*>(p + 8 * stride);
    const float2 v2 = *reinterpret_cast<const float2*>(p + 8), v3 = *reinterpret_cast<const float2*>(p + 8 * stride + 8);
    split3_pair(v0.x, v0.y, a.h[0], a.m[0], a.l[0]);
    split3_pair(v1.x, v1.y, a.h[1], a.m[1], a.l[1]);
    split3_pair(v2.x, v2.y, a.h[2], a.m[2], a.l[2]);
    split3_pair(v3.x, v3.y, a.h[3], a.m[3], a.l[3]);
}
__device__ __forceinline__ void tb_ldmatrix4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
// Operand terms in shared memory: [term][16 tokens][stride] bf16, stride = K rounded to 16, + 8 (eight rows of 16 bytes fall
// into different banks).
__device__ __forceinline__ void tb_put2(bf16* pl, int stride, int t, int c, float x, float y) {      // columns c, c + 1 (c even)
    uint32_t h, m, l;
    split3_pair(x, y, h, m, l);
    uint32_t* q = reinterpret_cast<uint32_t*>(pl + t * stride + c);
    q[0] = h; q[8 * stride] = m; q[16 * stride] = l;
}
__device__ __forceinline__ void tb_put1(bf16* pl, int stride, int t, int c, float x) {
    uint32_t h, m, l;
    split3_pair(x, 0.f, h, m, l);
    uint16_t* q = reinterpret_cast<uint16_t*>(pl + t * stride + c);
    q[0] = (uint16_t)h; q[16 * stride] = (uint16_t)m; q[32 * stride] = (uint16_t)l;
}

// ---------------------------------------------------------------------------
// Building blocks (a CTA of sixteen warps and 16 tokens)
// ---------------------------------------------------------------------------
// A matrix of up to eight tiles along N is cut in half along K between warps 0 - 7 and 8 - 15 (every other product has a tile for
// each warp): the k steps [from, to) of `half`.
__device__ __forceinline__ bool tb_cut(int nt) { return nt <= TBF_WARPS / 2; }
// A warp's own stream of weight tiles: phase after phase, pairs of tiles (columns 128 apart), k step by k step.
// Every lane copies and later reads its own 16 bytes of a tile, so the stream needs no barrier: it runs TBF_AHEAD tiles
// ahead of the products, across phases, and starts before the wait for the predecessor launch.
constexpr int TBF_SLOTS = 16, TBF_AHEAD = 12, TBF_BATCH = 4;
struct TbStream {
    const TbMat* mats;
    int ph, last;                      // phase being fetched, one past the last
    int j0, n, i, ks, to, nt;          // first tile of the pair, its tiles, tile, k step and its end; the matrix' tiles along N
    int from;
    const float *base, *src;           // lane's address of the matrix' first tile / of the next tile
    uint32_t ring;                     // lane's address of slot 0
    int put = 0, get = 0;
    __device__ TbStream(const TbMat* m, int first, int last_, unsigned char* mem) : mats(m), ph(first), last(last_) {
        ring = smem_u32(mem) + (threadIdx.x >> 5) * (TBF_SLOTS * 512) + (threadIdx.x & 31) * 16;
        open();
    }
    __device__ void aim() { n = j0 + TBF_WARPS < nt ? 2 : 1; ks = from; src = base + (long long)(from * nt + j0) * 128; i = 0; }
    __device__ void open() {           // first tile of phase `ph` (phases in which this warp has no tile are passed over)
        const int warp = threadIdx.x >> 5;
        for (; ph < last; ++ph) {
            nt = mats[ph].nt;
            const int n_ks = mats[ph].ks;
            const bool cut = tb_cut(nt), half = cut && warp >= TBF_WARPS / 2;
            from = half ? (n_ks + 1) / 2 : 0;
            to = cut && !half ? (n_ks + 1) / 2 : n_ks;
            base = mats[ph].w + (threadIdx.x & 31) * 4;
            j0 = half ? warp - TBF_WARPS / 2 : warp;
            if (j0 < nt && (!cut || j0 < TBF_WARPS / 2) && from < to) { aim(); return; }
        }
    }
    __device__ void issue() {
        if (ph < last) {
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(ring + put * 512), "l"(src) : "memory");
            put = (put + 1) & (TBF_SLOTS - 1);
            src += TBF_WARPS * 128;
            if (++i == n) {
                i = 0;
                src += (nt - n * TBF_WARPS) * 128;
                if (++ks == to) {
                    j0 += 2 * TBF_WARPS;
                    if (j0 < nt && !tb_cut(nt)) aim();
                    else { ++ph; open(); }
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    // The next `count` <= TBF_BATCH tiles, and as many sent for.
    __device__ void next(float4 (&v)[TBF_BATCH], int count) {
        asm volatile("cp.async.wait_group %0;" ::"n"(TBF_AHEAD - TBF_BATCH) : "memory");
#pragma unroll
        for (int e = 0; e < TBF_BATCH; ++e)
            if (e < count) {
                asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[e].x), "=f"(v[e].y), "=f"(v[e].z), "=f"(v[e].w)
                             : "r"(ring + ((get + e) & (TBF_SLOTS - 1)) * 512) : "memory");
            }
        get += count;
#pragma unroll 1
        for (int e = 0; e < count; ++e) issue();
    }
};

// acc += the k steps [from, to) of N tiles: batches of TBF_BATCH tiles are in registers before the first is split.
// Three accumulators per tile shorten the dependent chain of a k step to three.
template <int N>
__device__ __forceinline__ void tb_tiles(TbStream& st, int from, int to, uint32_t a0, uint32_t term, float (&v)[2][4]) {
    constexpr int KU = TBF_BATCH / N;
    float acc[N][3][4] = {};
#pragma unroll 1
    for (int ks = from; ks < to; ks += KU) {
        const int steps = min(KU, to - ks);
        float4 w[TBF_BATCH];
        st.next(w, steps * N);
#pragma unroll
        for (int k = 0; k < KU; ++k) {
            if (k < steps) {
                TbA a;
                const uint32_t ad = a0 + (ks + k) * 32;
                tb_ldmatrix4(a.h, ad); tb_ldmatrix4(a.m, ad + term); tb_ldmatrix4(a.l, ad + 2 * term);
#pragma unroll
                for (int i = 0; i < N; ++i) {
                    TbB b;
                    tb_split_b(b, w[k * N + i].x, w[k * N + i].y, w[k * N + i].z, w[k * N + i].w);
                    tb_mma(acc[i][0], a.m, b.m); tb_mma(acc[i][1 + (k & 1)], a.h, b.h); tb_mma(acc[i][0], a.h, b.l);
                    tb_mma(acc[i][0], a.l, b.h); tb_mma(acc[i][0], a.h, b.m); tb_mma(acc[i][0], a.m, b.h);
                }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) v[i][e] = (acc[i][2][e] + acc[i][1][e]) + acc[i][0][e];
}

// Partial results of warps 8 - 15 to warps 0 - 7, lane by lane (every thread of the CTA takes part).
__device__ __forceinline__ void tb_combine(float4* red, float (&v)[4]) {
    const int t = threadIdx.x, h = TBF_THREADS / 2;
    if (t >= h) red[t - h] = make_float4(v[0], v[1], v[2], v[3]);
    __syncthreads();
    if (t < h) { const float4 o = red[t]; v[0] += o.x; v[1] += o.y; v[2] += o.z; v[3] += o.w; }
}

// out = act W for the 16 tokens: act's terms at pl, W the stream's next matrix.  ep(n, v): columns n, n + 1 of rows lane / 4 (v[0], v[1])
// and lane / 4 + 8 (v[2], v[3]); called by whole warps.
template <class EP>
__device__ __forceinline__ void tb_product(TbStream& st, const TbMat& m, const bf16* pl, int stride, float4* red, EP ep) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t a0 = smem_u32(pl) + (((lane & 15) * stride) + (lane >> 4) * 8) * 2, term = 32 * stride;
    const int nt = m.nt, n_ks = m.ks;
    const bool cut = tb_cut(nt), half = cut && warp >= TBF_WARPS / 2;
    const int from = half ? (n_ks + 1) / 2 : 0, to = cut && !half ? (n_ks + 1) / 2 : n_ks;
    int j0 = half ? warp - TBF_WARPS / 2 : warp;
    do {
        const bool mine = j0 < nt, two = !cut && j0 + TBF_WARPS < nt;
        float v[2][4] = {};
        if (two) tb_tiles<2>(st, from, to, a0, term, v);
        else if (mine) tb_tiles<1>(st, from, to, a0, term, v);
        if (cut) tb_combine(red, v[0]);
        if (mine && !half) {
            ep(j0 * 8 + 2 * (lane & 3), v[0]);
            if (two) ep((j0 + TBF_WARPS) * 8 + 2 * (lane & 3), v[1]);
        }
        j0 += 2 * TBF_WARPS;
    } while (!cut && j0 < nt);
}

// Two consecutive floats of a row (zeros past n); `even`: the row starts on an 8-byte boundary.
__device__ __forceinline__ float2 tb_ld2(const float* __restrict__ p, int c, int n, bool even) {
    if (even && c + 1 < n) return __ldg(reinterpret_cast<const float2*>(p + c));
    return make_float2(c < n ? __ldg(p + c) : 0.f, c + 1 < n ? __ldg(p + c + 1) : 0.f);
}

// sc[(h * 16 + t) * ss + j] = sum_i act[t][(h0 + h) dh + i] X[j][(h0 + h) dh + i]: scores of the 16 tokens against all S tokens of
// the sample.  act: fp32 rows in shared memory, X: [S][r] in global memory.  A warp takes 32 keys of one head.
__device__ __forceinline__ void tb_scores(const float* __restrict__ X, int r, const float* act, int rs, int S, int dh, int h0, int hg, float* sc, int ss) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = lane >> 2, c2 = 2 * (lane & 3);
    const int chunks = (S + 31) >> 5;
    const bool even = ((dh | r) & 1) == 0;
    for (int w = warp; w < hg * chunks; w += TBF_WARPS) {
        const int h = w / chunks, n0 = (w - h * chunks) * 32, col = (h0 + h) * dh;
        float acc[4][4] = {};
        for (int k = 0; k < dh; k += 16) {
            // columns past the head's are zeros on the X side; what act holds there is finite
            TbA a;
            {
                float v[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int c = k + c2 + (i & 1) + (i >> 2) * 8;
                    v[i] = c < dh ? act[(q + ((i >> 1) & 1) * 8) * rs + col + c] : 0.f;
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) split3_pair(v[2 * i], v[2 * i + 1], a.h[i], a.m[i], a.l[i]);
            }
#pragma unroll
            for (int n = 0; n < 4; ++n) {
                if (n0 + n * 8 < S) {
                    const float* x = X + (long long)min(n0 + n * 8 + q, S - 1) * r + col + k;
                    const float2 v0 = tb_ld2(x, c2, dh - k, even), v1 = tb_ld2(x, c2 + 8, dh - k, even);
                    TbB b;
                    tb_split_b(b, v0.x, v0.y, v1.x, v1.y);
                    tb_mma6(acc[n], a, b);
                }
            }
        }
        float* o = sc + (h * 16 + q) * ss + n0 + c2;
#pragma unroll
        for (int n = 0; n < 4; ++n)
            if (n0 + n * 8 < S) {
                *reinterpret_cast<float2*>(o + n * 8) = make_float2(acc[n][0], acc[n][1]);
                *reinterpret_cast<float2*>(o + 8 * ss + n * 8) = make_float2(acc[n][2], acc[n][3]);
            }
    }
}

// ep(c, two, v) with v = rows (lane / 4, + 8) x columns (c, c + 1) of  sum_j sc[h][t][j] X[j][c],  c from h0 * dh to (h0 + hg) * dh: mixes the
// rows of all S tokens with the weights in shared memory (zero from S to the next multiple of 16).  c may be odd and c + 1 may lie
// past the head: `two` says whether it counts.  A warp takes eight columns of one head; up to eight such tasks: half of the rows each.
template <class EP>
__device__ __forceinline__ void tb_mix(const float* __restrict__ X, int r, const float* sc, int ss, int S, int dh, int h0, int hg, float4* red, EP ep) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = lane >> 2, c2 = 2 * (lane & 3);
    const int tiles = (dh + 7) >> 3, tasks = hg * tiles;
    const bool cut = tb_cut(tasks), half = cut && warp >= TBF_WARPS / 2;
    const int mid = ((S + 31) >> 5) * 16, from = half ? mid : 0, to = cut && !half ? min(mid, S) : S;
    int w = half ? warp - TBF_WARPS / 2 : warp;
    do {
        const bool mine = w < tasks;
        const int h = w / tiles, n0 = (w - h * tiles) * 8;
        float v[4] = {};
        if (mine) {
            const float* x = X + (h0 + h) * dh + min(n0 + q, dh - 1);
            const float* a_row = sc + (h * 16 + q) * ss + c2;
            float acc[2][4] = {};
#pragma unroll 4
            for (int k = from; k < to; k += 16) {
                const int j = k + c2;
                TbA a;
                TbB b;
                const float x0 = __ldg(x + (long long)min(j, S - 1) * r), x1 = __ldg(x + (long long)min(j + 1, S - 1) * r);
                const float x8 = __ldg(x + (long long)min(j + 8, S - 1) * r), x9 = __ldg(x + (long long)min(j + 9, S - 1) * r);
                tb_split_a(a, a_row + k, ss);
                tb_split_b(b, x0, x1, x8, x9);
                tb_mma(acc[0], a.m, b.m); tb_mma(acc[1], a.h, b.m); tb_mma(acc[0], a.h, b.l);
                tb_mma(acc[1], a.m, b.h); tb_mma(acc[0], a.l, b.h); tb_mma(acc[1], a.h, b.h);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] = acc[1][e] + acc[0][e];
        }
        if (cut) tb_combine(red, v);
        if (mine && !half && n0 + c2 < dh) ep((h0 + h) * dh + n0 + c2, n0 + c2 + 1 < dh, v);
        w += TBF_WARPS;
    } while (!cut && w < tasks);
}

// Sum over the 16 tokens of a column pair: v of tb_product's epilogue, the result in every lane of the column.
__device__ __forceinline__ float tb_col_sum(float top, float bottom) {
    float s = top + bottom;
    s += __shfl_xor_sync(0xffffffffu, s, 4);
    s += __shfl_xor_sync(0xffffffffu, s, 8);
    s += __shfl_xor_sync(0xffffffffu, s, 16);
    return s;
}

// Shared memory: tile ring | halves of sums | operand terms wide, narrow | fp32 rows xb, qf | score rows.
struct TbSmem { unsigned char* ring; float4* red; bf16 *wide, *narrow; float *xb, *qf, *sc; };
constexpr size_t TBF_FIXED = TBF_SLOTS * TBF_WARPS * 512 + TBF_THREADS / 2 * 16;
__host__ __device__ inline size_t tb_smem_terms(int stride) { return (size_t)3 * TBF_T * stride * 2; }
__device__ __forceinline__ TbSmem tb_carve(unsigned char* base, const TbLayerParams& p) {
    TbSmem s;
    s.ring = base;
    s.red = reinterpret_cast<float4*>(base + TBF_SLOTS * TBF_WARPS * 512);
    s.wide = reinterpret_cast<bf16*>(base + TBF_FIXED);
    s.narrow = s.wide + 3 * TBF_T * p.ka;
    s.xb = reinterpret_cast<float*>(s.narrow + 3 * TBF_T * p.kb);
    s.qf = s.xb + TBF_T * p.rs;
    s.sc = s.qf + TBF_T * p.rs;
    // the padding of the terms is multiplied with zero weights: it has to be finite
    uint32_t* z = reinterpret_cast<uint32_t*>(s.wide);
    for (int i = threadIdx.x; i < 3 * TBF_T * (p.ka + p.kb) / 2; i += TBF_THREADS) z[i] = 0u;
    return s;
}

// Phases: 0 x1 = x + o Wo, 1 hid = relu(LN2(x1) W1 + c1), 2 a = x1 + hid W2 + c2 (of `tail`), 3 q, k, v = LN1(x) [Wq Wk Wv] (of `head`).
// They run through ONE copy of the code: a phase is executed once per launch, so instructions it does not share are fetched
// from memory.
__global__ void __launch_bounds__(TBF_THREADS) tb_fwd_kernel(const __grid_constant__ TbLayerParams p) {
    extern __shared__ __align__(128) unsigned char tb_sm[];
    const int b = blockIdx.x / p.tiles, t0 = (blockIdx.x - b * p.tiles) * TBF_T;
    const int S = p.S, r = p.r, f = p.f, H = p.H, dh = r / H, nt = min(TBF_T, S - t0), rs = p.rs, ss = p.ss;
    const long long m0 = (long long)b * S + t0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, q = lane >> 2;
    const int first = p.tail >= 0 ? 0 : 3, last = p.head >= 0 ? 4 : 3;
    TbStream st(p.mats, first, last, tb_sm);
    for (int i = 0; i < TBF_AHEAD; ++i) st.issue();             // the packed weights were final before the predecessor started
    const TbSmem sm = tb_carve(tb_sm, p);
    pdl_wait();
    pdl_trigger();
    __syncthreads();
    const TbStacks& s = p.s;
    const bool even = (r & 1) == 0;
    const bool live0 = q < nt, live1 = q + 8 < nt;
    if (p.tail >= 0) {
        const int l = p.tail;
        const float* qkv = s.qkv + 3 * l * s.sMr;
        for (int c = lane; c < r; c += 32) sm.qf[warp * rs + c] = warp < nt ? __ldg(qkv + (m0 + warp) * r + c) : 0.f;
        __syncthreads();
        const float scale = 1.f / sqrtf((float)dh);
        const int S16 = tb_up16(S);
#pragma unroll 1
        for (int h0 = 0; h0 < H; h0 += p.hg) {
            const int hg = min(p.hg, H - h0);
            tb_scores(qkv + s.sMr + (long long)b * S * r, r, sm.qf, rs, S, dh, h0, hg, sm.sc, ss);
            __syncthreads();
            // softmax over the keys: a warp takes four rows at a time, so that four dependent chains overlap
            for (int w = warp * 4; w < hg * TBF_T; w += TBF_WARPS * 4) {
                float* row = sm.sc + w * ss;
                const int t = w & (TBF_T - 1), h = h0 + (w >> 4);
                float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY}, se[4] = {};
#pragma unroll 2
                for (int j = lane; j < S; j += 32)
#pragma unroll
                    for (int i = 0; i < 4; ++i) mx[i] = fmaxf(mx[i], row[i * ss + j] * scale);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                    for (int i = 0; i < 4; ++i) mx[i] = fmaxf(mx[i], __shfl_xor_sync(0xffffffffu, mx[i], o));
#pragma unroll 2
                for (int j = lane; j < S; j += 32)
#pragma unroll
                    for (int i = 0; i < 4; ++i) { const float e = expf(row[i * ss + j] * scale - mx[i]); row[i * ss + j] = e; se[i] += e; }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                    for (int i = 0; i < 4; ++i) se[i] += __shfl_xor_sync(0xffffffffu, se[i], o);
                float* P = s.P + l * s.sP + (((long long)b * H + h) * S + t0 + t) * S;
#pragma unroll 2
                for (int j = lane; j < S16; j += 32)
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float e = j < S ? row[i * ss + j] / se[i] : 0.f;
                        row[i * ss + j] = e;
                        if (p.train && t + i < nt && j < S) P[i * S + j] = e;
                    }
            }
            __syncthreads();
            tb_mix(qkv + 2 * s.sMr + (long long)b * S * r, r, sm.sc, ss, S, dh, h0, hg, sm.red, [&](int c, bool two, const float (&v)[4]) {
                tb_put1(sm.narrow, p.kb, q, c, v[0]); tb_put1(sm.narrow, p.kb, q + 8, c, v[2]);
                if (two) { tb_put1(sm.narrow, p.kb, q, c + 1, v[1]); tb_put1(sm.narrow, p.kb, q + 8, c + 1, v[3]); }
                if (p.train) {
                    float* o = s.o + l * s.sMr + (m0 + q) * r + c;
                    if (live0) { o[0] = v[0]; if (two) o[1] = v[1]; }
                    if (live1) { o[8LL * r] = v[2]; if (two) o[8LL * r + 1] = v[3]; }
                }
            });
            __syncthreads();
        }
    }
#pragma unroll 1
    for (int ph = first; ph < last; ++ph) {
        if (ph & 1) {
            // LayerNorm 2 of `tail`, or merge and LayerNorm 1 of `head`; a row per warp, lanes over the columns
            const bool one = ph == 3;
            const int l = one ? p.head : p.tail;
            const long long o = l * s.sMr + m0 * r;
            const float *g = one ? p.g1 : p.g2, *be = one ? p.b1 : p.b2;
            float *xh_out = (one ? s.xhat1 : s.xhat2) + o, *n_out = (one ? s.n1 : s.n2) + o, *x_out = s.x + o;
            const float* u = p.u + l * p.u_stride + m0 * r;
            const float lm = one ? __ldg(p.lam + l) : 0.f;
            for (int t = warp; t < TBF_T; t += TBF_WARPS) {
                float v[TBF_MAX_R / 32], sum = 0.f, var = 0.f;
#pragma unroll
                for (int i = 0; i < TBF_MAX_R / 32; ++i) {
                    const int c = lane + 32 * i;
                    v[i] = 0.f;
                    if (c < r) {
                        v[i] = one && p.tail < 0 ? 0.f : sm.xb[t * rs + c];
                        if (one) {
                            v[i] = lm * (t < nt ? __ldg(u + t * r + c) : 0.f) + (1.f - lm) * v[i];
                            if (t < nt) x_out[t * r + c] = v[i];
                        }
                        sum += v[i];
                    }
                }
                const float mu = warp_sum(sum) / (float)r;
#pragma unroll
                for (int i = 0; i < TBF_MAX_R / 32; ++i)
                    if (lane + 32 * i < r) { const float d = v[i] - mu; var = fmaf(d, d, var); }
                const float rstd = 1.f / sqrtf(warp_sum(var) / (float)r + TB_LN_EPS);
#pragma unroll
                for (int i = 0; i < TBF_MAX_R / 32; ++i) {
                    const int c = lane + 32 * i;
                    if (c < r) {
                        const float xh = (v[i] - mu) * rstd, n = xh * __ldg(g + c) + __ldg(be + c);
                        tb_put1(sm.narrow, p.kb, t, c, n);
                        if (p.train && t < nt) { xh_out[t * r + c] = xh; n_out[t * r + c] = n; }
                    }
                }
                if (lane == 0 && t < nt) (one ? s.rstd1 : s.rstd2)[l * s.sM + m0 + t] = rstd;
            }
            __syncthreads();
        }
        const bool wide_in = ph == 2;
        const long long o_tail = p.tail * s.sMr + m0 * r, o_hid = p.tail * s.sMf + m0 * f, o_a = p.tail * p.u_stride + m0 * r;
        const int r8 = tb_up8(r);
        tb_product(st, p.mats[ph], wide_in ? sm.wide : sm.narrow, wide_in ? p.ka : p.kb, sm.red, [&](int n, const float (&v)[4]) {
            if (ph == 1) {
                const float2 c = tb_ld2(p.c1, n, f, false);
                float h[4] = {fmaxf(v[0] + c.x, 0.f), fmaxf(v[1] + c.y, 0.f), fmaxf(v[2] + c.x, 0.f), fmaxf(v[3] + c.y, 0.f)};
                if (n + 1 >= f) { h[1] = 0.f; h[3] = 0.f; }
                if (n < f) {
                    tb_put2(sm.wide, p.ka, q, n, h[0], h[1]); tb_put2(sm.wide, p.ka, q + 8, n, h[2], h[3]);
                    if (p.train) {
                        float* out = s.hid + o_hid + (long long)q * f + n;
                        if (live0) { out[0] = h[0]; if (n + 1 < f) out[1] = h[1]; }
                        if (live1) { out[8LL * f] = h[2]; if (n + 1 < f) out[8LL * f + 1] = h[3]; }
                    }
                }
            } else if (ph < 3) {
                if (n < r) {
                    const bool two = n + 1 < r;
                    float* x = sm.xb + q * rs + n;
                    const float2 z = make_float2(0.f, 0.f);
                    float2 a0, a1;
                    if (ph == 0) {
                        const float* xg = s.x + o_tail + (long long)q * r;
                        a0 = live0 ? tb_ld2(xg, n, r, even) : z; a1 = live1 ? tb_ld2(xg + 8LL * r, n, r, even) : z;
                    } else {
                        const float2 c = tb_ld2(p.c2, n, r, false);
                        a0 = make_float2(x[0] + c.x, x[1] + c.y); a1 = make_float2(x[8 * rs] + c.x, x[8 * rs + 1] + c.y);
                    }
                    const float y0 = v[0] + a0.x, y1 = v[1] + a0.y, y2 = v[2] + a1.x, y3 = v[3] + a1.y;
                    *reinterpret_cast<float2*>(x) = make_float2(y0, y1);
                    *reinterpret_cast<float2*>(x + 8 * rs) = make_float2(y2, y3);
                    if (ph == 2) {
                        float* out = s.a + o_a + (long long)q * r + n;
                        if (live0) { out[0] = y0; if (two) out[1] = y1; }
                        if (live1) { out[8LL * r] = y2; if (two) out[8LL * r + 1] = y3; }
                    }
                }
            } else {
                const int k = n / r8, c = n - k * r8;
                if (c < r) {
                    float* out = s.qkv + (3 * p.head + k) * s.sMr + (m0 + q) * r + c;
                    if (live0) { out[0] = v[0]; if (c + 1 < r) out[1] = v[1]; }
                    if (live1) { out[8LL * r] = v[2]; if (c + 1 < r) out[8LL * r + 1] = v[3]; }
                }
            }
        });
        __syncthreads();
    }
}

// Phases: 0 dn1 = [dq | dk | dv] [Wq | Wk | Wv]^T (of `tail`); 1 dhid = da W2^T, 2 dn2 = dpre W1^T, 3 do = dx1 Wo^T (of `head`).
__global__ void __launch_bounds__(TBF_THREADS) tb_bwd_kernel(const __grid_constant__ TbLayerParams p) {
    extern __shared__ __align__(128) unsigned char tb_sm[];
    __shared__ float lam_red[32];
    const int b = blockIdx.x / p.tiles, t0 = (blockIdx.x - b * p.tiles) * TBF_T;
    const int S = p.S, r = p.r, f = p.f, H = p.H, dh = r / H, nt = min(TBF_T, S - t0), rs = p.rs, ss = p.ss, S16 = tb_up16(S);
    const long long m0 = (long long)b * S + t0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, q = lane >> 2;
    const float scale = 1.f / sqrtf((float)dh);
    const int first = p.tail >= 0 ? 0 : 1, last = p.head >= 0 ? 4 : 1;
    TbStream st(p.mats, first, last, tb_sm);
    for (int i = 0; i < TBF_AHEAD; ++i) st.issue();
    const TbSmem sm = tb_carve(tb_sm, p);
    pdl_wait();
    pdl_trigger();
    __syncthreads();
    const TbStacks& s = p.s;
    const bool even = (r & 1) == 0, live0 = q < nt, live1 = q + 8 < nt;
    if (p.tail >= 0) {
        const int l = p.tail;
        float* dqkv = s.dqkv + 3 * l * s.sMr + m0 * r;
        const bool vec = (S & 3) == 0;
        // dk[t] = scale sum_s dS[s][t] q[s],  dv[t] = sum_s P[s][t] do[s]   (own tokens t, all tokens s)
#pragma unroll 1
        for (int hk = 0, hg; hk < 2 * H; hk += hg) {
            const int k = hk >= H, h0 = k ? hk - H : hk;
            hg = min(p.hg, H - h0);
            const float* src = (k ? s.P + l * s.sP : s.dS[l & 1]) + ((long long)b * H + h0) * S * S + t0;
            // columns t0 .. t0 + 15 of the S x S matrices, transposed into score rows: a thread moves four tokens of one row
            for (int e = threadIdx.x; e < hg * 4 * S16; e += TBF_THREADS) {
                const int hq = e / S16, j = e - hq * S16, t = (hq & 3) * 4;
                float v[4] = {0.f, 0.f, 0.f, 0.f};
                if (j < S) {
                    const float* g = src + ((long long)(hq >> 2) * S + j) * S + t;
                    if (vec && t < nt) { const float4 x = __ldg(reinterpret_cast<const float4*>(g)); v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w; }
                    else
#pragma unroll
                        for (int i = 0; i < 4; ++i) if (t + i < nt) v[i] = __ldg(g + i);
                }
                float* o = sm.sc + ((hq >> 2) * TBF_T + t) * ss + j;
#pragma unroll
                for (int i = 0; i < 4; ++i) o[i * ss] = v[i];
            }
            __syncthreads();
            const float* X = (k ? s.dob[l & 1] : s.qkv + 3 * l * s.sMr) + (long long)b * S * r;
            const float sc = k ? 1.f : scale;
            tb_mix(X, r, sm.sc, ss, S, dh, h0, hg, sm.red, [&](int c, bool two, const float (&v)[4]) {
                const float y0 = v[0] * sc, y1 = v[1] * sc, y2 = v[2] * sc, y3 = v[3] * sc;
                const int w = (k + 1) * r + c;
                tb_put1(sm.wide, p.ka, q, w, y0); tb_put1(sm.wide, p.ka, q + 8, w, y2);
                if (two) { tb_put1(sm.wide, p.ka, q, w + 1, y1); tb_put1(sm.wide, p.ka, q + 8, w + 1, y3); }
                float* o = dqkv + (k + 1) * s.sMr + (long long)q * r + c;
                if (live0) { o[0] = y0; if (two) o[1] = y1; }
                if (live1) { o[8LL * r] = y2; if (two) o[8LL * r + 1] = y3; }
            });
            __syncthreads();
        }
        for (int c = lane; c < r; c += 32) tb_put1(sm.wide, p.ka, warp, c, warp < nt ? __ldg(dqkv + warp * r + c) : 0.f);
    } else {
        // da_L: the same vector for every token of the sample
        const int t = warp;
        for (int c = lane; c < r; c += 32) {
            const int e = t * r + c;
            const float v = t < nt ? __ldg(p.daL + (long long)b * r + c) : 0.f;
            sm.xb[t * rs + c] = v;
            tb_put1(sm.narrow, p.kb, t, c, v);
            if (t < nt) s.da[p.head * s.sMr + m0 * r + e] = v;
        }
    }
    __syncthreads();
#pragma unroll 1
    for (int ph = first; ph < last; ++ph) {
        const int l = ph ? p.head : p.tail;
        const long long o = l * s.sMr + m0 * r, o_hid = l * s.sMf + m0 * f;
        float* part = s.part + ((long long)l * gridDim.x + blockIdx.x) * s.part_w;
        const float* xhat = (ph ? s.xhat2 : s.xhat1) + o;
        if (ph == 1)                                   // dc2: column sums of da
            for (int c = threadIdx.x; c < r; c += TBF_THREADS) {
                float a = 0.f;
#pragma unroll
                for (int t = 0; t < TBF_T; ++t) a += sm.xb[t * rs + c];
                part[4 * r + c] = a;
            }
        const bool wide_in = !(ph & 1);
        tb_product(st, p.mats[ph], wide_in ? sm.wide : sm.narrow, wide_in ? p.ka : p.kb, sm.red, [&](int n, const float (&v)[4]) {
            if (ph == 1) {                             // dpre = dhid where the unit is open; dc1
                const float2 z = make_float2(0.f, 0.f);
                const float* hid = s.hid + o_hid + (long long)q * f;
                const bool ev = (f & 1) == 0;
                const float2 h0 = live0 ? tb_ld2(hid, n, f, ev) : z, h1 = live1 ? tb_ld2(hid + 8LL * f, n, f, ev) : z;
                const float y0 = h0.x > 0.f ? v[0] : 0.f, y1 = h0.y > 0.f ? v[1] : 0.f, y2 = h1.x > 0.f ? v[2] : 0.f, y3 = h1.y > 0.f ? v[3] : 0.f;
                const float c0 = tb_col_sum(y0, y2), c1 = tb_col_sum(y1, y3);
                if (n < f) {
                    const bool two = n + 1 < f;
                    tb_put2(sm.wide, p.ka, q, n, y0, y1); tb_put2(sm.wide, p.ka, q + 8, n, y2, y3);
                    float* out = s.dpre + o_hid + (long long)q * f + n;
                    if (live0) { out[0] = y0; if (two) out[1] = y1; }
                    if (live1) { out[8LL * f] = y2; if (two) out[8LL * f + 1] = y3; }
                    if (q == 0) { part[5 * r + n] = c0; if (two) part[5 * r + n + 1] = c1; }
                }
            } else {
                const bool norm = ph < 3, two = n + 1 < r;
                float gx = 0.f, gy = 0.f, bx = 0.f, by = 0.f;
                if (norm) {                            // dg = sum dn xhat, db = sum dn
                    const float2 z = make_float2(0.f, 0.f);
                    const float2 x0 = live0 ? tb_ld2(xhat + (long long)q * r, n, r, even) : z, x1 = live1 ? tb_ld2(xhat + (long long)(q + 8) * r, n, r, even) : z;
                    gx = tb_col_sum(v[0] * x0.x, v[2] * x1.x); gy = tb_col_sum(v[1] * x0.y, v[3] * x1.y);
                    bx = tb_col_sum(v[0], v[2]); by = tb_col_sum(v[1], v[3]);
                }
                if (n < r) {
                    float* d = sm.qf + q * rs + n;
                    *reinterpret_cast<float2*>(d) = make_float2(v[0], v[1]);
                    *reinterpret_cast<float2*>(d + 8 * rs) = make_float2(v[2], v[3]);
                    if (norm && q == 0) {
                        float* w = part + (ph ? 2 * r : 0) + n;
                        w[0] = gx; w[r] = bx;
                        if (two) { w[1] = gy; w[r + 1] = by; }
                    }
                    if (!norm) {
                        float* out = s.dob[l & 1] + (m0 + q) * r + n;
                        if (live0) { out[0] = v[0]; if (two) out[1] = v[1]; }
                        if (live1) { out[8LL * r] = v[2]; if (two) out[8LL * r + 1] = v[3]; }
                    }
                }
            }
        });
        __syncthreads();
        if (ph & 1) continue;
        // LayerNorm backward, a row per warp: dx = (gradient past the norm) + (dxhat - mean(dxhat) - xhat mean(dxhat xhat)) rstd;
        // then dx1 of `head`, or the merge x = lambda u + (1 - lambda) a_prev of `tail`, whose da goes on to the layer below
        const float* g = ph ? p.g2 : p.g1;
        const float* rstd = (ph ? s.rstd2 : s.rstd1) + l * s.sM + m0;
        const float* dx1 = s.dx1 + o;
        const float lm = __ldg(p.lam + l);
        const float *u = p.u + l * p.u_stride + m0 * r, *ap = l > 0 ? s.a + (l - 1) * p.u_stride + m0 * r : nullptr;
        float acc = 0.f;
        for (int t = warp; t < TBF_T; t += TBF_WARPS) {
            float dxh[TBF_MAX_R / 32], xh[TBF_MAX_R / 32], s1 = 0.f, s2 = 0.f;
            const bool live = t < nt;
#pragma unroll
            for (int i = 0; i < TBF_MAX_R / 32; ++i) {
                const int c = lane + 32 * i;
                dxh[i] = xh[i] = 0.f;
                if (c < r && live) {
                    dxh[i] = sm.qf[t * rs + c] * __ldg(g + c);
                    xh[i] = __ldg(xhat + t * r + c);
                    s1 += dxh[i];
                    s2 = fmaf(dxh[i], xh[i], s2);
                }
            }
            s1 = warp_sum(s1) / (float)r;
            s2 = warp_sum(s2) / (float)r;
            const float rsd = live ? __ldg(rstd + t) : 0.f;
#pragma unroll
            for (int i = 0; i < TBF_MAX_R / 32; ++i) {
                const int c = lane + 32 * i, e = t * r + c;
                if (c >= r) continue;
                float y = 0.f;
                if (live) {
                    y = (ph ? sm.xb[t * rs + c] : __ldg(dx1 + e)) + (dxh[i] - s1 - xh[i] * s2) * rsd;
                    if (ph) s.dx1[o + e] = y;
                    else {
                        acc = fmaf(y, __ldg(u + e) - (ap ? __ldg(ap + e) : 0.f), acc);
                        p.du[l * p.u_stride + m0 * r + e] = lm * y;
                        y *= 1.f - lm;
                        if (p.head >= 0) s.da[p.head * s.sMr + m0 * r + e] = y;
                    }
                }
                sm.xb[t * rs + c] = y;
                tb_put1(sm.narrow, p.kb, t, c, y);
            }
        }
        if (ph == 0) {
            const float tot = block_sum(acc, lam_red);
            if (threadIdx.x == 0) part[5 * r + f] = tot;
        }
        __syncthreads();
    }
    if (p.head < 0) return;
    const int l = p.head;
    // own queries: dP = do v^T, dS = P (dP - sum dP P), dq = scale dS k
#pragma unroll 1
    for (int h0 = 0; h0 < H; h0 += p.hg) {
        const int hg = min(p.hg, H - h0);
        tb_scores(s.qkv + (3 * l + 2) * s.sMr + (long long)b * S * r, r, sm.qf, rs, S, dh, h0, hg, sm.sc, ss);
        __syncthreads();
        for (int w = warp * 4; w < hg * TBF_T; w += TBF_WARPS * 4) {
            float* row = sm.sc + w * ss;
            const int t = w & (TBF_T - 1), h = h0 + (w >> 4);
            const long long po = (((long long)b * H + h) * S + t0 + t) * S;
            const float* P = s.P + l * s.sP + po;
            float* dS = s.dS[l & 1] + po;
            float dot[4] = {};
#pragma unroll 4
            for (int j = lane; j < S; j += 32)
#pragma unroll
                for (int i = 0; i < 4; ++i) dot[i] = fmaf(row[i * ss + j], t + i < nt ? __ldg(P + i * S + j) : 0.f, dot[i]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int i = 0; i < 4; ++i) dot[i] += __shfl_xor_sync(0xffffffffu, dot[i], o);
#pragma unroll 4
            for (int j = lane; j < S16; j += 32)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const bool live = t + i < nt && j < S;
                    const float v = live ? __ldg(P + i * S + j) * (row[i * ss + j] - dot[i]) : 0.f;
                    row[i * ss + j] = v;
                    if (live) dS[i * S + j] = v;
                }
        }
        __syncthreads();
        tb_mix(s.qkv + (3 * l + 1) * s.sMr + (long long)b * S * r, r, sm.sc, ss, S, dh, h0, hg, sm.red, [&](int c, bool two, const float (&v)[4]) {
            float* o = s.dqkv + 3 * l * s.sMr + (m0 + q) * r + c;
            if (live0) { o[0] = v[0] * scale; if (two) o[1] = v[1] * scale; }
            if (live1) { o[8LL * r] = v[2] * scale; if (two) o[8LL * r + 1] = v[3] * scale; }
        });
        __syncthreads();
    }
}

// Column sums of the CTAs' partial sums, in CTA order within each of eight lanes-of-CTAs: grid (part_w / 32, L).
__global__ void __launch_bounds__(256) tb_reduce_parts_kernel(const float* __restrict__ part, int ctas, int part_w, int r, int f, BodyLayout bl,
                                                              float* __restrict__ gbody, float* __restrict__ glam) {
    __shared__ float sm[8][33];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, c = blockIdx.x * 32 + lane, l = blockIdx.y;
    float acc = 0.f;
    if (c < part_w)
        for (int i = w; i < ctas; i += 8) acc += part[((long long)l * ctas + i) * part_w + c];
    sm[w][lane] = acc;
    __syncthreads();
    if (w != 0 || c >= part_w) return;
    float v = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) v += sm[i][lane];
    if (c == 5 * r + f) { glam[l] = v; return; }
    float* g = gbody + l * bl.per_layer;
    const int q = c / r, j = c - q * r;
    if (c >= 5 * r) g[bl.c1 + c - 5 * r] = v;
    else g[(q == 0 ? bl.g1 : q == 1 ? bl.b1 : q == 2 ? bl.g2 : q == 3 ? bl.b2 : bl.c2) + j] = v;
}

// The six weight products' row slices added up in slice order; their parameters of layer l follow wq.
__global__ void __launch_bounds__(256) tb_reduce_slices_kernel(const float* __restrict__ part, int slices, long long slice_stride, long long per_layer,
                                                               BodyLayout bl, float* __restrict__ gbody) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= per_layer) return;
    const float* p = part + blockIdx.y * per_layer + e;
    float v = p[0];
    for (int s = 1; s < slices; ++s) v += p[s * slice_stride];
    // compact order: Wq Wk Wv Wo | W1 | W2
    const long long rr4 = 4LL * bl.r * bl.r, rf = (long long)bl.r * bl.f;
    float* g = gbody + blockIdx.y * bl.per_layer;
    g[e < rr4 ? bl.wq + e : e < rr4 + rf ? bl.w1 + e - rr4 : bl.w2 + e - rr4 - rf] = v;
}

struct TbPlan {
    bool ok = false;
    int hg = 0, ka = 0, kb = 0, rs = 0, ss = 0;
    size_t smem = 0;
};

inline TbPlan tb_plan(int S, int r, int f, int H, int max_smem) {
    TbPlan pl;
    if (r > TBF_MAX_R || (long long)f * r > (1 << 22)) return pl;
    pl.ka = tb_up16(f > 3 * r ? f : 3 * r) + 8;
    pl.kb = tb_up16(r) + 8;
    pl.rs = (r + 31) / 32 * 32 + 8;            // = 8 mod 32: the fragments' pairs of four rows fall into different banks
    pl.ss = (tb_up16(S) + 31) / 32 * 32 + 8;
    const size_t fixed = TBF_FIXED + tb_smem_terms(pl.ka) + tb_smem_terms(pl.kb) + sizeof(float) * 2 * TBF_T * pl.rs;
    const size_t per_head = sizeof(float) * TBF_T * pl.ss;
    const size_t most = (size_t)max_smem - 1024;
    if (fixed + per_head > most) return pl;
    const int fit = (int)((most - fixed) / per_head);
    const int groups = (H + fit - 1) / fit;
    pl.hg = (H + groups - 1) / groups;         // heads in even groups
    pl.smem = fixed + pl.hg * per_head;
    if (smem_opt_in((const void*)tb_fwd_kernel, pl.smem) != cudaSuccess || smem_opt_in((const void*)tb_bwd_kernel, pl.smem) != cudaSuccess) {
        cudaGetLastError();
        return pl;
    }
    pl.ok = true;
    return pl;
}

inline int tb_ctas(int B, int S) { return B * ((S + TBF_T - 1) / TBF_T); }

inline cudaError_t tb_layer_launch(const TbPlan& pl, TbLayerParams p, bool backward, cudaStream_t stream) {
    p.tiles = (p.S + TBF_T - 1) / TBF_T;
    p.hg = pl.hg; p.ka = pl.ka; p.kb = pl.kb; p.rs = pl.rs; p.ss = pl.ss;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    pdl_launch_config(&cfg, attr, dim3((unsigned)tb_ctas(p.B, p.S)), dim3(TBF_THREADS), pl.smem, stream);
    return backward ? cudaLaunchKernelEx(&cfg, tb_bwd_kernel, p) : cudaLaunchKernelEx(&cfg, tb_fwd_kernel, p);
}

}  // namespace pac
