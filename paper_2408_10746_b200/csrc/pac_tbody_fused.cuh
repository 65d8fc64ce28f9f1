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
//
// A launch is one chain of about ten dependent phases on 16 warps, so latency bounds it, not a rate: everything that is final before the
// phase that needs it is requested ahead (weights through a ring of asynchronous copies that runs across phases, q, k, v and the residual rows
// before the attention, gate bits before the product ahead of them), scores, softmax and its reverse stay in the registers of
// the tensor instructions' fragments, a token's residual row stays in the registers of the warp that owns it, and halves of sums along K meet in
// the row phase that reads them instead of in a phase of their own.  Weights arrive split and in the order in which a warp consumes them
// (tb_pack_kernel).  Against scores, weights and rows in shared memory and weights split by their readers the step at B = 16, S = 128, r = 64, 12 layers went
// from 953 to 769 us; parameter vectors as asynchronous copies and plain addresses where nothing needs clamping made it 748.  Twice the warps with half the registers
// took 1028: what does not fit spills past an L1 that shared memory leaves no room.  Loads of the second attention's operands ahead of the product before them cost 64 us in spilled registers.
#pragma once
#include "pac_tbody.cuh"
#include "pac_tensor.cuh"

namespace pac {

constexpr int TBF_THREADS = 512, TBF_WARPS = TBF_THREADS / 32, TBF_T = 16, TBF_MAX_R = 192;

__host__ __device__ inline int tb_up16(int x) { return (x + 15) & ~15; }
__host__ __device__ inline int tb_up8(int x) { return (x + 7) & ~7; }

// One weight matrix: K x N in 16 x 8 tiles, ks along K, nt along N.  A product whose output is r wide and has up to eight tiles along N is cut in half along K
// between warps 0 - 7 and 8 - 15, every other one has its tiles dealt to the warps in turn.  A warp takes its tiles in pairs 16 apart, k step by k step, or
// one tile two k steps at a time: two tiles either way, one unit of its stream.
struct TbMat {
    int ks, nt;
    bool cut;
    __host__ __device__ int from(int warp) const { return cut && warp >= TBF_WARPS / 2 ? (ks + 1) / 2 : 0; }
    __host__ __device__ int to(int warp) const { return cut && warp < TBF_WARPS / 2 ? (ks + 1) / 2 : ks; }
    __host__ __device__ int first(int warp) const { return cut ? warp & (TBF_WARPS / 2 - 1) : warp; }
    __host__ __device__ int tiles(int warp) const {            // of this warp
        const int j = first(warp);
        return j >= nt ? 0 : cut ? 1 : (nt - j + TBF_WARPS - 1) / TBF_WARPS;
    }
    __host__ __device__ int units(int warp) const {
        const int n = tiles(warp);
        return (n >> 1) * ks + (n & 1) * ((to(warp) - from(warp) + 1) >> 1);
    }
};

// A unit: two tiles in three bf16 terms.  512 bytes each of first and second terms (lane l of a tile holds, of column l / 4, rows 2 (l % 4) + {0, 1} and
// {8, 9}: two words per term), then 256 bytes each of third terms.
constexpr int TB_UNIT = 1536;

// The packed weights of one layer: four streams (Wo W1 W2 | Wqkv | Wqkv^T | W2^T W1^T Wo^T: what one launch reads of a layer), a warp's units consecutive in each.
struct TbPack {
    int r, f;
    int off[4][TBF_WARPS + 1];         // first unit of a warp in a stream; total
    int base[5];                       // first unit of a stream; per layer
    static __host__ __device__ int stream(int m) { return m < 3 ? 0 : m - 2 < 3 ? m - 2 : 3; }
    __host__ __device__ TbMat mat(int m) const {
        const int K = m == 2 || m == 6 ? f : m == 4 ? 3 * r : r, n8 = m == 1 || m == 5 ? tb_up8(f) : m == 3 ? 3 * tb_up8(r) : tb_up8(r);
        return TbMat{tb_up16(K) / 16, n8 / 8, m != 1 && m != 3 && m != 5 && n8 / 8 <= TBF_WARPS / 2};
    }
    static TbPack make(int r, int f) {
        TbPack p;
        p.r = r; p.f = f;
        int at = 0;
        for (int s = 0; s < 4; ++s) {
            int o = 0;
            for (int w = 0; w < TBF_WARPS; ++w) {
                p.off[s][w] = o;
                for (int m = 0; m < 8; ++m) if (stream(m) == s) o += p.mat(m).units(w);
            }
            p.off[s][TBF_WARPS] = o;
            p.base[s] = at;
            at += o;
        }
        p.base[4] = at;
        return p;
    }
    size_t layer_bytes() const { return (size_t)base[4] * TB_UNIT; }
    int tiles() const { int t = 0; for (int m = 0; m < 8; ++m) t += mat(m).ks * mat(m).nt; return t; }
};

__device__ __forceinline__ void tb_split_b(uint32_t (&h)[2], uint32_t (&m)[2], uint32_t (&l)[2], float k0, float k1, float k8, float k9) {
    split3_pair(k0, k1, h[0], m[0], l[0]);
    split3_pair(k8, k9, h[1], m[1], l[1]);
}

// Splits the weights of every layer and lays them out in stream order, a tile per warp: grid (tiles / 8, L).
__global__ void __launch_bounds__(256) tb_pack_kernel(const float* __restrict__ body, long long body_per, BodyLayout bl,
                                                      const __grid_constant__ TbPack p, unsigned char* __restrict__ packed) {
    const float* w = body + blockIdx.y * body_per;
    const int r = p.r, f = p.f, r8 = tb_up8(r), lane = threadIdx.x & 31;
    int tile = blockIdx.x * 8 + (threadIdx.x >> 5), m = 0;
    TbMat mt = p.mat(0);
    while (tile >= mt.ks * mt.nt) {
        tile -= mt.ks * mt.nt;
        if (++m == 8) return;
        mt = p.mat(m);
    }
    const int ks = tile / mt.nt, j = tile - ks * mt.nt, K = m == 2 || m == 6 ? f : m == 4 ? 3 * r : r;
    const int k0 = ks * 16 + 2 * (lane & 3), n = j * 8 + (lane >> 2);
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
        else if (m == 4) { const int s = k / r, c = k - s * r; if (n < r) v[i] = w[bl.wq + (s * r + n) * r + c]; }
        else if (m == 5) { if (n < f) v[i] = w[bl.w2 + n * r + k]; }
        else if (m == 6) { if (n < r) v[i] = w[bl.w1 + n * f + k]; }
        else if (n < r) v[i] = w[bl.wo + n * r + k];
    }
    const int half = mt.cut && ks >= (mt.ks + 1) / 2 ? TBF_WARPS / 2 : 0, warp = mt.cut ? j + half : j & (TBF_WARPS - 1), step = ks - mt.from(warp);
    const int i = mt.cut ? 0 : j / TBF_WARPS, pairs = i >> 1;
    const bool pair = (i | 1) < mt.tiles(warp);
    const int s = TbPack::stream(m);
    int unit = p.base[s] + p.off[s][warp] + pairs * mt.ks + (pair ? step : step >> 1);
    for (int q = 0; q < m; ++q) if (TbPack::stream(q) == s) unit += p.mat(q).units(warp);
    const int sub = pair ? i & 1 : step & 1;
    uint32_t h[2], mm[2], l[2];
    tb_split_b(h, mm, l, v[0], v[1], v[2], v[3]);
    unsigned char* dst = packed + (blockIdx.y * (long long)p.base[4] + unit) * TB_UNIT;
    *reinterpret_cast<uint4*>(dst + sub * 512 + lane * 16) = make_uint4(h[0], h[1], mm[0], mm[1]);
    *reinterpret_cast<uint2*>(dst + 1024 + sub * 256 + lane * 8) = make_uint2(l[0], l[1]);
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
    const unsigned char *w0, *w1;      // packed streams: of `tail`'s phases, then of `head`'s
    int off0[TBF_WARPS + 1], off1[TBF_WARPS + 1];
    int tail, head;                    // forward: layer whose attention + feed-forward half runs / layer whose q, k, v are formed (-1: none);
                                       // backward: layer whose dk, dv + merge run / layer whose feed-forward + dq run
    int B, S, r, f, H;
    int nc, hg;                        // warps per head (32 keys each and round), heads at a time
    int tiles;                         // CTAs per sample
    int train;
    int ka, kb, rs;                    // row strides in shared memory: wide and narrow operand terms (bf16), fp32 rows
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
__device__ __forceinline__ void tb_split_a(TbA& a, const float (&v)[8]) {      // pairs (row q, q + 8) x (columns c2, c2 + 8)
#pragma unroll
    for (int i = 0; i < 4; ++i) split3_pair(v[2 * i], v[2 * i + 1], a.h[i], a.m[i], a.l[i]);
}
// The products in two accumulators: first terms, and the smaller ones.
__device__ __forceinline__ void tb_mma6(float (&big)[4], float (&small)[4], const TbA& a, const TbB& b) {
    tb_mma(small, a.m, b.m); tb_mma(big, a.h, b.h); tb_mma(small, a.h, b.l);
    tb_mma(small, a.l, b.h); tb_mma(small, a.h, b.m); tb_mma(small, a.m, b.h);
}
__device__ __forceinline__ void tb_ldmatrix4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
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
// A warp's own stream of weight units, U of them in flight: it runs ahead of the products, across phases, and starts before the wait for the
// predecessor launch.  Copies are per lane and read by the whole warp, so the ring needs no barrier beyond the warp.
template <int U>
struct TbStream {
    const unsigned char *src, *next_src;
    int left, next_left;
    uint32_t ring;                     // of the warp
    uint32_t put = 0, get = 0;         // byte offsets in it
    __device__ __forceinline__ TbStream(const TbLayerParams& p, unsigned char* mem) {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        ring = smem_u32(mem) + warp * (U * TB_UNIT);
        src = p.w0 + (long long)p.off0[warp] * TB_UNIT + lane * 16;
        left = p.tail >= 0 ? p.off0[warp + 1] - p.off0[warp] : 0;
        next_src = p.w1 + (long long)p.off1[warp] * TB_UNIT + lane * 16;
        next_left = p.head >= 0 ? p.off1[warp + 1] - p.off1[warp] : 0;
    }
    __device__ __forceinline__ void issue() {
        if (left == 0) { src = next_src; left = next_left; next_left = 0; }
        if (left > 0) {
            const uint32_t d = ring + put + (threadIdx.x & 31) * 16;
#pragma unroll
            for (int i = 0; i < 3; ++i) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + i * 512), "l"(src + i * 512) : "memory");
            src += TB_UNIT;
            --left;
        }
        put = put + TB_UNIT == U * TB_UNIT ? 0 : put + TB_UNIT;
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    // The next unit's tiles, and another unit sent for.
    __device__ __forceinline__ void next(TbB (&b)[2]) {
        asm volatile("cp.async.wait_group %0;" ::"n"(U - 1) : "memory");
        __syncwarp();
        const uint32_t a = ring + get, lane = threadIdx.x & 31;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(b[i].h[0]), "=r"(b[i].h[1]), "=r"(b[i].m[0]), "=r"(b[i].m[1]) : "r"(a + i * 512 + lane * 16) : "memory");
            asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(b[i].l[0]), "=r"(b[i].l[1]) : "r"(a + 1024 + i * 256 + lane * 8) : "memory");
        }
        get = get + TB_UNIT == U * TB_UNIT ? 0 : get + TB_UNIT;
        __syncwarp();
        issue();
    }
};

// out = act W for the 16 tokens: act's terms at pl, W the stream's next matrix.  ep(half, i, n, v): columns n, n + 1 of rows lane / 4 (v[0], v[1])
// and lane / 4 + 8 (v[2], v[3]), the half's share of the sum where the matrix is cut; i counts the warp's tiles; called by whole warps.
// First terms are added up in two accumulators per tile, the smaller products in a third.
template <int U, class EP>
__device__ __forceinline__ void tb_product(TbStream<U>& st, const TbMat& m, const bf16* pl, int stride, EP ep) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, half = m.cut ? warp >> 3 : 0;
    const uint32_t a00 = smem_u32(pl) + (((lane & 15) * stride) + (lane >> 4) * 8) * 2, term = 32 * stride;
    const int tiles = m.tiles(warp), from = m.from(warp), steps = m.to(warp) - from, j = m.first(warp);
#pragma unroll 1
    for (int i = 0; i < tiles; i += 2) {
        const bool pair = i + 1 < tiles;
        const int units = pair ? steps : (steps + 1) >> 1;
        const uint32_t to_second = pair ? 0 : 32, step = pair ? 32 : 64;
        uint32_t ad = a00 + from * 32;
        float acc[2][3][4] = {};
#pragma unroll 1
        for (int u = 0; u < units; u += 2) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                if (u + e >= units) break;
                TbB b[2];
                TbA a;
                tb_ldmatrix4(a.h, ad); tb_ldmatrix4(a.m, ad + term); tb_ldmatrix4(a.l, ad + 2 * term);
                st.next(b);
                tb_mma6(acc[0][1 + e], acc[0][0], a, b[0]);
                if (pair || 2 * (u + e) + 1 < steps) {
                    if (!pair) { tb_ldmatrix4(a.h, ad + to_second); tb_ldmatrix4(a.m, ad + to_second + term); tb_ldmatrix4(a.l, ad + to_second + 2 * term); }
                    tb_mma6(acc[1][1 + e], acc[1][0], a, b[1]);
                }
                ad += step;
            }
        }
        float v[2][4];
#pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
            for (int e = 0; e < 4; ++e) v[k][e] = (acc[k][2][e] + acc[k][1][e]) + acc[k][0][e];
        const int n = (j + i * TBF_WARPS) * 8 + 2 * (lane & 3);
        if (pair) {
            ep(half, i, n, v[0]);
            ep(half, i + 1, n + TBF_WARPS * 8, v[1]);
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) v[0][e] += v[1][e];
            ep(half, i, n, v[0]);
        }
    }
}

// Two consecutive floats of a row (zeros past n); `even`: the row starts on an 8-byte boundary.
__device__ __forceinline__ float2 tb_ld2(const float* __restrict__ p, int c, int n, bool even) {
    if (even && c + 1 < n) return __ldg(reinterpret_cast<const float2*>(p + c));
    return make_float2(c < n ? __ldg(p + c) : 0.f, c + 1 < n ? __ldg(p + c + 1) : 0.f);
}
__device__ __forceinline__ void tb_st2(float* p, float x, float y, bool two, bool even) {
    if (even && two) *reinterpret_cast<float2*>(p) = make_float2(x, y);
    else { p[0] = x; if (two) p[1] = y; }
}

// First key of a warp's round w.  With several rounds the compiler would form the addresses of all of them ahead of the loops and spill them; the value is therefore opaque.
template <int CW>
__device__ __forceinline__ int tb_round(int key0, int key_step, int w) {
    int k = key0 + w * key_step;
    if (CW > 1) asm volatile("" : "+r"(k));
    return k;
}
// 32 rows (keys) x 16 columns of a head, as the B operand of scores: pair (c2, c2 + 1) and (c2 + 8, + 9) of row 8 n + lane / 4.  X: the head's first column
// of the sample's rows; columns from `cols` on are zeros, rows from S on repeat the last one.
struct TbKeys { float2 x[4][2]; };
__device__ __forceinline__ void tb_load_keys(TbKeys& o, const float* __restrict__ X, int r, int key0, int S, int k, int cols, bool even) {
    const int lane = threadIdx.x & 31, q = lane >> 2, c2 = 2 * (lane & 3);
    if (even && key0 + 32 <= S && k + 16 <= cols) {            // nothing to clamp
        const float* x = X + (key0 + q) * r + k + c2;
#pragma unroll
        for (int n = 0; n < 4; ++n, x += 8 * r) { o.x[n][0] = __ldg(reinterpret_cast<const float2*>(x)); o.x[n][1] = __ldg(reinterpret_cast<const float2*>(x) + 4); }
        return;
    }
#pragma unroll
    for (int n = 0; n < 4; ++n) {
        const float* x = X + min(key0 + n * 8 + q, S - 1) * r;
        o.x[n][0] = tb_ld2(x, k + c2, cols, even); o.x[n][1] = tb_ld2(x, k + c2 + 8, cols, even);
    }
}
// acc[n] += act (16 tokens x 16 columns) keys^T: scores of 32 keys.
__device__ __forceinline__ void tb_scores(float (&acc)[4][4], const TbA& a, const TbKeys& k) {
#pragma unroll
    for (int n = 0; n < 4; ++n) {
        TbB b;
        tb_split_b(b.h, b.m, b.l, k.x[n][0].x, k.x[n][0].y, k.x[n][1].x, k.x[n][1].y);
        float small[4] = {};
        tb_mma6(acc[n], small, a, b);
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[n][e] += small[e];
    }
}
// 32 rows x 16 columns of a head, as the B operand of a mix over rows.
struct TbVals { float v[2][2][4]; };
__device__ __forceinline__ void tb_load_vals(TbVals& o, const float* __restrict__ X, int r, int key0, int S, int n0, int dh) {
    const int lane = threadIdx.x & 31, q = lane >> 2, c2 = 2 * (lane & 3);
    const bool full = key0 + 32 <= S;
    const float *x0 = X + min(n0 + q, dh - 1), *x1 = X + min(n0 + 8 + q, dh - 1);
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int j = key0 + 16 * k + c2 + (i & 1) + (i >> 1) * 8, at = (full ? j : min(j, S - 1)) * r;
            o.v[k][0][i] = __ldg(x0 + at);
            o.v[k][1][i] = __ldg(x1 + at);
        }
}
// acc[n] += weights (16 tokens x 16 rows, zero past the last row) vals, k the k step of the 32 rows.
__device__ __forceinline__ void tb_mix(float (&big)[2][4], float (&small)[2][4], const TbA& a, const TbVals& x, int k) {
#pragma unroll
    for (int n = 0; n < 2; ++n) {
        TbB b;
        tb_split_b(b.h, b.m, b.l, x.v[k][n][0], x.v[k][n][1], x.v[k][n][2], x.v[k][n][3]);
        tb_mma6(big[n], small[n], a, b);
    }
}
// Score fragments (tiles 2 k, 2 k + 1) as the A operand of k step k.
__device__ __forceinline__ void tb_frag_a(TbA& a, const float (&sc)[4][4], int k) {
    const float v[8] = {sc[2 * k][0], sc[2 * k][1], sc[2 * k][2], sc[2 * k][3], sc[2 * k + 1][0], sc[2 * k + 1][1], sc[2 * k + 1][2], sc[2 * k + 1][3]};
    tb_split_a(a, v);
}

// Shares of a mix: 16 tokens x 16 columns per warp; columns of every other row pair are swapped by eights, which spreads the fragments' rows over the banks.
constexpr int TB_SHARE = TBF_T * 16;
__device__ __forceinline__ void tb_share_put(float* part, const float (&big)[2][4], const float (&small)[2][4]) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = lane >> 2, c2 = 2 * (lane & 3), sw = ((q >> 1) & 1) * 8;
    float* o = part + warp * TB_SHARE + q * 16;
#pragma unroll
    for (int n = 0; n < 2; ++n) {
        *reinterpret_cast<float2*>(o + ((n * 8 + c2) ^ sw)) = make_float2(big[n][0] + small[n][0], big[n][1] + small[n][1]);
        *reinterpret_cast<float2*>(o + 8 * 16 + ((n * 8 + c2) ^ sw)) = make_float2(big[n][2] + small[n][2], big[n][3] + small[n][3]);
    }
}
// Sums of the nc shares of each of n heads, in order: ep(head, column, value) for token `warp`, columns n0 .. n0 + 15 of a head dh wide.
template <class EP>
__device__ __forceinline__ void tb_share_sum(const float* part, int nc, int n, int n0, int dh, EP ep) {
    const int t = threadIdx.x >> 5, lane = threadIdx.x & 31, sw = ((t >> 1) & 1) * 8, cc = lane & 15;
    for (int h = lane >> 4; h < n; h += 2) {
        if (n0 + cc >= dh) continue;
        const float* s = part + h * nc * TB_SHARE + t * 16 + (cc ^ sw);
        float v = s[0];
        for (int i = 1; i < nc; ++i) v += s[i * TB_SHARE];
        ep(h, n0 + cc, v);
    }
}

// Sum over the 16 tokens of a column pair: v of tb_product's epilogue, the result in every lane of the column.
__device__ __forceinline__ float tb_col_sum(float top, float bottom) {
    float s = top + bottom;
    s += __shfl_xor_sync(0xffffffffu, s, 4);
    s += __shfl_xor_sync(0xffffffffu, s, 8);
    s += __shfl_xor_sync(0xffffffffu, s, 16);
    return s;
}
// Column sums of 16 rows in shared memory: a warp four columns at a time, eight lanes each.
__device__ __forceinline__ void tb_col_sums(const float* rows, int rs, int r, float* __restrict__ out) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, t = lane & 7;
    for (int c0 = warp * 4; c0 < r; c0 += TBF_WARPS * 4) {
        const int c = c0 + (lane >> 3), cc = min(c, r - 1);
        float s = rows[t * rs + cc] + rows[(t + 8) * rs + cc];
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (t == 0 && c < r) out[c] = s;
    }
}
__device__ __forceinline__ float tb_quad_max(float v) {
    v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 1));
    return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 2));
}
__device__ __forceinline__ float tb_quad_sum(float v) {
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    return v + __shfl_xor_sync(0xffffffffu, v, 2);
}

// e / d, rounded correctly for a correctly rounded inverse (Markstein, IBM J. Res. Dev. 34, 1990).
__device__ __forceinline__ float tb_quotient(float e, float d, float inverse) {
    const float x = e * inverse;
    return fmaf(fmaf(-x, d, e), inverse, x);
}

// Shared memory: weight ring | operand terms wide, narrow | fp32 rows (four products' worth) | parameter vectors | row statistics | shares of mixes, two rounds.
struct TbSmem { unsigned char* ring; bf16 *wide, *narrow; float *rows, *vec, *stat0, *stat1, *share; };
__host__ __device__ inline size_t tb_smem_terms(int stride) { return (size_t)3 * TBF_T * stride * 2; }
__host__ __device__ inline int tb_vec_floats(int r, int f) { return tb_up8(5 * r + f); }
__host__ __device__ inline size_t tb_smem_fixed(int ka, int kb, int rs, int r, int f) {
    return tb_smem_terms(ka) + tb_smem_terms(kb) + sizeof(float) * (4 * TBF_T * rs + tb_vec_floats(r, f) + 2 * TBF_WARPS * TBF_T + 2 * TBF_WARPS * TB_SHARE);
}
__device__ __forceinline__ TbSmem tb_carve(unsigned char* base, size_t ring, const TbLayerParams& p) {
    TbSmem s;
    s.ring = base;
    s.wide = reinterpret_cast<bf16*>(base + ring);
    s.narrow = s.wide + 3 * TBF_T * p.ka;
    s.rows = reinterpret_cast<float*>(s.narrow + 3 * TBF_T * p.kb);
    s.vec = s.rows + 4 * TBF_T * p.rs;
    s.stat0 = s.vec + tb_vec_floats(p.r, p.f);
    s.stat1 = s.stat0 + TBF_WARPS * TBF_T;
    s.share = s.stat1 + TBF_WARPS * TBF_T;
    return s;
}
// The padding of the terms is multiplied with zero weights: it has to be finite.
__device__ __forceinline__ void tb_zero_terms(const TbSmem& s, const TbLayerParams& p) {
    uint4* z = reinterpret_cast<uint4*>(s.wide);
    for (int i = threadIdx.x; i < 3 * TBF_T * (p.ka + p.kb) / 8; i += TBF_THREADS) z[i] = make_uint4(0u, 0u, 0u, 0u);
}
// Parameter vectors arrive as asynchronous copies, the oldest group of every thread's ring: tb_vec_wait and a barrier before their first use.
__device__ __forceinline__ void tb_vec_in(float* dst, const float* __restrict__ src, int n) {
    for (int i = threadIdx.x; i < n; i += TBF_THREADS) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst + i)), "l"(src + i) : "memory");
}
template <int U>
__device__ __forceinline__ void tb_vec_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(U) : "memory"); }
// A row's columns lane, lane + 32, ... (zeros past n or where the row is not live).
template <int NR>
__device__ __forceinline__ void tb_row_in(float (&v)[NR], const float* __restrict__ row, int n, bool live) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < NR; ++i) v[i] = live && lane + 32 * i < n ? __ldg(row + lane + 32 * i) : 0.f;
}

// Phases: 0 x1 = x + o Wo, 1 hid = relu(LN2(x1) W1 + c1), 2 a = x1 + hid W2 + c2 (of `tail`), 3 q, k, v = LN1(x) [Wq Wk Wv] (of `head`).
// They run through ONE copy of the code: a phase is executed once per launch, so instructions it does not share are fetched
// from memory.  NR: columns per lane of a row, U: weight units in flight, CW: rounds of 32 keys per warp.
template <int NR, int U, int CW>
__global__ void __launch_bounds__(TBF_THREADS) tb_fwd_kernel(const __grid_constant__ TbLayerParams p) {
    extern __shared__ __align__(128) unsigned char tb_sm[];
    const int b = blockIdx.x / p.tiles, t0 = (blockIdx.x - b * p.tiles) * TBF_T;
    const int S = p.S, r = p.r, f = p.f, H = p.H, dh = r / H, nt = min(TBF_T, S - t0), rs = p.rs;
    const long long m0 = (long long)b * S + t0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, q = lane >> 2, c2 = 2 * (lane & 3);
    const int first = p.tail >= 0 ? 0 : 3, last = p.head >= 0 ? 4 : 3;
    const TbSmem sm = tb_carve(tb_sm, (size_t)TBF_WARPS * U * TB_UNIT, p);
    // (parameters and packed weights were final before the predecessor started)
    if (p.head >= 0) { tb_vec_in(sm.vec, p.g1, r); tb_vec_in(sm.vec + r, p.b1, r); }
    if (p.tail >= 0) {
        tb_vec_in(sm.vec + 2 * r, p.g2, r); tb_vec_in(sm.vec + 3 * r, p.b2, r); tb_vec_in(sm.vec + 4 * r, p.c2, r);
        tb_vec_in(sm.vec + 5 * r, p.c1, f);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    TbStream<U> st(p, tb_sm);
#pragma unroll 1
    for (int i = 0; i < U; ++i) st.issue();
    tb_zero_terms(sm, p);
    const float lm = p.head >= 0 ? __ldg(p.lam + p.head) : 0.f;
    pdl_wait();
    pdl_trigger();
    const TbStacks& s = p.s;
    const bool live = warp < nt;                                // token `warp` is this warp's row
    float res[NR], un[NR];                                      // residual row of `tail`, u row of `head` (ahead of the attention where registers allow it)
    const auto rows_in = [&] {
        if (p.tail >= 0) tb_row_in(res, s.x + p.tail * s.sMr + (m0 + warp) * r, r, live);
        if (p.head >= 0) tb_row_in(un, p.u + p.head * p.u_stride + (m0 + warp) * r, r, live);
    };
    if (CW == 1) rows_in();
    tb_vec_wait<U>();
    __syncthreads();
    if (p.tail >= 0) {
        const float* qkv = s.qkv + 3 * p.tail * s.sMr + (long long)b * S * r;
        const float scale = 1.f / sqrtf((float)dh);
        const bool even = ((dh | r) & 1) == 0, evenS = (S & 1) == 0;
        const int hl = warp / p.nc, key0 = (warp - hl * p.nc) * 32, key_step = p.nc * 32;
        int buf = 0;
#pragma unroll 1
        for (int h0 = 0; h0 < H; h0 += p.hg) {
            const int hg = min(p.hg, H - h0), col = (h0 + hl) * dh;
            const bool mine = hl < hg;
            float sc[CW][4][4] = {};
            TbVals vals;
            float mx[2] = {-INFINITY, -INFINITY};
            if (mine) {
#pragma unroll 1
                for (int k = 0; k < dh; k += 16) {
                    TbKeys keys;
                    float2 qa[2][2];
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const float* row = qkv + (long long)min(t0 + q + 8 * i, S - 1) * r + col;
                        qa[i][0] = tb_ld2(row, k + c2, dh, even); qa[i][1] = tb_ld2(row, k + c2 + 8, dh, even);
                    }
                    if (CW == 1) {
                        tb_load_keys(keys, qkv + s.sMr + col, r, key0, S, k, dh, even);
                        if (k == 0) tb_load_vals(vals, qkv + 2 * s.sMr + col, r, key0, S, 0, dh);
                    }
                    TbA a;
                    const float v[8] = {qa[0][0].x, qa[0][0].y, qa[1][0].x, qa[1][0].y, qa[0][1].x, qa[0][1].y, qa[1][1].x, qa[1][1].y};
                    tb_split_a(a, v);
#pragma unroll
                    for (int w = 0; w < CW; ++w) {
                        if (CW > 1) {
                            const int k0 = tb_round<CW>(key0, key_step, w);
                            if (k0 >= S) break;
                            tb_load_keys(keys, qkv + s.sMr + col, r, k0, S, k, dh, even);
                        }
                        tb_scores(sc[w], a, keys);
                    }
                }
                // softmax over the keys: fragments of rows q and q + 8, keys from S on weigh nothing
#pragma unroll
                for (int w = 0; w < CW; ++w)
#pragma unroll
                    for (int n = 0; n < 4; ++n)
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const bool in = key0 + w * key_step + n * 8 + c2 + (e & 1) < S;
                            sc[w][n][e] = in ? sc[w][n][e] * scale : -INFINITY;
                            mx[e >> 1] = fmaxf(mx[e >> 1], sc[w][n][e]);
                        }
            }
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                mx[i] = tb_quad_max(mx[i]);
                if ((lane & 3) == 0) sm.stat0[warp * TBF_T + q + 8 * i] = mx[i];
            }
            __syncthreads();
            float sum[2] = {};
            if (mine) {
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    mx[i] = -INFINITY;
                    for (int c = 0; c < p.nc; ++c) mx[i] = fmaxf(mx[i], sm.stat0[(hl * p.nc + c) * TBF_T + q + 8 * i]);
                }
#pragma unroll
                for (int w = 0; w < CW; ++w)
#pragma unroll
                    for (int n = 0; n < 4; ++n)
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const bool in = key0 + w * key_step + n * 8 + c2 + (e & 1) < S;
                            sc[w][n][e] = in ? expf(sc[w][n][e] - mx[e >> 1]) : 0.f;
                            sum[e >> 1] += sc[w][n][e];
                        }
            }
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                sum[i] = tb_quad_sum(sum[i]);
                if ((lane & 3) == 0) sm.stat1[warp * TBF_T + q + 8 * i] = sum[i];
            }
            __syncthreads();
            if (mine) {
                float* P = s.P + p.tail * s.sP + (((long long)b * H + h0 + hl) * S + t0 + q) * S;
                float inv[2];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    sum[i] = 0.f;
                    for (int c = 0; c < p.nc; ++c) sum[i] += sm.stat1[(hl * p.nc + c) * TBF_T + q + 8 * i];
                    inv[i] = __frcp_rn(sum[i]);
                }
#pragma unroll
                for (int w = 0; w < CW; ++w) {
                    const int k0 = tb_round<CW>(key0, key_step, w);
                    if (CW > 1 && k0 >= S) break;
#pragma unroll
                    for (int n = 0; n < 4; ++n) {
                        const int key = k0 + n * 8 + c2;
#pragma unroll
                        for (int e = 0; e < 4; ++e) sc[w][n][e] = tb_quotient(sc[w][n][e], sum[e >> 1], inv[e >> 1]);
                        if (p.train && key < S) {
                            if (q < nt) tb_st2(P + key, sc[w][n][0], sc[w][n][1], key + 1 < S, evenS);
                            if (q + 8 < nt) tb_st2(P + 8LL * S + key, sc[w][n][2], sc[w][n][3], key + 1 < S, evenS);
                        }
                    }
                }
            }
#pragma unroll 1
            for (int n0 = 0; n0 < dh; n0 += 16, buf ^= 1) {
                float* share = sm.share + buf * TBF_WARPS * TB_SHARE;
                if (mine) {
                    float big[2][4] = {}, small[2][4] = {};
#pragma unroll
                    for (int w = 0; w < CW; ++w) {
                        const int k0 = tb_round<CW>(key0, key_step, w);
                        if (CW > 1 && k0 >= S) break;
                        if (CW > 1 || n0 > 0) tb_load_vals(vals, qkv + 2 * s.sMr + col, r, k0, S, n0, dh);
#pragma unroll
                        for (int k = 0; k < 2; ++k) {
                            TbA a;
                            tb_frag_a(a, sc[w], k);
                            tb_mix(big, small, a, vals, k);
                        }
                    }
                    tb_share_put(share, big, small);
                }
                __syncthreads();
                float* o = s.o + p.tail * s.sMr + (m0 + warp) * r + h0 * dh;
                tb_share_sum(share, p.nc, hg, n0, dh, [&](int h, int c, float v) {
                    tb_put1(sm.narrow, p.kb, warp, (h0 + h) * dh + c, v);
                    if (p.train && live) o[h * dh + c] = v;
                });
            }
        }
        __syncthreads();
    }
    if (CW > 1) rows_in();
#pragma unroll 1
    for (int ph = first; ph < last; ++ph) {
        if (ph & 1) {
            // LayerNorm 2 of `tail`, or merge and LayerNorm 1 of `head`
            const bool one = ph == 3;
            const int l = one ? p.head : p.tail;
            const long long o = l * s.sMr + (m0 + warp) * r;
            const float *g = sm.vec + (one ? 0 : 2 * r), *be = g + r;
            float *xh_out = (one ? s.xhat1 : s.xhat2) + o, *n_out = (one ? s.n1 : s.n2) + o;
            float v[NR], sum = 0.f, var = 0.f;
#pragma unroll
            for (int i = 0; i < NR; ++i) {
                const int c = lane + 32 * i;
                v[i] = 0.f;
                if (c < r) {
                    if (p.tail >= 0) {
                        const float* y = sm.rows + warp * rs + c;
                        v[i] = res[i];
                        if (one) v[i] += sm.vec[4 * r + c];
                        v[i] = (p.mats[0].cut ? y[0] + y[TBF_T * rs] : y[0]) + v[i];       // (phases 0 and 2 are r wide: cut alike)
                        if (one && live) s.a[p.tail * p.u_stride + (m0 + warp) * r + c] = v[i];
                    }
                    if (one) {
                        v[i] = lm * un[i] + (1.f - lm) * v[i];
                        if (live) s.x[o + c] = v[i];
                    } else {
                        res[i] = v[i];
                    }
                    sum += v[i];
                }
            }
            const float mu = warp_sum(sum) / (float)r;
#pragma unroll
            for (int i = 0; i < NR; ++i)
                if (lane + 32 * i < r) { const float d = v[i] - mu; var = fmaf(d, d, var); }
            const float rstd = 1.f / sqrtf(warp_sum(var) / (float)r + TB_LN_EPS);
#pragma unroll
            for (int i = 0; i < NR; ++i) {
                const int c = lane + 32 * i;
                if (c < r) {
                    const float xh = (v[i] - mu) * rstd, n = xh * g[c] + be[c];
                    tb_put1(sm.narrow, p.kb, warp, c, n);
                    if (p.train && live) { xh_out[c] = xh; n_out[c] = n; }
                }
            }
            if (lane == 0 && live) (one ? s.rstd1 : s.rstd2)[l * s.sM + m0 + warp] = rstd;
            __syncthreads();
        }
        const bool wide_in = ph == 2;
        const int r8 = tb_up8(r);
        tb_product(st, p.mats[ph], wide_in ? sm.wide : sm.narrow, wide_in ? p.ka : p.kb, [&](int half, int, int n, const float (&v)[4]) {
            if (ph == 1) {
                if (n < f) {
                    const bool two = n + 1 < f;
                    const float x = sm.vec[5 * r + n], y = two ? sm.vec[5 * r + n + 1] : 0.f;
                    const float h[4] = {fmaxf(v[0] + x, 0.f), two ? fmaxf(v[1] + y, 0.f) : 0.f, fmaxf(v[2] + x, 0.f), two ? fmaxf(v[3] + y, 0.f) : 0.f};
                    tb_put2(sm.wide, p.ka, q, n, h[0], h[1]); tb_put2(sm.wide, p.ka, q + 8, n, h[2], h[3]);
                    if (p.train) {
                        float* out = s.hid + p.tail * s.sMf + (m0 + q) * f + n;
                        const bool even = (f & 1) == 0;
                        if (q < nt) tb_st2(out, h[0], h[1], two, even);
                        if (q + 8 < nt) tb_st2(out + 8LL * f, h[2], h[3], two, even);
                    }
                }
            } else if (ph < 3) {
                if (n < r) {
                    float* x = sm.rows + (half * TBF_T + q) * rs + n;
                    *reinterpret_cast<float2*>(x) = make_float2(v[0], v[1]);
                    *reinterpret_cast<float2*>(x + 8 * rs) = make_float2(v[2], v[3]);
                }
            } else {
                const int k = n >= 2 * r8 ? 2 : n >= r8 ? 1 : 0, c = n - k * r8;
                if (c < r) {
                    float* out = s.qkv + (3 * p.head + k) * s.sMr + (m0 + q) * r + c;
                    const bool even = (r & 1) == 0, two = c + 1 < r;
                    if (q < nt) tb_st2(out, v[0], v[1], two, even);
                    if (q + 8 < nt) tb_st2(out + 8LL * r, v[2], v[3], two, even);
                }
            }
        });
        if (ph < 3) __syncthreads();
    }
    if (p.tail >= 0 && p.head < 0) {
        // the last layer's a, which nothing in this launch reads
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            const int c = lane + 32 * i;
            const float* y = sm.rows + warp * rs + c;
            if (c < r && live)
                s.a[p.tail * p.u_stride + (m0 + warp) * r + c] = (p.mats[0].cut ? y[0] + y[TBF_T * rs] : y[0]) + (res[i] + sm.vec[4 * r + c]);
        }
    }
}

// Phases: 0 dn1 = [dq | dk | dv] [Wq | Wk | Wv]^T (of `tail`); 1 dhid = da W2^T, 2 dn2 = dpre W1^T, 3 do = dx1 Wo^T (of `head`).
template <int NR, int U, int CW>
__global__ void __launch_bounds__(TBF_THREADS) tb_bwd_kernel(const __grid_constant__ TbLayerParams p) {
    extern __shared__ __align__(128) unsigned char tb_sm[];
    const int b = blockIdx.x / p.tiles, t0 = (blockIdx.x - b * p.tiles) * TBF_T;
    const int S = p.S, r = p.r, f = p.f, H = p.H, dh = r / H, nt = min(TBF_T, S - t0), rs = p.rs;
    const long long m0 = (long long)b * S + t0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, q = lane >> 2, c2 = 2 * (lane & 3);
    const float scale = 1.f / sqrtf((float)dh);
    const int first = p.tail >= 0 ? 0 : 1, last = p.head >= 0 ? 4 : 1;
    const int hl = warp / p.nc, key0 = (warp - hl * p.nc) * 32, key_step = p.nc * 32;
    const bool live = warp < nt;                                // token `warp` is this warp's row
    const TbStacks& s = p.s;
    const TbSmem sm = tb_carve(tb_sm, (size_t)TBF_WARPS * U * TB_UNIT, p);
    if (p.tail >= 0) tb_vec_in(sm.vec, p.g1, r);
    if (p.head >= 0) tb_vec_in(sm.vec + r, p.g2, r);
    asm volatile("cp.async.commit_group;" ::: "memory");
    TbStream<U> st(p, tb_sm);
#pragma unroll 1
    for (int i = 0; i < U; ++i) st.issue();
    // What the forward pass left was final before the predecessor started, except for the first launch, whose predecessor triggers nothing.
    float xh[NR], up[NR], ap[NR], rstd = 0.f;                   // normalised row; u, a_prev
    float lm = 0.f;
    if (p.tail >= 0) {
        const int l = p.tail;
        tb_row_in(xh, s.xhat1 + l * s.sMr + (m0 + warp) * r, r, live);
        tb_row_in(up, p.u + l * p.u_stride + (m0 + warp) * r, r, live);
        tb_row_in(ap, s.a + (l - 1) * p.u_stride + (m0 + warp) * r, r, live && l > 0);
        rstd = live ? __ldg(s.rstd1 + l * s.sM + m0 + warp) : 0.f;
        lm = __ldg(p.lam + l);
    }
    tb_zero_terms(sm, p);
    pdl_wait();
    pdl_trigger();
    float res[NR];                                              // gradient past the norm: dx1 of `tail`, then da of `head`
    unsigned open = 0;                                          // hidden units of this warp's first eight tiles
    if (p.head >= 0) {
        const float* hid = s.hid + p.head * s.sMf + (m0 + q) * f;
        const int tiles = p.mats[1].tiles(warp);
        const bool even = (f & 1) == 0;
#pragma unroll 2
        for (int i = 0; i < min(8, tiles); ++i) {
            const int n = (warp + i * TBF_WARPS) * 8 + c2;
            const float2 h0 = q < nt ? tb_ld2(hid, n, f, even) : make_float2(0.f, 0.f), h1 = q + 8 < nt ? tb_ld2(hid + 8LL * f, n, f, even) : make_float2(0.f, 0.f);
            open |= (unsigned)((h0.x > 0.f ? 1 : 0) | (h0.y > 0.f ? 2 : 0) | (h1.x > 0.f ? 4 : 0) | (h1.y > 0.f ? 8 : 0)) << (4 * i);
        }
    }
    tb_vec_wait<U>();
    __syncthreads();
    if (p.tail >= 0) {
        const int l = p.tail;
        float* dqkv = s.dqkv + 3 * l * s.sMr + (m0 + warp) * r;
        float dq[NR];
        tb_row_in(dq, dqkv, r, live);
        tb_row_in(res, s.dx1 + l * s.sMr + (m0 + warp) * r, r, live);
        // dk[t] = scale sum_s dS[s][t] q[s],  dv[t] = sum_s P[s][t] do[s]   (own tokens t, all tokens s): 2 H heads of one mix
        int buf = 0;
#pragma unroll 1
        for (int hk0 = 0; hk0 < 2 * H; hk0 += p.hg) {
            const int hg = min(p.hg, 2 * H - hk0);
            const bool mine = hl < hg;
            const int hk = hk0 + hl, k = hk >= H, h = hk - k * H;
            const float* W = (k ? s.P + l * s.sP : s.dS[l & 1]) + ((long long)b * H + h) * S * S + t0;
            const float* X = (k ? s.dob[l & 1] : s.qkv + 3 * l * s.sMr) + (long long)b * S * r + h * dh;
#pragma unroll 1
            for (int n0 = 0; n0 < dh; n0 += 16, buf ^= 1) {
                float* share = sm.share + buf * TBF_WARPS * TB_SHARE;
                if (mine) {
                    float big[2][4] = {}, small[2][4] = {};
#pragma unroll 1
                    for (int w = 0; w < CW; ++w) {
                        const int s0 = key0 + w * key_step;
                        if (CW > 1 && s0 >= S) break;
                        float wt[2][8];
                        TbVals x;
                        if (s0 + 32 <= S && nt == TBF_T) {     // nothing to leave out
                            const float* w0 = W + (s0 + c2) * S + q;
#pragma unroll
                            for (int j = 0; j < 2; ++j)
#pragma unroll
                                for (int i = 0; i < 8; ++i) wt[j][i] = __ldg(w0 + (16 * j + (i & 1) + (i >> 2) * 8) * S + ((i >> 1) & 1) * 8);
                        } else
#pragma unroll
                        for (int j = 0; j < 2; ++j)
#pragma unroll
                            for (int i = 0; i < 8; ++i) {      // pairs (row q, q + 8) x (k c2, c2 + 8)
                                const int k_ = s0 + 16 * j + c2 + (i & 1) + (i >> 2) * 8, t = q + ((i >> 1) & 1) * 8;
                                wt[j][i] = k_ < S && t < nt ? __ldg(W + (long long)k_ * S + t) : 0.f;
                            }
                        tb_load_vals(x, X, r, s0, S, n0, dh);
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            TbA a;
                            tb_split_a(a, wt[j]);
                            tb_mix(big, small, a, x, j);
                        }
                    }
                    tb_share_put(share, big, small);
                }
                __syncthreads();
                tb_share_sum(share, p.nc, hg, n0, dh, [&](int i, int c, float v) {
                    const int k1 = hk0 + i >= H ? 2 : 1, at = (hk0 + i - (k1 - 1) * H) * dh + c;
                    if (k1 == 1) v *= scale;
                    tb_put1(sm.wide, p.ka, warp, k1 * r + at, v);
                    if (live) dqkv[k1 * s.sMr + at] = v;
                });
            }
        }
#pragma unroll
        for (int i = 0; i < NR; ++i)
            if (lane + 32 * i < r) tb_put1(sm.wide, p.ka, warp, lane + 32 * i, dq[i]);
    } else {
        // da_L: the same vector for every token of the sample
        tb_row_in(res, p.daL + (long long)b * r, r, live);
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            const int c = lane + 32 * i;
            if (c >= r) continue;
            sm.rows[(2 * TBF_T + warp) * rs + c] = res[i];
            tb_put1(sm.narrow, p.kb, warp, c, res[i]);
            if (live) s.da[p.head * s.sMr + (m0 + warp) * r + c] = res[i];
        }
    }
    __syncthreads();
#pragma unroll 1
    for (int ph = first; ph < last; ++ph) {
        const int l = ph ? p.head : p.tail;
        const long long o = l * s.sMr + (m0 + warp) * r;
        float* part = s.part + ((long long)l * gridDim.x + blockIdx.x) * p.s.part_w;
        if (ph == 1) {
            tb_col_sums(sm.rows + 2 * TBF_T * rs, rs, r, part + 4 * r);               // dc2: column sums of da
            tb_row_in(xh, s.xhat2 + o, r, live);
            rstd = live ? __ldg(s.rstd2 + l * s.sM + m0 + warp) : 0.f;
        }
        const bool wide_in = !(ph & 1);
        tb_product(st, p.mats[ph], wide_in ? sm.wide : sm.narrow, wide_in ? p.ka : p.kb, [&](int half, int i, int n, const float (&v)[4]) {
            if (ph == 1) {                             // dpre = dhid where the unit is open; dc1
                unsigned on = open >> (4 * i);
                if (i >= 8) {
                    const float* hid = s.hid + l * s.sMf + (m0 + q) * f;
                    const float2 z = make_float2(0.f, 0.f), h0 = q < nt ? tb_ld2(hid, n, f, false) : z, h1 = q + 8 < nt ? tb_ld2(hid + 8LL * f, n, f, false) : z;
                    on = (h0.x > 0.f ? 1 : 0) | (h0.y > 0.f ? 2 : 0) | (h1.x > 0.f ? 4 : 0) | (h1.y > 0.f ? 8 : 0);
                }
                const float y0 = on & 1 ? v[0] : 0.f, y1 = on & 2 ? v[1] : 0.f, y2 = on & 4 ? v[2] : 0.f, y3 = on & 8 ? v[3] : 0.f;
                const float s0 = tb_col_sum(y0, y2), s1 = tb_col_sum(y1, y3);
                if (n < f) {
                    const bool two = n + 1 < f, ev = (f & 1) == 0;
                    tb_put2(sm.wide, p.ka, q, n, y0, y1); tb_put2(sm.wide, p.ka, q + 8, n, y2, y3);
                    float* out = s.dpre + l * s.sMf + (m0 + q) * f + n;
                    if (q < nt) tb_st2(out, y0, y1, two, ev);
                    if (q + 8 < nt) tb_st2(out + 8LL * f, y2, y3, two, ev);
                    if (q == 0) { part[5 * r + n] = s0; if (two) part[5 * r + n + 1] = s1; }
                }
            } else if (n < r) {
                float* d = sm.rows + (((ph == 3 ? 2 : 0) + half) * TBF_T + q) * rs + n;
                *reinterpret_cast<float2*>(d) = make_float2(v[0], v[1]);
                *reinterpret_cast<float2*>(d + 8 * rs) = make_float2(v[2], v[3]);
            }
        });
        __syncthreads();
        if (ph & 1) continue;
        // LayerNorm backward: dx = (gradient past the norm) + (dxhat - mean(dxhat) - xhat mean(dxhat xhat)) rstd;
        // then dx1 of `head`, or the merge x = lambda u + (1 - lambda) a_prev of `tail`, whose da goes on to the layer below.
        // dn and dn xhat go where the products' halves were (a row is read and written by its own warp): their column sums are db and dg.
        const float* g = sm.vec + (ph ? r : 0);
        float* row = sm.rows + warp * rs;
        float dn[NR], s1 = 0.f, s2 = 0.f, acc = 0.f;
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            const int c = lane + 32 * i;
            dn[i] = 0.f;
            if (c < r) {
                if (live) dn[i] = p.mats[ph].cut ? row[c] + row[TBF_T * rs + c] : row[c];
                const float dxh = dn[i] * g[c];
                s1 += dxh;
                s2 = fmaf(dxh, xh[i], s2);
            }
        }
        s1 = warp_sum(s1) / (float)r;
        s2 = warp_sum(s2) / (float)r;
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            const int c = lane + 32 * i;
            if (c >= r) continue;
            float y = 0.f;
            if (live) {
                y = res[i] + (dn[i] * g[c] - s1 - xh[i] * s2) * rstd;
                if (ph) s.dx1[o + c] = y;
                else {
                    acc = fmaf(y, up[i] - ap[i], acc);
                    p.du[l * p.u_stride + (m0 + warp) * r + c] = lm * y;
                    y *= 1.f - lm;
                    if (p.head >= 0) s.da[p.head * s.sMr + (m0 + warp) * r + c] = y;
                }
            }
            row[c] = dn[i];
            row[TBF_T * rs + c] = dn[i] * xh[i];
            if (!ph) { row[2 * TBF_T * rs + c] = y; res[i] = y; }
            tb_put1(sm.narrow, p.kb, warp, c, y);
        }
        if (ph == 0) {
            acc = warp_sum(acc);
            if (lane == 0) sm.stat0[warp] = acc;
        }
        __syncthreads();
        tb_col_sums(sm.rows, rs, r, part + (ph ? 3 * r : r));
        tb_col_sums(sm.rows + TBF_T * rs, rs, r, part + (ph ? 2 * r : 0));
        if (ph == 0 && threadIdx.x == 0) {
            float tot = 0.f;
            for (int i = 0; i < TBF_WARPS; ++i) tot += sm.stat0[i];
            part[5 * r + f] = tot;
        }
    }
    if (p.head < 0) return;
    const int l = p.head;
    TbKeys keys;                       // v of the first 16 columns of a head, k as a mix operand, and P: operands of the second attention
    TbVals vals;
    float P[4][4];
    const bool even = ((dh | r) & 1) == 0, evenS = (S & 1) == 0;
    const float* qkv = s.qkv + 3 * l * s.sMr + (long long)b * S * r;
    const auto load_P = [&](int h, int k0) {
        const float* Pg = s.P + l * s.sP + (((long long)b * H + h) * S + t0 + q) * S;
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            const int key = k0 + n * 8 + c2;
            const float2 x = q < nt ? tb_ld2(Pg, key, S, evenS) : make_float2(0.f, 0.f), y = q + 8 < nt ? tb_ld2(Pg + 8LL * S, key, S, evenS) : make_float2(0.f, 0.f);
            P[n][0] = x.x; P[n][1] = x.y; P[n][2] = y.x; P[n][3] = y.y;
        }
    };
    // own queries: dP = do v^T, dS = P (dP - sum dP P), dq = scale dS k; do stands in two halves
    const float *do0 = sm.rows + 2 * TBF_T * rs, *do1 = do0 + TBF_T * rs;
    const bool halves = p.mats[3].cut;
    if (live)
        for (int c = lane; c < r; c += 32) s.dob[l & 1][(m0 + warp) * r + c] = halves ? do0[warp * rs + c] + do1[warp * rs + c] : do0[warp * rs + c];
    int buf = 0;
#pragma unroll 1
    for (int h0 = 0; h0 < H; h0 += p.hg) {
        const int hg = min(p.hg, H - h0), h = h0 + hl;
        const bool mine = hl < hg;
        float sc[CW][4][4] = {}, dot[2] = {};
        if (mine) {
            if (CW == 1) {
                tb_load_keys(keys, qkv + 2 * s.sMr + h * dh, r, key0, S, 0, dh, even);
                tb_load_vals(vals, qkv + s.sMr + h * dh, r, key0, S, 0, dh);
                load_P(h, key0);
            }
#pragma unroll 1
            for (int k = 0; k < dh; k += 16) {
                if (CW == 1 && k > 0) tb_load_keys(keys, qkv + 2 * s.sMr + h * dh, r, key0, S, k, dh, even);
                // columns past the head's are zeros on the v side; what do holds there is finite
                float v[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int c = k + c2 + (i & 1) + (i >> 2) * 8, at = (q + ((i >> 1) & 1) * 8) * rs + h * dh + c;
                    v[i] = c < dh ? (halves ? do0[at] + do1[at] : do0[at]) : 0.f;
                }
                TbA a;
                tb_split_a(a, v);
#pragma unroll
                for (int w = 0; w < CW; ++w) {
                    if (CW > 1) {
                        const int k0 = tb_round<CW>(key0, key_step, w);
                        if (k0 >= S) break;
                        tb_load_keys(keys, qkv + 2 * s.sMr + h * dh, r, k0, S, k, dh, even);
                    }
                    tb_scores(sc[w], a, keys);
                }
            }
#pragma unroll
            for (int w = 0; w < CW; ++w) {
                if (CW > 1) {
                    const int k0 = tb_round<CW>(key0, key_step, w);
                    if (k0 >= S) break;
                    load_P(h, k0);
                }
#pragma unroll
                for (int n = 0; n < 4; ++n)
#pragma unroll
                    for (int e = 0; e < 4; ++e) dot[e >> 1] = fmaf(sc[w][n][e], P[n][e], dot[e >> 1]);
            }
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            dot[i] = tb_quad_sum(dot[i]);
            if ((lane & 3) == 0) sm.stat0[warp * TBF_T + q + 8 * i] = dot[i];
        }
        __syncthreads();
        if (mine) {
            float* dS = s.dS[l & 1] + (((long long)b * H + h) * S + t0 + q) * S;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                dot[i] = 0.f;
                for (int c = 0; c < p.nc; ++c) dot[i] += sm.stat0[(hl * p.nc + c) * TBF_T + q + 8 * i];
            }
#pragma unroll
            for (int w = 0; w < CW; ++w) {
                const int k0 = tb_round<CW>(key0, key_step, w);
                if (CW > 1) {
                    if (k0 >= S) break;
                    load_P(h, k0);
                }
#pragma unroll
                for (int n = 0; n < 4; ++n) {
                    const int key = k0 + n * 8 + c2;
#pragma unroll
                    for (int e = 0; e < 4; ++e) sc[w][n][e] = key + (e & 1) < S ? P[n][e] * (sc[w][n][e] - dot[e >> 1]) : 0.f;
                    if (key < S) {
                        if (q < nt) tb_st2(dS + key, sc[w][n][0], sc[w][n][1], key + 1 < S, evenS);
                        if (q + 8 < nt) tb_st2(dS + 8LL * S + key, sc[w][n][2], sc[w][n][3], key + 1 < S, evenS);
                    }
                }
            }
        }
#pragma unroll 1
        for (int n0 = 0; n0 < dh; n0 += 16, buf ^= 1) {
            float* share = sm.share + buf * TBF_WARPS * TB_SHARE;
            if (mine) {
                float big[2][4] = {}, small[2][4] = {};
#pragma unroll
                for (int w = 0; w < CW; ++w) {
                    const int k0 = tb_round<CW>(key0, key_step, w);
                    if (CW > 1 && k0 >= S) break;
                    if (CW > 1 || n0 > 0) tb_load_vals(vals, qkv + s.sMr + h * dh, r, k0, S, n0, dh);
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        TbA a;
                        tb_frag_a(a, sc[w], k);
                        tb_mix(big, small, a, vals, k);
                    }
                }
                tb_share_put(share, big, small);
            }
            __syncthreads();
            if (live) {
                float* dq = s.dqkv + 3 * l * s.sMr + (m0 + warp) * r + h0 * dh;
                tb_share_sum(share, p.nc, hg, n0, dh, [&](int i, int c, float v) { dq[i * dh + c] = v * scale; });
            }
        }
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

// Variant of the kernels for a shape: NR by the width, as many units in flight as shared memory leaves room for, and three rounds of keys per warp for
// sequences beyond 16 warps of 32.  Up to 24 rounds two heads go at a time, three rounds to each of a head's warps; beyond, one.  In several rounds operands are fetched
// round by round (those of all three at a time spilled 0.4 to 2 KB per thread) and rounds past the sequence are left out; step at B = 4, L = 3, r = 64, 4 heads, S = 513 / 600 / 820:
// 1051 / 1886 / 1994 us with every round taken and all operands held, 503 / 830 / 1204 so (score rows in shared memory before: 858 / 1670 / 2122).
struct TbPlan {
    bool ok = false;
    int variant = 0, ka = 0, kb = 0, rs = 0, nc = 0, hg = 0;
    size_t smem = 0;
};
struct TbVariant { int nr, u, cw; const void *fwd, *bwd; };
#define TB_VARIANT(NR, U, CW) {NR, U, CW, (const void*)tb_fwd_kernel<NR, U, CW>, (const void*)tb_bwd_kernel<NR, U, CW>}
inline const TbVariant* tb_variants(int* n) {
    static const TbVariant v[] = {TB_VARIANT(2, 5, 1), TB_VARIANT(2, 3, 1), TB_VARIANT(3, 4, 1), TB_VARIANT(6, 3, 1), TB_VARIANT(6, 2, 1), TB_VARIANT(2, 5, 3), TB_VARIANT(3, 4, 3), TB_VARIANT(6, 2, 3)};
    *n = (int)(sizeof(v) / sizeof(v[0]));
    return v;
}
#undef TB_VARIANT

inline TbPlan tb_plan(int S, int r, int f, int H, int max_smem) {
    TbPlan pl;
    if (r > TBF_MAX_R || (long long)f * r > (1 << 22)) return pl;
    pl.ka = tb_up16(f > 3 * r ? f : 3 * r) + 8;
    pl.kb = tb_up16(r) + 8;
    pl.rs = (r + 31) / 32 * 32 + 8;            // = 8 mod 32: the fragments' pairs of four rows fall into different banks
    const int chunks = (S + 31) / 32;
    pl.nc = chunks <= TBF_WARPS ? chunks : chunks <= 3 * (TBF_WARPS / 2) ? (chunks + 2) / 3 : TBF_WARPS;
    pl.hg = TBF_WARPS / pl.nc;
    int n;
    const TbVariant* v = tb_variants(&n);
    for (int i = 0; i < n; ++i) {
        if (r > 32 * v[i].nr || chunks > pl.nc * v[i].cw) continue;
        pl.smem = (size_t)TBF_WARPS * v[i].u * TB_UNIT + tb_smem_fixed(pl.ka, pl.kb, pl.rs, r, f);
        if (pl.smem + 1024 > (size_t)max_smem) continue;
        if (smem_opt_in(v[i].fwd, pl.smem) != cudaSuccess || smem_opt_in(v[i].bwd, pl.smem) != cudaSuccess) { cudaGetLastError(); continue; }
        pl.variant = i;
        pl.ok = true;
        return pl;
    }
    return pl;
}

inline int tb_ctas(int B, int S) { return B * ((S + TBF_T - 1) / TBF_T); }

inline cudaError_t tb_layer_launch(const TbPlan& pl, TbLayerParams p, bool backward, cudaStream_t stream) {
    p.tiles = (p.S + TBF_T - 1) / TBF_T;
    p.nc = pl.nc; p.hg = pl.hg; p.ka = pl.ka; p.kb = pl.kb; p.rs = pl.rs;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    pdl_launch_config(&cfg, attr, dim3((unsigned)tb_ctas(p.B, p.S)), dim3(TBF_THREADS), pl.smem, stream);
    int n;
    const TbVariant& v = tb_variants(&n)[pl.variant];
    void* args[] = {&p};
    return cudaLaunchKernelExC(&cfg, backward ? v.bwd : v.fwd, args);
}

}  // namespace pac
