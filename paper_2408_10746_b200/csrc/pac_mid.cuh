// The part of a classifier-head train step that sits between the two passes over the
// cache, fused into one kernel, and the gradient finalisation (+ AdamW) fused into another.
//
// mid_cls_kernel: one thread-block cluster per batch sample.  From the down-projections
// u_l it runs the lambda-merge / adapter-body chain (Section IV-A) for all layers, pools a_L over
// the sample's tokens through distributed shared memory, evaluates head, loss and their
// gradients for the sample.  On the tensor-core path that is all: one gate byte per element and da_L
// per sample are what the second pass over the cache builds du_l from (see MidParams).  On the plain path
// it walks the chain backwards to emit du_l (fp32) and per-block partial sums of dlambda_l.
//
// All cross-thread sums use a fixed order, so results are bit-reproducible.
#pragma once
#include <cooperative_groups.h>
#include <type_traits>

#include "pac_common.cuh"
#include "pac_simt.cuh"
#include "pac_tensor.cuh"

namespace pac {

namespace cg = cooperative_groups;

struct MidParams {
    const int* ids; long long N; const int* labels;
    int L, S, d, r, C, B;
    int G;                      // cluster size: CTAs per sample
    int Sg;                     // tokens per CTA = ceil(S / G)
    int dg;                     // head columns per CTA = ceil(d / G)
    int train;
    int scratch;                // floats of block-local reduction scratch
    int aL_floats;              // floats of the a_L tile in shared memory (Sg * r; 0 when the chain ran elsewhere)
    int layers_per_cta;         // one-kernel forward: layers whose down-projections each CTA of the cluster computes
    int early_ids;              // 1: no kernel ahead of this one in the stream writes the ids (device memory)
    int* ids_copy;              // one-kernel forward: device copy of the batch's ids for the finalisation, or null
    // STATE_POOLED: what the down-projection kernel's epilogue left behind
    const float* pool_part;     // [B][n_pool_parts][r] token sums of a_L per token group
    int n_pool_parts;
    const float* u; long long lstride;
    const float* lam; const float* W_up; const float* W_head; const float* b_head; const float* hbar;
    void* du;                   // [L][max_rows][r] bf16 or fp32
    float* pooled_a;            // [B][r]   mean_s a_L, for the gradient finalisation
    float* dlogits;             // [B][C]
    float* loss_b;              // [B]
    float* lam_part;            // [L][B*G]
    float* logits_out;          // [B][C] (train: scratch copy; eval: caller's buffer)
    unsigned* status;
    // What the second pass needs of the reverse chain (tensor-core path).  da_L is the same vector for every token of a sample and a
    // gate multiplies by exactly 1 or 0, so dz_l[t][j] = cprod_l * (gates l .. L of (t, j) all open ? da_L[j] : 0) with
    // cprod_l = prod_{l' > l} (1 - lambda_l'): one byte per element and one vector per sample describe it for all layers.
    uint8_t* tc;                // [max_rows][r]: 1 + the highest layer whose gate is closed (0: none)
    bf16* da16; long long da_stride;      // [2][max_batch][r]: da_L in two bf16 terms
    float* coef;                // [L]: lambda_l cprod_l, the factor of dW_down^l
    const float* prodW;         // optional [r][C]: W_up W_head, formed once per step by head_matrix_kernel (else per CTA)
};

constexpr int MID_MAX_C = 32;
constexpr size_t MID_SMEM_BUDGET = 220 * 1024;    // dynamic shared memory the fused kernel may use
constexpr int MID_MAX_L = 32;     // ReLU masks of all layers live in one 32-bit word per element

__device__ __forceinline__ void cp_async_4(void* smem_dst, const void* gsrc) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(smem_dst)), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_16(void* smem_dst, const void* gsrc) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem_dst)), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait_group() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Shared-memory chain state, [layer][thread] 16-byte groups: group c4 of a CTA's token s_local sits at group
// c4 ^ state_swizzle(s_local, groups per token) of the token's row, so that rows written one per lane (an
// accumulator row per thread) and rows read one group per lane are both free of bank conflicts.
__device__ __forceinline__ int state_swizzle(int s_local, int groups_per_tok) {
    const int m = (groups_per_tok & (groups_per_tok - 1)) ? 0 : min(groups_per_tok, 8) - 1;
    return s_local & m;
}

// Where u_l comes from.
enum {
    STATE_SMEM = 0,      // this CTA's shared memory, prefetched from the global u buffer with cp.async
    STATE_GLOBAL = 1,    // the global u buffer, a few layers in flight per thread
    STATE_POOLED = 2     // nowhere: the forward chain ran in the down-projection kernel's epilogue, which left token sums of
                         // a_L per token group and the gates
};

// The small per-CTA vectors of the head computation, carved from one shared-memory region.
struct MidShared {
    float *aL, *colsum, *prodq, *prod, *plq, *daL, *py, *lg, *lam_s, *cprod, *wh_s, *lred;
};
__device__ __forceinline__ MidShared mid_carve(float* sm, const MidParams& p) {
    MidShared h;
    const size_t rc = (size_t)(p.r + 1) * p.C;
    h.aL = sm;                                        // [Sg][r]   a_L of this CTA's tokens
    h.colsum = h.aL + (size_t)p.aL_floats;            // [r]       exchanged through DSMEM
    h.prodq = h.colsum + p.r;                         // [r+1][C]  this CTA's partial head products, exchanged
    h.prod = h.prodq + rc;                            // [r+1][C]  their sum over the cluster
    h.plq = h.prod + rc;                              // [MID_MAX_C] this CTA's tokens' share of S * (mean_s a_L)(W_up W_head), exchanged
    h.daL = h.plq + MID_MAX_C;                        // [r]
    h.py = h.daL + p.r;                               // [dg]  slice of mean_s h_L
    h.lg = h.py + p.dg;                               // [MID_MAX_C] logits, then dlogits
    h.lam_s = h.lg + MID_MAX_C;                       // [MID_MAX_L]
    h.cprod = h.lam_s + MID_MAX_L;                    // [MID_MAX_L] prod_{l' > l} (1 - lambda_l')
    h.wh_s = h.cprod + MID_MAX_L;                     // [dg][C] slice of W_head
    h.lred = h.wh_s + (size_t)p.dg * p.C;             // [nwarps][MID_MAX_L]; also [parts][r] scratch
    return h;
}

// cp.async requests for the head operands of CTA rank q (hbar slice of sample `id`, W_head slice)
// and plain loads of lambda, issued by threads t0 .. t0 + nthr - 1 of the block.
__device__ __forceinline__ void mid_prefetch_head(const MidParams& p, const MidShared& h, int q, long long id, int t, int nthr) {
    const int k0 = q * p.dg, kn = max(0, min(p.dg, p.d - k0));
    for (int kk = t; kk < kn; kk += nthr) cp_async_4(h.py + kk, p.hbar + id * p.d + k0 + kk);
    for (int e = t; e < kn * p.C; e += nthr) cp_async_4(h.wh_s + e, p.W_head + (long long)k0 * p.C + e);
    for (int l = t; l < MID_MAX_L; l += nthr) h.lam_s[l] = l < p.L ? p.lam[l] : 0.f;
    if (t == nthr - 1) {
        // prod_{l' > l} (1 - lambda_l'), multiplied in the order the reverse recursion meets the layers
        float c = 1.f;
        for (int l = p.L - 1; l >= 0; --l) {
            h.cprod[l] = c;
            c *= 1.f - p.lam[l];
        }
    }
}

// The head is linear in mean_s a_L, so both directions through it reduce to one small matrix:
//   logits = b_head + hbar W_head + (mean_s a_L) (W_up W_head),      d loss / d mean_s a_L = (W_up W_head) dlogits.
// Each CTA forms the products over its own slice of the hidden width (operands already in shared
// memory):  prodq[j][c] = sum_k W_up[j][k] W_head[k][c]  (j < r),  prodq[r][c] = sum_k hbar[k] W_head[k][c];
// the slices are added across the cluster afterwards.  Called by nw whole warps, w = the caller's
// index among them; none of it depends on u, so it can run while u is still being produced.
__device__ __forceinline__ void mid_head_products(const MidParams& p, const MidShared& h, int q, int w, int nw, int lane) {
    const int k0 = q * p.dg, kn = max(0, min(p.dg, p.d - k0));
    // with the sample-independent rows already formed for the whole step only the hbar row is left
    for (int j = p.prodW ? p.r + w : w; j <= p.r; j += nw) {
        for (int c0 = 0; c0 < p.C; c0 += 4) {
            float acc[4] = {0.f, 0.f, 0.f, 0.f};
            for (int kk = lane; kk < kn; kk += 32) {
                const float a = j == p.r ? h.py[kk] : p.W_up[(long long)j * p.d + k0 + kk];     // each W_up element is read once
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (c0 + c < p.C) acc[c] = fmaf(a, h.wh_s[kk * p.C + c0 + c], acc[c]);
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float v = warp_sum(acc[c]);
                if (lane == 0 && c0 + c < p.C) h.prodq[j * p.C + c0 + c] = v;
            }
        }
    }
}
// prodW[j][c] = sum_k W_up[j][k] W_head[k][c], one warp per entry, k in lane order then a fixed shuffle tree.  The
// product does not depend on the sample: the stand-alone head kernels take it from here instead of forming
// it again in every CTA (the one-launch forward forms it on warps that would otherwise idle under the stream).
// behind: the kernel ahead lets this one start only when everything ahead of itself is complete, so the parameters are final; it runs beside that kernel and ends after it, so
// that whoever waits for this one finds both done (smallest blocking fp32 step 50.7 -> 48.4 us, fp32 step at T5-Base widths 91.6 -> 86.3, T5-Large step 436 -> 430).
// Otherwise the first block stores the step's ids, where they travel as an argument (the kernel ahead does so then).
constexpr int HEAD_MATRIX_THREADS = 256;
static_assert(ARG_IDS <= HEAD_MATRIX_THREADS, "the first block stores the ids, one per thread");
__global__ void __launch_bounds__(HEAD_MATRIX_THREADS) head_matrix_kernel(const float* __restrict__ W_up, const float* __restrict__ W_head, int d, int r,
                                                          int C, float* __restrict__ prodW, int behind, const __grid_constant__ ArgIds arg, int* __restrict__ ids) {
    // not behind: the parameters come from the optimizer update before this kernel, and the ids of the step before may be read until then; the down-projections are let in after
    // the wait, too: their CTAs beside the kernels before this one, which still run then, cost more than their start hides (d = 768, S = 151, B = 2, L = 8: step 35.2 -> 33.8 us, three
    // of an epoch 101.0 -> 97.2)
    if (!behind) pdl_wait();
    pdl_trigger();
    if (blockIdx.x == 0 && (int)threadIdx.x < arg.n) ids[threadIdx.x] = arg.v[threadIdx.x];
    const int e = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (e < r * C) {
        const int j = e / C, c = e - j * C;
        float acc = 0.f;
#pragma unroll 8
        for (int k = lane; k < d; k += 32) acc = fmaf(__ldg(W_up + (long long)j * d + k), __ldg(W_head + (long long)k * C + c), acc);
        acc = warp_sum(acc);
        if (lane == 0) prodW[e] = acc;
    }
    if (behind) pdl_wait();
}

// Classifier head of the plain path, one CTA per sample: token mean of a_L, logits from the C-vectors (the head's matrix
// product prodW = W_up W_head stands in for the d-wide ones), loss, dlogits and da_L / S.  What the parameters' gradients
// need of the d-wide vectors the finalisation kernel rebuilds.  (The kernel that formed mean_s y and g per sample
// read W_up twice per sample: 93 us at T5-Base widths against 9.)
// Dynamic shared memory: 9 r + C + 32 floats.
__global__ void __launch_bounds__(256) plain_head_kernel(const float* __restrict__ aL, const float* __restrict__ hbar, const int* __restrict__ ids,
                                                         long long N, const int* __restrict__ labels, const float* __restrict__ prodW,
                                                         const float* __restrict__ W_head, const float* __restrict__ b_head, int B, int S, int d, int r,
                                                         int C, int train, float* __restrict__ pooled_a, float* __restrict__ logits_out,
                                                         float* __restrict__ loss_b, float* __restrict__ dlogits, float* __restrict__ daL, unsigned* status) {
    extern __shared__ float hsm[];
    float *pa = hsm, *part = pa + r, *lg = part + 8 * r, *red = lg + C;
    const int b = blockIdx.x, t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const long long id = safe_id(ids, b, N, t == 0 ? status : nullptr);
    for (int c = lane; c < r; c += 32) {
        const float* col = aL + (long long)b * S * r + c;
        float acc = 0.f;
#pragma unroll 8
        for (int s = warp; s < S; s += 8) acc += __ldg(col + (long long)s * r);
        part[warp * r + c] = acc;
    }
    __syncthreads();
    for (int c = t; c < r; c += 256) {
        float acc = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) acc += part[w * r + c];
        pa[c] = acc / (float)S;
        if (train) pooled_a[(long long)b * r + c] = pa[c];
    }
    __syncthreads();
    for (int c = 0; c < C; ++c) {
        float acc = 0.f;
#pragma unroll 4
        for (int k = t; k < d; k += 256) acc = fmaf(__ldg(hbar + id * d + k), __ldg(W_head + (long long)k * C + c), acc);
        for (int j = t; j < r; j += 256) acc = fmaf(pa[j], __ldg(prodW + j * C + c), acc);
        acc = warp_sum(acc);
        if (lane == 0) red[warp] = acc;
        __syncthreads();
        if (t == 0) {
            float v = 0.f;
#pragma unroll
            for (int w = 0; w < 8; ++w) v += red[w];
            lg[c] = v + b_head[c];
        }
        __syncthreads();
    }
    for (int c = t; c < C; c += 256) logits_out[(long long)b * C + c] = lg[c];
    if (!train) return;
    float mx = -INFINITY, se = 0.f;
    for (int c = 0; c < C; ++c) mx = fmaxf(mx, lg[c]);
    for (int c = 0; c < C; ++c) se += expf(lg[c] - mx);
    const int label = labels[id];
    if (t == 0) loss_b[b] = mx + logf(se) - lg[label];
    __syncthreads();
    for (int c = t; c < C; c += 256) {
        const float g = (expf(lg[c] - mx) / se - (c == label ? 1.f : 0.f)) / (float)B;
        lg[c] = g;
        dlogits[(long long)b * C + c] = g;
    }
    __syncthreads();
    for (int j = t; j < r; j += 256) {
        float acc = 0.f;
        for (int c = 0; c < C; ++c) acc = fmaf(__ldg(prodW + j * C + c), lg[c], acc);
        daL[(long long)b * r + j] = acc / (float)S;
    }
}

// After a cluster-wide barrier behind mid_head_products: the sum over the cluster, in rank order.  The
// last row also takes the classifier bias, so the head needs no global load of its own later on.
__device__ __forceinline__ void mid_sum_products(const MidParams& p, const MidShared& h, cg::cluster_group& cluster, int t, int nthr) {
    for (int e = t; e < (p.r + 1) * p.C; e += nthr) {
        if (p.prodW && e < p.r * p.C) { h.prod[e] = p.prodW[e]; continue; }
        float acc = 0.f;
        for (int g = 0; g < p.G; ++g) acc += cluster.map_shared_rank(h.prodq, g)[e];
        if (e >= p.r * p.C) acc = p.b_head[e - p.r * p.C] + acc;      // b_head + (mean_s h_L) W_head
        h.prod[e] = acc;
    }
}

// Everything after the down-projections for one sample, executed by one CTA (rank q) of the
// sample's cluster.  GPT: 4-column groups per thread.  u_s: STATE_SMEM: [L][GPT][nt] float4 state;
// products_ready: the caller has already prefetched the head
// operands, run mid_head_products and passed a cluster barrier.  n_landed > 0 (STATE_SMEM): the state of the
// top n_landed layers is not fetched from the u buffer: the cluster's CTAs write it into u_s directly and the
// mbarrier land_bar (shared-memory address, phase 0) completes when all of it has arrived.
template <int ACT, typename DU, int GPT, int STATE>
__device__ __forceinline__ void mid_body(const MidParams& p, cg::cluster_group& cluster, float4* u_s, const MidShared& h,
                                         bool products_ready, long long known_id = -1, int n_landed = 0, uint32_t land_bar = 0,
                                         volatile int* abort_flag = nullptr) {
    constexpr int LT = MID_MAX_L;
    const int q = (int)cluster.block_rank();
    const int b = blockIdx.x / p.G;
    const int t = threadIdx.x, nt = blockDim.x;
    const int r = p.r, L = p.L, C = p.C;
    const int warp = t >> 5, lane = t & 31, nwarps = nt >> 5;
    float *aL = h.aL, *colsum = h.colsum, *prod = h.prod, *plq = h.plq,
          *lg = h.lg, *lam_s = h.lam_s, *lred = h.lred, *cprod = h.cprod, *daL = h.daL;

    const int groups_per_tok = r >> 2;
    int s_local[GPT], j4[GPT], ts[GPT];                   // ts: this thread's slot in a layer's plane of the shared-memory state
    bool live[GPT];
    long long base[GPT];
#pragma unroll
    for (int g = 0; g < GPT; ++g) {
        const int gi = t + g * nt;                       // this thread's g-th group of 4 adapter columns
        s_local[g] = gi / groups_per_tok;
        j4[g] = (gi - s_local[g] * groups_per_tok) << 2;
        const int s = q * p.Sg + s_local[g];
        live[g] = s_local[g] < p.Sg && s < p.S;
        base[g] = ((long long)b * p.S + s) * r + j4[g];
        ts[g] = t ^ state_swizzle(s_local[g], groups_per_tok);
    }
    constexpr bool GATES = sizeof(DU) == 2;              // tensor-core path: gates and da_L go out instead of du (see MidParams)
    DU* du = reinterpret_cast<DU*>(p.du);
    // layer l of group g: read u, keep / fetch the reverse-pass state (fp32 du only)
    auto load_u = [&](int l, int g) -> float4 {
        if constexpr (STATE == STATE_SMEM) return u_s[((size_t)l * GPT + g) * nt + ts[g]];
        else return *reinterpret_cast<const float4*>(p.u + (long long)l * p.lstride + base[g]);
    };
    auto store_w = [&](int l, int g, const float* wv) {
        if constexpr (STATE == STATE_SMEM) {
            u_s[((size_t)l * GPT + g) * nt + ts[g]] = make_float4(wv[0], wv[1], wv[2], wv[3]);
        } else {
            *reinterpret_cast<float4*>(du + (long long)l * p.lstride + base[g]) = make_float4(wv[0], wv[1], wv[2], wv[3]);
        }
    };
    auto load_w = [&](int l, int g) -> float4 {
        if constexpr (STATE == STATE_SMEM) {
            return u_s[((size_t)l * GPT + g) * nt + ts[g]];
        } else {
            return *reinterpret_cast<const float4*>(du + (long long)l * p.lstride + base[g]);
        }
    };
    const long long id = known_id >= 0 ? known_id : safe_id(p.ids, b, p.N, (t == 0 && q == 0) ? p.status : nullptr);
    if (!products_ready) mid_prefetch_head(p, h, q, id, t, nt);
    cp_async_commit();                                                          // group: head operands
    if constexpr (STATE == STATE_SMEM) {
#pragma unroll
        for (int g = 0; g < GPT; ++g)
            if (live[g])
                for (int l = 0; l < L - n_landed; ++l) cp_async_16(u_s + ((size_t)l * GPT + g) * nt + ts[g], p.u + (long long)l * p.lstride + base[g]);
    }
    cp_async_commit();                                                          // group: u
    const int label = p.train ? p.labels[id] : 0;                               // fetched long before the head needs it
    if (!products_ready) {
        cp_async_wait_group<1>();                                               // head operands have landed ...
        __syncthreads();                                                        // ... those of every thread
        mid_head_products(p, h, q, warp, nwarps, lane);                         // overlaps the u copies in flight
        cluster.sync();
    }
    mid_sum_products(p, h, cluster, t, nt);              // read after the block barriers below
    cp_async_wait_group<0>();                            // own u values have landed

    // ---- forward chain over each group of 4 adapter columns of one token.  The slot that held
    // u_l is overwritten with u_l - a_{l-1} (= d z_l / d lambda_l) for the reverse pass; the ReLU
    // masks stay in registers (bit l of mask[g][e]).  Layers are taken four at a time so that the
    // loads of a batch are in flight together; the outer loops stay rolled (every CTA runs this
    // code once, so small code beats unrolled code).
    unsigned mask[GPT][4];                               // fp32 du: bit l = gate of layer l open; gates: 1 + highest closed layer
    float ap[GPT][4];
    bool landed = false;
    // column sums of a_L straight from registers when a warp holds whole tokens (one group per thread, 4, 8 or 16 groups per token)
    const bool shuffle_sums = GPT == 1 && STATE != STATE_POOLED && groups_per_tok <= 32 && (32 % groups_per_tok) == 0;
#pragma unroll
    for (int g = 0; g < GPT; ++g) {
#pragma unroll
        for (int e = 0; e < 4; ++e) { mask[g][e] = 0u; ap[g][e] = 0.f; }      // a_0 = 0
        if constexpr (STATE == STATE_POOLED) continue;       // the chain ran in the down-projection kernel's epilogue
        if (live[g]) {
#pragma unroll 1
            for (int l0 = 0; l0 < L; l0 += 4) {
                if (n_landed > 0 && !landed && l0 + 4 > L - n_landed) {
                    mbar_wait(land_bar, 0, abort_flag, p.status);      // the handed-over layers have arrived
                    landed = true;
                }
                float4 uq[4];
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (l0 + i < L) uq[i] = load_u(l0 + i, g);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int l = l0 + i;
                    if (l < L) {
                        const float uv[4] = {uq[i].x, uq[i].y, uq[i].z, uq[i].w};
                        const float lm = lam_s[l];
                        float wv[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float z = lm * uv[e] + (1.f - lm) * ap[g][e];
                            if constexpr (!GATES) wv[e] = uv[e] - ap[g][e];
                            if (ACT == PAC_ACT_RELU) {
                                const bool on = z > 0.f;
                                if constexpr (GATES) mask[g][e] = on ? mask[g][e] : (unsigned)(l + 1);
                                else mask[g][e] |= (on ? 1u : 0u) << l;
                                ap[g][e] = on ? z : 0.f;
                            } else {
                                ap[g][e] = z;
                            }
                        }
                        if constexpr (!GATES) store_w(l, g, wv);
                    }
                }
            }
            if constexpr (GATES)
                if (p.train) *reinterpret_cast<uint32_t*>(p.tc + base[g]) = mask[g][0] | (mask[g][1] << 8) | (mask[g][2] << 16) | (mask[g][3] << 24);
        }
        if (!shuffle_sums && s_local[g] < p.Sg) {
#pragma unroll
            for (int e = 0; e < 4; ++e) aL[(size_t)s_local[g] * r + j4[g] + e] = live[g] ? ap[g][e] : 0.f;
        }
    }
    if (shuffle_sums) {
        // the lanes of a warp that hold the same four columns (one per token of the warp) add up by shuffles, in a
        // fixed order; one partial sum per warp and column goes to shared memory
        float v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = live[0] ? ap[0][e] : 0.f;
        for (int off = groups_per_tok; off < 32; off <<= 1)
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] += __shfl_xor_sync(0xffffffffu, v[e], off);
        if (lane < groups_per_tok)
#pragma unroll
            for (int e = 0; e < 4; ++e) lred[warp * r + (lane << 2) + e] = v[e];
    }
    __syncthreads();
    // column sums over this CTA's tokens: `parts` partial sums per column over contiguous token
    // ranges, then added in range order
    {
        int parts = 1;
        if (shuffle_sums) {
            parts = nwarps;
        } else if constexpr (STATE == STATE_POOLED) {
            // token-group sums from the down-projection kernel; CTA q of the cluster takes groups q, q + G, ...
            if (t < r) {
                float acc = 0.f;
                for (int pp = q; pp < p.n_pool_parts; pp += p.G) acc += p.pool_part[((long long)b * p.n_pool_parts + pp) * r + t];
                lred[t] = acc;
            }
        } else {
            parts = max(1, min(nt / r, p.Sg));
            const int per = (p.Sg + parts - 1) / parts;
            if (t < parts * r) {
                const int j = t % r, part = t / r;
                float acc = 0.f;
                for (int sl = part * per; sl < min(p.Sg, (part + 1) * per); ++sl) acc += aL[(size_t)sl * r + j];
                lred[part * r + j] = acc;
            }
        }
        if (!shuffle_sums) __syncthreads();
        if (t < r) {
            float acc = 0.f;
            for (int part = 0; part < parts; ++part) acc += lred[part * r + t];
            colsum[t] = acc;
        }
        // What the head needs of a_L is its token sum times the head's product matrix; this CTA's tokens'
        // share of that, plq[c] = sum_j colsum[j] prod[j][c], is formed here (warp c), so that only C numbers
        // per CTA cross the cluster on the way to the logits.
        for (int c = warp; c < C; c += nwarps) {
            float pl = 0.f;
            for (int j = lane; j < r; j += 32) {
                float cs = 0.f;
                for (int part = 0; part < parts; ++part) cs += lred[part * r + j];
                pl = fmaf(cs, prod[j * C + c], pl);
            }
            pl = warp_sum(pl);
            if (lane == 0) plq[c] = pl;
        }
    }
    cluster.sync();
    // ---- head, by ONE warp: logits from the cluster's C-vectors, loss, dlogits, d loss / d a_L; everybody
    // else waits at one block barrier.  The same in every CTA of the cluster.  A second warp of the first
    // CTA forms mean_s a_L for the gradient finalisation meanwhile.
    if (warp == 0) {
        float mylogit = -INFINITY;                        // lane c holds logit c (C <= 32)
        if (lane < C) {
            float acc = 0.f;
            for (int g = 0; g < p.G; ++g) acc += cluster.map_shared_rank(plq, g)[lane];
            mylogit = prod[r * C + lane] + acc / (float)p.S;      // b_head + (mean_s h_L) W_head + (mean_s a_L)(W_up W_head)
            if (q == 0) p.logits_out[(long long)b * C + lane] = mylogit;
        }
        if (p.train) {
            const float mx = warp_max(mylogit);
            const float ex = lane < C ? expf(mylogit - mx) : 0.f;
            const float se = warp_sum(ex);
            const float lab_logit = __shfl_sync(0xffffffffu, mylogit, label);
            if (lane == 0 && q == 0) p.loss_b[b] = mx + logf(se) - lab_logit;
            const float my = lane < C ? (ex / se - (lane == label ? 1.f : 0.f)) / (float)p.B : 0.f;     // dlogits
            if (lane < C) {
                lg[lane] = my;
                if (q == 0) p.dlogits[(long long)b * C + lane] = my;
            }
            __syncwarp();
            for (int j = lane; j < r; j += 32) {
                float acc = 0.f;
                for (int c = 0; c < C; ++c) acc = fmaf(prod[j * C + c], lg[c], acc);
                const float v = acc / (float)p.S;         // da_L, the same for every token of the sample
                if constexpr (GATES) {
                    if (q == 0) {
                        const bf16 hi = __float2bfloat16(v);
                        p.da16[(long long)b * r + j] = hi;
                        p.da16[p.da_stride + (long long)b * r + j] = __float2bfloat16(v - __bfloat162float(hi));
                    }
                } else {
                    daL[j] = v;
                }
            }
        }
    } else if (warp == 1 && q == 0 && p.train) {
        for (int j = lane; j < r; j += 32) {
            float acc = 0.f;
            for (int g = 0; g < p.G; ++g) acc += cluster.map_shared_rank(colsum, g)[j];
            p.pooled_a[(long long)b * r + j] = acc / (float)p.S;      // mean_s a_L
        }
    } else if (GATES && warp == 2 && blockIdx.x == 0 && p.train) {
        for (int l = lane; l < L; l += 32) p.coef[l] = lam_s[l] * cprod[l];
    }
    // That was this CTA's last access to a peer's shared memory: say so now and wait, at the very end, only
    // for the peers to have said the same (a CTA must not exit while a peer may still read its memory).
    cluster.barrier_arrive();
    if constexpr (GATES) {
        cluster.barrier_wait();                           // peers may still be reading this CTA's shared memory
        return;
    } else {
    __syncthreads();
    if (!p.train) {
        cluster.barrier_wait();
        return;
    }

    // ---- reverse chain, in closed form.  da_L is the same vector for every token of the sample and a ReLU
    // gate only ever multiplies by exactly 1 or 0, so for an element whose gates l..L are all open
    //     dz_l = da_L[j] * prod_{l' > l} (1 - lambda_l'),   du_l = lambda_l dz_l,
    // and 0 as soon as one gate at or above l is closed (cprod[l] holds the product, formed once per CTA in
    // layer order).  No value depends on another layer's, so four layers are in flight at a time, the warp
    // sums of this thread's shares of dlambda_l = sum gate * dz_l * (u_l - a_{l-1}) included. ----
    float daLr[GPT][4];
#pragma unroll
    for (int g = 0; g < GPT; ++g)
#pragma unroll
        for (int e = 0; e < 4; ++e) daLr[g][e] = live[g] ? daL[j4[g] + e] : 0.f;
    int top_closed[GPT][4];                               // highest layer whose gate is closed (-1: none): open from there up only
#pragma unroll
    for (int g = 0; g < GPT; ++g)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const unsigned closed = (ACT == PAC_ACT_RELU) ? (~mask[g][e] & (L >= 32 ? 0xffffffffu : ((1u << L) - 1u))) : 0u;
            top_closed[g][e] = 31 - __clz(closed);        // __clz(0) = 32
        }
    // one layer of one group: du_l out, this thread's share of dlambda_l added to `part`
    auto reverse_step = [&](int l, int g, const float4& w4, float& part, float cp, float lm, DU* dst) {
        const float wv[4] = {w4.x, w4.y, w4.z, w4.w};
        float dv[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const bool open = l > top_closed[g][e];            // gates l .. L all open
            const float dz = open ? daLr[g][e] * cp : 0.f;
            part = fmaf(dz, wv[e], part);
            dv[e] = lm * dz;                                   // du_l
        }
        *reinterpret_cast<float4*>(dst) = make_float4(dv[0], dv[1], dv[2], dv[3]);
    };
    {
        // layers per batch: about four state loads in flight per thread whatever the number of groups it owns
        constexpr int LB = GPT >= 4 ? 1 : 4 / GPT;
        DU* dstp[GPT];                                        // running pointers into du, one layer down per step
#pragma unroll
        for (int g = 0; g < GPT; ++g) dstp[g] = du + (long long)(L - 1) * p.lstride + base[g];
#pragma unroll 1
        for (int l0 = L - 1; l0 >= 0; l0 -= LB) {
            float4 wq[LB][GPT];
#pragma unroll
            for (int i = 0; i < LB; ++i)
#pragma unroll
                for (int g = 0; g < GPT; ++g)
                    if (l0 - i >= 0 && live[g]) wq[i][g] = load_w(l0 - i, g);
            float part[LB];
#pragma unroll
            for (int i = 0; i < LB; ++i) {
                part[i] = 0.f;
                if (l0 - i >= 0) {
                    const float cp = cprod[l0 - i], lm = lam_s[l0 - i];
#pragma unroll
                    for (int g = 0; g < GPT; ++g) {
                        if (live[g]) reverse_step(l0 - i, g, wq[i][g], part[i], cp, lm, dstp[g]);
                        dstp[g] -= p.lstride;
                    }
                }
            }
            // this warp's shares of dlambda of the batch's layers: independent shuffle trees
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int i = 0; i < LB; ++i) part[i] += __shfl_xor_sync(0xffffffffu, part[i], o);
            if (lane == 0)
#pragma unroll
                for (int i = 0; i < LB; ++i)
                    if (l0 - i >= 0) lred[warp * LT + (l0 - i)] = part[i];
        }
    }
    __syncthreads();
    if (t < L) {
        float acc = 0.f;
        for (int wv = 0; wv < nwarps; ++wv) acc += lred[wv * LT + t];
        p.lam_part[(long long)t * (p.B * p.G) + blockIdx.x] = acc;
    }
    cluster.barrier_wait();                               // keep shared memory alive until every peer has read it
    }
}

// The stand-alone kernel: u comes from the global buffer written by the down-projection kernel.
template <int ACT, typename DU, int GPT, int STATE>
__global__ void __launch_bounds__(512, STATE == STATE_SMEM ? 1 : 2) mid_cls_kernel(MidParams p) {
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ float4 sm4[];
    float4* u_s = sm4;                           // [L][GPT][nt] each thread's own u values, later u_l - a_{l-1}
    float* sm = reinterpret_cast<float*>(sm4 + (STATE == STATE_SMEM ? (size_t)p.L * GPT * blockDim.x
                                               : 0));
    const MidShared h = mid_carve(sm, p);
    pdl_trigger();
    pdl_wait();             // u (or the token sums) comes from the kernel before this one
    mid_body<ACT, DU, GPT, STATE>(p, cluster, u_s, h, false);
}

// ---------------------------------------------------------------------------
// Gradient finalisation for the classifier head:
//   W_down : sum of the second pass's row splits (split order), on the tensor-core path times the layer's factor; or already final
//   lambda : from <D_l, W_down^l> (lambda_grad), on the plain path the sum of per-block partials (block order); or already final
//   W_up   : pooled_a^T g        W_head : pooled_y^T dlogits        b_head : sum_b dlogits
// plus the mean loss.  With adam != 0 the AdamW update of the same element follows at once.
// ---------------------------------------------------------------------------
struct FinalizeParams {
    ParamLayout lay;
    int B, d, r, C, L;
    const float* dw_part; int splits; long long dw_elems;     // splits < 1: W_down gradient already in grads
    // Tensor-core path: dw_part holds D_l = h_l^T (open_l daL) (see MidParams), dW_down^l = coef[l] D_l, and P_l = <D_l, W_down^l>
    // is all that dlambda needs (see lambda_grad): every W_down block leaves its share in dot_part [L][wd_per_layer], block 0 waits for
    // them and updates lambda.
    const float* coef; unsigned long long* dot_part;
    const float* lam_part; int lam_blocks;                   // null: the lambda gradients are already in grads
    const float *pooled_a, *dlogits, *loss_b;                // per-sample vectors the forward half left: mean_s a_L, dlogits, loss
    const float* hbar; const int* ids; long long N;          // token mean of the last cached layer, per cache sample; the batch's ids
    const float* params_in;                                  // the parameters the forward half used (W_up, W_head are read)
    float* grads; float* loss_out;
    int wd_blocks, wd_per_layer, wd_layer_elems;             // blocks that handle W_down, 4 elements per thread, within one layer each
    int rest_blocks;                                         // blocks that handle the head side: FIN_KB columns of the hidden width each
    // AdamW
    int adam;
    float *params, *m, *v;
    pac_adamw hp; float bc1, bc2;
    float grad_scale;                                        // factor on every gradient entering the fused update
    WdShadow wdT;                                            // bf16 terms of W_down (p may be null)
    // Device status words: when a bounded wait of this step's passes or of an earlier step has run out, the gradients
    // are not trustworthy, so nothing is written to the gradients, parameters or moments.  The wait for the shares of P_l in this
    // kernel itself is different: should it run out, lambda stays as it is while blocks that had left their share have
    // updated what they own, and the caller goes back to a checkpoint.
    unsigned* status;
};

constexpr int FIN_KB = 4;       // hidden-width columns per head-side block of the finalisation kernel

// dlambda_l = sum dz_l (u_l - a_{l-1}) without u or a.  With dz_l = cprod_l open_l daL and u_l = h_l W_l the first half is cprod_l P_l,
// P_l = <D_l, W_l>; and where gates l .. L are open, a_{l-1} = sum over i < l with gates i .. l-1 open of
// lambda_i prod_{i < l' < l} (1 - lambda_l') u_i, so the second half is sum_{i<l} lambda_i (prod_{l' > i, l' != l} (1 - lambda_l')) P_i.
__device__ __forceinline__ float lambda_grad(const float* lam, const float* P, int L, int l) {
    float e = 1.f;
    for (int k = L - 1; k > l; --k) e *= 1.f - lam[k];
    float g = e * P[l];
    for (int i = l - 1; i >= 0; --i) {
        g -= lam[i] * e * P[i];
        e *= 1.f - lam[i];
    }
    return g;
}
// Four consecutive elements of sum_j part[j], j in order, requested three splits at a time.
__device__ __forceinline__ float4 sum_parts4(const float* __restrict__ part, int splits, long long stride) {
    float4 a = *reinterpret_cast<const float4*>(part);
    for (int j = 1; j < splits; j += 3) {
        float4 q[3];
#pragma unroll
        for (int k = 0; k < 3; ++k)
            if (j + k < splits) q[k] = *reinterpret_cast<const float4*>(part + (j + k) * stride);
#pragma unroll
        for (int k = 0; k < 3; ++k)
            if (j + k < splits) { a.x += q[k].x; a.y += q[k].y; a.z += q[k].z; a.w += q[k].w; }
    }
    return a;
}
// Shares of P_l travel as (value, 1) in one 64-bit word, so that a block leaves its share with a plain store: no fence, no counter, and the
// block's slot is free a memory round trip earlier.  The collecting block puts the words back to zero.
// Blocks of 256 threads: the block's sum of `dot` goes to dot_part[blk].
__device__ __forceinline__ void publish_dot(float dot, unsigned long long* __restrict__ dot_part, int blk) {
    __shared__ float red[8];
    dot = warp_sum(dot);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = dot;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) t += red[w];
        const unsigned long long word = 1ull << 32 | __float_as_uint(t);
        asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(dot_part + blk), "l"(word) : "memory");
    }
}
constexpr int DOT_POLLS = 1 << 24;      // bound on a wait for one share, about ten seconds: another stream's kernel may hold the other blocks back
// P_l from the blocks' shares, warp per layer, and lambda, into shared memory: one block of 256 threads that runs beside those that publish
// (it holds one slot, so they all get to run).  False if a share did not arrive; *ok_sh is shared memory.
__device__ __forceinline__ bool collect_dots(const float* lam, unsigned long long* dot_part, int per_layer, int L, float* lam_s, float* dot_s,
                                             int* ok_sh, unsigned* status, int polls = DOT_POLLS) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) *ok_sh = 1;
    for (int l = threadIdx.x; l < L; l += 256) lam_s[l] = lam[l];
    __syncthreads();
    for (int l = warp; l < L; l += 8) {
        float acc = 0.f;
        for (int k = lane; k < per_layer; k += 32) {
            unsigned long long* at = dot_part + (long long)l * per_layer + k;
            unsigned long long word = 0;
            for (int n = 0; n < polls; ++n) {
                asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(word) : "l"(at) : "memory");
                if (word != 0ull || *reinterpret_cast<volatile int*>(ok_sh) == 0) break;
            }
            if (word == 0ull && atomicExch(ok_sh, 0) && status) atomicAdd(&status[ST_TIMEOUT], 1u);
            *at = 0ull;
            acc += __uint_as_float((unsigned)word);
        }
        acc = warp_sum(acc);
        if (lane == 0) dot_s[l] = acc;
    }
    __syncthreads();
    return *ok_sh != 0;
}
// Self-test: collects two layers of three shares with a short limit; the caller has left one share out.  result[0] = 1 if the wait was reported
// as run out.
__global__ void __launch_bounds__(256) selftest_collect_kernel(const float* lam, unsigned long long* dot_part, unsigned* status, unsigned* result) {
    __shared__ float lam_s[2], dot_s[2];
    __shared__ int ok;
    const bool all = collect_dots(lam, dot_part, 3, 2, lam_s, dot_s, &ok, status, 64);
    if (threadIdx.x == 0) result[0] = all ? 0u : 1u;
}
// The gradients of W_down (four elements per thread, blocks within one layer each) and lambda (the first block) from the second pass's
// partial sums where no finalisation kernel follows (L <= 256).
__global__ void __launch_bounds__(256) gated_grads_kernel(const float* __restrict__ part, int splits, long long n, int dr, int per_layer, int L,
                                                          const float* __restrict__ w, const float* __restrict__ lam, const float* __restrict__ coef,
                                                          unsigned long long* __restrict__ dot_part, float* __restrict__ gW, float* __restrict__ glam, unsigned* status) {
    if (blockIdx.x == 0) {
        __shared__ float lam_s[256], dot_s[256];
        __shared__ int ok;
        if (collect_dots(lam, dot_part, per_layer, L, lam_s, dot_s, &ok, status))
            for (int k = threadIdx.x; k < L; k += 256) glam[k] = lambda_grad(lam_s, dot_s, L, k);
        return;
    }
    const int blk = blockIdx.x - 1, l = blk / per_layer, o = ((blk - l * per_layer) * 256 + threadIdx.x) * 4;
    const long long i = (long long)l * dr + o;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f), p = a;
    if (o < dr) {
        p = *reinterpret_cast<const float4*>(w + i);
        a = sum_parts4(part + i, splits, n);
    }
    publish_dot(fmaf(a.x, p.x, fmaf(a.y, p.y, fmaf(a.z, p.z, a.w * p.w))), dot_part, blk);
    if (o < dr) {
        const float c = coef[l];
        *reinterpret_cast<float4*>(gW + i) = make_float4(a.x * c, a.y * c, a.z * c, a.w * c);
    }
}
// lambda_l with its moments, requested before its gradient is known.
struct LambdaState { float p, m, v; };
__device__ __forceinline__ LambdaState lambda_load(const FinalizeParams& f, int l) {
    const long long i = f.lay.lam + l;
    return f.adam ? LambdaState{f.params[i], f.m[i], f.v[i]} : LambdaState{0.f, 0.f, 0.f};
}
__device__ __forceinline__ void lambda_update(const FinalizeParams& f, int l, float g, LambdaState s) {
    const long long i = f.lay.lam + l;
    f.grads[i] = g;
    if (!f.adam) return;
    f.params[i] = adamw_math(s.p, s.m, s.v, g * f.grad_scale, false, f.hp, f.bc1, f.bc2);
    f.m[i] = s.m;
    f.v[i] = s.v;
}

// (five blocks per SM: 48 registers, no spills; T5-Base step 51.0 -> 50.3 us against the 63 registers of an open bound)
__global__ void __launch_bounds__(256, 5) finalize_cls_kernel(FinalizeParams f) {
    pdl_trigger();
    const ParamLayout& lay = f.lay;
    // W_down blocks fetch the old parameter and moments while the predecessor still runs: nothing since the
    // previous finalisation writes them, and that one was over before the predecessor's own predecessor
    // finished (every kernel of a step lets its successor start only after its own wait has returned or
    // does not touch these arrays before its wait)
    // block 0 takes dlambda and the loss (scheduled first, so it runs at once), the next rest_blocks blocks the
    // head parameters, the remaining wd_blocks blocks W_down
    const int blk = (int)blockIdx.x - 1;
    const int l_wd = blk >= f.rest_blocks ? (blk - f.rest_blocks) / f.wd_per_layer : 0;
    const int o_wd = ((blk - f.rest_blocks - l_wd * f.wd_per_layer) * (int)blockDim.x + (int)threadIdx.x) * 4;      // inside the layer
    const long long i_wd = (long long)l_wd * f.wd_layer_elems + o_wd;
    const bool wd_thread = blk >= f.rest_blocks && o_wd < f.wd_layer_elems;
    float4 p4 = make_float4(0.f, 0.f, 0.f, 0.f), m4 = p4, v4 = p4;
    if (wd_thread && f.coef && !f.adam) p4 = *reinterpret_cast<const float4*>(f.params_in + i_wd);
    if (wd_thread && f.adam) {
        p4 = *reinterpret_cast<const float4*>(f.params + i_wd);
        m4 = *reinterpret_cast<const float4*>(f.m + i_wd);
        v4 = *reinterpret_cast<const float4*>(f.v + i_wd);
    }
    // Block 0: the mean loss needs only what the forward half left behind, which is complete whenever this kernel runs
    // (see above), so a loss that goes straight to host memory is on its way long before the step ends.
    // Set by a wait that ran out in this step's forward half or in any earlier step since the last
    // pac_sync (the forward half has completed whenever this kernel runs); a wait that runs out in this
    // step's second pass is seen by the W_down blocks behind their own wait below.
    const bool dead = status_timed_out(f.status);
    if (blk < 0) {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
        if (dead && f.adam && threadIdx.x == 0) atomicAdd(&f.status[ST_SKIPPED_STEPS], 1u);
        if (warp == nw - 1) {
            float acc = 0.f;
            for (int b = lane; b < f.B; b += 32) acc += f.loss_b[b];
            acc = warp_sum(acc);
            if (lane == 0) *f.loss_out = acc / (float)f.B;
        }
        // dlambda where it does not come from the W_down blocks: warp per layer, lanes over its partial sums, fixed shuffle order
        for (int l = warp; l < f.L && !f.coef && !dead; l += nw) {
            float acc = 0.f;
            const LambdaState old = lambda_load(f, l);
            if (f.lam_part) {
#pragma unroll 4
                for (int k = lane; k < f.lam_blocks; k += 32) acc += f.lam_part[(long long)l * f.lam_blocks + k];
                acc = warp_sum(acc);
            } else {
                acc = f.grads[lay.lam + l];
            }
            if (lane == 0) lambda_update(f, l, acc, old);
        }
        if (!f.coef) return;
        const LambdaState old = lambda_load(f, min((int)threadIdx.x, f.L - 1));
        pdl_wait();
        if (status_timed_out(f.status)) return;          // (as in the W_down blocks: final behind the wait)
        __shared__ float lam_s[MID_MAX_L], dot_s[MID_MAX_L];
        __shared__ int ok;
        if (collect_dots(f.params_in + lay.lam, f.dot_part, f.wd_per_layer, f.L, lam_s, dot_s, &ok, f.status) && threadIdx.x < f.L)
            lambda_update(f, threadIdx.x, lambda_grad(lam_s, dot_s, f.L, threadIdx.x), old);
        return;
    }
    if (blk < f.rest_blocks) {
        // Head-side parameters: like block 0 these blocks need only what the forward half left behind, so
        // they finish (and make room for the W_down blocks) while the second pass still runs.  A block owns
        // FIN_KB columns k of the hidden width: W_up[:, k] and W_head[k, :] (the last block also b_head).
        // It first rebuilds, for its columns, the two per-sample vectors of the head's backward,
        //     g[b][k]  = d loss / d mean_s y = sum_c W_head[k][c] dlogits[b][c]
        //     py[b][k] = mean_s y = hbar[id_b][k] + sum_j pooled_a[b][j] W_up[j][k]
        // from the OLD values of exactly the parameters it owns (read before any of them is updated), then
        //     dW_up[j][k] = sum_b pooled_a[b][j] g[b][k],   dW_head[k][c] = sum_b py[b][k] dlogits[b][c].
        extern __shared__ float fsm[];
        float* g_s = fsm;                                    // [B][FIN_KB]
        float* py_s = g_s + (size_t)f.B * FIN_KB;            // [B][FIN_KB]
        float* wup_s = py_s + (size_t)f.B * FIN_KB;          // [r][FIN_KB]   old W_up[:, k0..]
        float* wh_s = wup_s + (size_t)f.r * FIN_KB;          // [FIN_KB][C]   old W_head[k0.., :]
        const int k0 = blk * FIN_KB, kn = min(FIN_KB, f.d - k0), t = threadIdx.x, nt = blockDim.x;
        const float* W_up = f.params_in + lay.w_up;
        const float* W_head = f.params_in + lay.w_head;
        if (dead) return;
        for (int e = t; e < f.r * FIN_KB; e += nt) {
            const int j = e / FIN_KB, kk = e - j * FIN_KB;
            wup_s[e] = kk < kn ? W_up[(long long)j * f.d + k0 + kk] : 0.f;
        }
        for (int e = t; e < FIN_KB * f.C; e += nt) {
            const int kk = e / f.C;
            wh_s[e] = kk < kn ? W_head[(long long)k0 * f.C + e] : 0.f;
        }
        __syncthreads();
        for (int e = t; e < f.B * FIN_KB; e += nt) {
            const int b = e / FIN_KB, kk = e - b * FIN_KB;
            float gv = 0.f, acc = 0.f;
            for (int c = 0; c < f.C; ++c) gv = fmaf(wh_s[kk * f.C + c], f.dlogits[(long long)b * f.C + c], gv);
            for (int j = 0; j < f.r; ++j) acc = fmaf(f.pooled_a[(long long)b * f.r + j], wup_s[j * FIN_KB + kk], acc);
            const long long id = safe_id(f.ids, b, f.N, nullptr);
            g_s[e] = gv;
            py_s[e] = kk < kn ? f.hbar[id * f.d + k0 + kk] + acc : 0.f;
        }
        __syncthreads();
        const int n_up = f.r * FIN_KB, n_head = FIN_KB * f.C;
        const bool last = blk == f.rest_blocks - 1;
        for (int e = t; e < n_up + n_head + (last ? f.C : 0); e += nt) {
            long long i;
            float g = 0.f;
            if (e < n_up) {
                const int j = e / FIN_KB, kk = e - j * FIN_KB;
                if (kk >= kn) continue;
                i = lay.w_up + (long long)j * f.d + k0 + kk;
#pragma unroll 8
                for (int b = 0; b < f.B; ++b) g = fmaf(f.pooled_a[(long long)b * f.r + j], g_s[b * FIN_KB + kk], g);
            } else if (e < n_up + n_head) {
                const int kk = (e - n_up) / f.C, c = (e - n_up) - kk * f.C;
                if (kk >= kn) continue;
                i = lay.w_head + (long long)(k0 + kk) * f.C + c;
#pragma unroll 8
                for (int b = 0; b < f.B; ++b) g = fmaf(py_s[b * FIN_KB + kk], f.dlogits[(long long)b * f.C + c], g);
            } else {
                const int c = e - n_up - n_head;
                i = lay.b_head + c;
                for (int b = 0; b < f.B; ++b) g += f.dlogits[(long long)b * f.C + c];
            }
            f.grads[i] = g;
            if (f.adam) adamw_element(f.params, f.m, f.v, i, g * f.grad_scale, f.lay, f.hp, f.bc1, f.bc2, f.wdT, f.d, f.r);
        }
        return;
    }
    const float cf = f.coef ? f.coef[l_wd] : 1.f;
    pdl_wait();
    // W_down block, four consecutive elements per thread
    const long long i = i_wd;
    const unsigned late = f.status ? *reinterpret_cast<const volatile unsigned*>(f.status + ST_TIMEOUT) : 0u;     // (on its way beside the sums)
    float4 g4 = make_float4(0.f, 0.f, 0.f, 0.f);
    if (wd_thread) g4 = f.splits >= 1 ? sum_parts4(f.dw_part + i, f.splits, f.dw_elems) : *reinterpret_cast<const float4*>(f.grads + i);
    if (late) return;
    if (f.coef) publish_dot(fmaf(g4.x, p4.x, fmaf(g4.y, p4.y, fmaf(g4.z, p4.z, g4.w * p4.w))), f.dot_part, blk - f.rest_blocks);
    if (wd_thread) {
        if (f.splits >= 1) {
            g4.x *= cf; g4.y *= cf; g4.z *= cf; g4.w *= cf;
            *reinterpret_cast<float4*>(f.grads + i) = g4;
        }
        if (f.adam) {
            g4.x *= f.grad_scale; g4.y *= f.grad_scale; g4.z *= f.grad_scale; g4.w *= f.grad_scale;
            adamw_w_down4_loaded(f.params, f.m, f.v, i, l_wd, p4, m4, v4, g4, f.hp, f.bc1, f.bc2, f.wdT, f.d, f.r);
        }
    }
}

// Shape test and launch geometry of the fused kernel: G CTAs per sample, one 4-column
// group per thread, chain state in shared memory.
struct MidPlan {
    bool ok = false;
    int G = 1, Sg = 0, dg = 0, threads = 0, scratch = 0;
    int gpt = 1, smem_state = 1;      // 4-column groups per thread; u through shared memory, or from global memory as it is used
    int aL_floats = 0;                // a_L tile in shared memory (0: the chain ran in the down-projection kernel)
    size_t smem = 0;
};

// Shared-memory floats the kernel needs besides the chain state and the W_up slice.
inline size_t mid_base_floats(const Dims& dm, int Sg, int dg, int th, int* scratch_out, bool with_aL = true) {
    const int nw = th / 32;
    int scratch = nw * MID_MAX_L;
    const int parts = th / dm.r > 0 ? th / dm.r : 1;
    if (parts * dm.r > scratch) scratch = parts * dm.r;
    if (nw * dm.r > scratch) scratch = nw * dm.r;              // one partial column sum per warp
    *scratch_out = scratch;
    return (with_aL ? (size_t)Sg * dm.r : 0) + 2 * (size_t)dm.r + MID_MAX_C + 2 * (size_t)(dm.r + 1) * dm.C + (size_t)dg + MID_MAX_C + MID_MAX_L + scratch +
           (size_t)dg * dm.C + MID_MAX_L + 4;
}

inline MidPlan mid_plan(const Dims& dm) {
    MidPlan mp;
    if (dm.r % 4 != 0 || dm.C > MID_MAX_C || dm.L > MID_MAX_L) return mp;
    const size_t budget = MID_SMEM_BUDGET / sizeof(float);
    // first choice: one group per thread, chain state in shared memory, fewest CTAs per sample
    for (int G = 1; G <= 8; G *= 2) {
        const int Sg = (dm.S + G - 1) / G, dg = (dm.d + G - 1) / G;
        const long long need = (long long)Sg * (dm.r / 4);
        if (need > 512) continue;
        int th = (int)((need + 31) / 32 * 32);
        if (th < 128) th = 128;
        int scratch;
        size_t floats = mid_base_floats(dm, Sg, dg, th, &scratch) + 4 * (size_t)dm.L * th;
        if (floats > budget) continue;
        mp.G = G; mp.Sg = Sg; mp.dg = dg; mp.threads = th; mp.scratch = scratch; mp.gpt = 1; mp.smem_state = 1;
        mp.smem = sizeof(float) * floats;
        mp.ok = true;
        return mp;
    }
    // otherwise: 8 CTAs per sample, up to 4 groups per thread, u read from global memory
    {
        const int G = 8, Sg = (dm.S + G - 1) / G, dg = (dm.d + G - 1) / G;
        const long long need = (long long)Sg * (dm.r / 4);
        if (need > 4 * 512) return mp;
        const int gpt = need <= 512 ? 1 : need <= 1024 ? 2 : 4;
        int th = (int)(((need + gpt - 1) / gpt + 31) / 32 * 32);
        if (th < 128) th = 128;
        int scratch;
        size_t floats = mid_base_floats(dm, Sg, dg, th, &scratch);
        if (floats > budget) return mp;
        mp.G = G; mp.Sg = Sg; mp.dg = dg; mp.threads = th; mp.scratch = scratch; mp.gpt = gpt; mp.smem_state = 0;
        mp.smem = sizeof(float) * floats;
        mp.ok = true;
    }
    return mp;
}

// Geometry behind a kernel that already ran the chain: only the head is left, one CTA per sample.
inline MidPlan mid_plan_pooled(const Dims& dm) {
    MidPlan mp;
    if (dm.r % 4 != 0 || dm.r > 256 || dm.C > MID_MAX_C || dm.L > MID_MAX_L) return mp;
    int scratch;
    const size_t floats = mid_base_floats(dm, dm.S, dm.d, 256, &scratch, false);
    if (floats > MID_SMEM_BUDGET / sizeof(float)) return mp;
    mp.G = 1; mp.Sg = dm.S; mp.dg = dm.d; mp.threads = 256; mp.scratch = scratch; mp.gpt = 1; mp.smem_state = 0;
    mp.smem = sizeof(float) * floats;
    mp.ok = true;
    return mp;
}

template <int ACT, typename DU, int GPT, int STATE>
inline cudaError_t mid_launch_one(const MidPlan& mp, const MidParams& p, cudaStream_t stream) {
    {
        cudaError_t e = smem_opt_in((const void*)mid_cls_kernel<ACT, DU, GPT, STATE>, MID_SMEM_BUDGET);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(p.B * mp.G), 1, 1);
    cfg.blockDim = dim3((unsigned)mp.threads, 1, 1);
    cfg.dynamicSmemBytes = mp.smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)mp.G;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, mid_cls_kernel<ACT, DU, GPT, STATE>, p);
}

template <int ACT, typename DU>
inline cudaError_t mid_launch_shape(const MidPlan& mp, const MidParams& p, cudaStream_t stream) {
    if (mp.smem_state) return mid_launch_one<ACT, DU, 1, STATE_SMEM>(mp, p, stream);
    switch (mp.gpt) {
        case 1: return mid_launch_one<ACT, DU, 1, STATE_GLOBAL>(mp, p, stream);
        case 2: return mid_launch_one<ACT, DU, 2, STATE_GLOBAL>(mp, p, stream);
        default: return mid_launch_one<ACT, DU, 4, STATE_GLOBAL>(mp, p, stream);
    }
}

// The same kernel behind a down-projection kernel that already ran the forward chain.
inline cudaError_t mid_launch_pooled(const MidPlan& mp, const MidParams& p, int act, cudaStream_t stream) {
    return act == PAC_ACT_RELU ? mid_launch_one<PAC_ACT_RELU, bf16, 1, STATE_POOLED>(mp, p, stream)
                               : mid_launch_one<PAC_ACT_IDENTITY, bf16, 1, STATE_POOLED>(mp, p, stream);
}

// gates: the tensor-core path's form (see MidParams), else du in fp32.
inline cudaError_t mid_launch(const MidPlan& mp, const MidParams& p, int act, bool gates, cudaStream_t stream) {
    if (act == PAC_ACT_RELU)
        return gates ? mid_launch_shape<PAC_ACT_RELU, bf16>(mp, p, stream) : mid_launch_shape<PAC_ACT_RELU, float>(mp, p, stream);
    return gates ? mid_launch_shape<PAC_ACT_IDENTITY, bf16>(mp, p, stream) : mid_launch_shape<PAC_ACT_IDENTITY, float>(mp, p, stream);
}

}  // namespace pac
