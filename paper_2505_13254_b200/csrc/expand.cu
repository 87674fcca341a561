// hs_expand_init / hs_expand_level / hs_rerank: the draft tree of Sec. 2.2 grown and reranked on the device.
//
// The candidate tree of a sequence lives in caller-owned arrays of `cap` slots in creation order (candidate 0 = the
// root, parents precede children).  One expansion level (one CTA per sequence): every frontier node gets the k most
// likely tokens of its draft row as children - the Top-K tokens and logits of that row and its log-sum-exp are
// what hs_entropy_quantify writes -, a child's value is its parent's plus its log-confidence (ln V_i = sum ln c_j),
// and the k children with the largest value (ties: created first) become the next frontier.  Reranking (one CTA
// per sequence): the N candidates with the largest value, compacted in creation order with parents re-indexed: a
// topologically ordered tree ready for the verification calls.  A level ranks its children by counting, the reranking
// finds the N-th largest value by binary search; compaction by warp ballots and a prefix sum over the warps.
#include <math_constants.h>

#include "expand_child.h"
#include "hs_common.cuh"
#include "hs_layout.h"
#include "hs_ptx.cuh"

#define EX_THREADS 256
#define EX_MAX_CAP 2048        // candidates per sequence the reranking holds in shared memory

__global__ void expand_init_kernel(hs_expand_state st) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    pdl_launch_dependents();
    pdl_wait();
    if (b >= st.batch) return;
    const size_t o = (size_t)b * st.cap;
    st.n_cand[b] = 1;
    st.parent[o] = -1; st.token[o] = -1; st.depth[o] = 0; st.logc[o] = 0.f; st.score[o] = 0.f;
    st.frontier[(size_t)b * st.top_k] = 0;
    st.n_frontier[b] = 1;
    st.status[b] = HS_OK;
}

// Two round trips to global memory: the sequence's numbers and the frontier, then the row statistics of the frontier's children
// and their parents' values.  The rank among the new children reads four values per shared-memory access.
__global__ void __launch_bounds__(EX_THREADS) expand_level_kernel(hs_expand_state st, const float* topk_val,
                                                                  const int* topk_idx, const float* row_lse, int K) {
    __shared__ __align__(16) float s_S[HS_MAX_TOPK * HS_MAX_TOPK];
    const int b = blockIdx.x, tid = threadIdx.x;
    const int k = st.top_k;
    const size_t o = (size_t)b * st.cap;
    pdl_launch_dependents();
    pdl_wait();                                    // the row statistics come from the kernel ahead
    const int status = st.status[b], n0 = st.n_cand[b], nf = st.n_frontier[b];
    const int par = tid < k * k ? st.frontier[(size_t)b * k + tid / k] : -1;      // (slots past the frontier hold older candidates: not used)
    if (status != HS_OK) return;
    const int nnew = nf * k;
    if (n0 + nnew > st.cap) {                      // the arrays cannot take another level
        if (tid == 0) st.status[b] = HS_ERR_SHAPE;
        return;
    }
    int tok = -1, dep = 0;
    float lc = 0.f;
    float S = __int_as_float(0x7fc00000);          // (NaN: compares false, ranks nobody)
    if (load_child(tid, b, k, nf, K, topk_val, topk_idx, row_lse, tok, lc)) {
        S = st.score[o + par] + lc;
        dep = st.depth[o + par] + 1;
    }
    s_S[tid] = S;
    if (__syncthreads_or(tid < nnew && tok < 0)) { // a row had fewer than k finite logits
        if (tid == 0) st.status[b] = HS_ERR_BAD_TREE;
        return;
    }
    if (tid < nnew) {
        const int c = n0 + tid;
        st.parent[o + c] = par; st.token[o + c] = tok; st.depth[o + c] = dep;
        st.logc[o + c] = lc; st.score[o + c] = S;
        int rank = 0;                              // by (value descending, creation order)
        const float4* S4 = reinterpret_cast<const float4*>(s_S);
        for (int q = 0; q < nnew; q += 4) {
            const float4 v = S4[q >> 2];
            rank += (v.x > S || (v.x == S && q < tid)) + (v.y > S || (v.y == S && q + 1 < tid)) +
                    (v.z > S || (v.z == S && q + 2 < tid)) + (v.w > S || (v.w == S && q + 3 < tid));
        }
        if (rank < k) st.frontier[(size_t)b * k + rank] = c;
    }
    if (tid == 0) {
        st.n_cand[b] = n0 + nnew;
        st.n_frontier[b] = min(k, nnew);
    }
}

struct RerankParams {
    hs_expand_state st;
    const int* n_top;      // [B] or NULL
    int n_default;
    int* node_off;         // [B+1]
    int* parent;
    int* token;
    int* cand_id;
    int* depth;
};

__device__ __forceinline__ int rerank_count(const RerankParams& p, int b) {
    if (p.st.status[b] != HS_OK) return 0;
    const int want = p.n_top ? p.n_top[b] : p.n_default;
    return max(0, min(want, p.st.n_cand[b]));
}

// The Top-N of up to 2048 candidates: the N-th largest value by binary search over its 32 order bits (each thread holds two
// candidates, a step is one counting barrier), ties to the candidate created first.  Ranking by counting compared every
// pair (711 candidates: 28.9 us alone, this: 10.1 us).
#define RR_THREADS 1024
__global__ void __launch_bounds__(RR_THREADS) rerank_kernel(const RerankParams p) {
    __shared__ short s_new[EX_MAX_CAP];
    __shared__ int s_warp[2][RR_THREADS / 32];
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthr = blockDim.x, nw = nthr >> 5;
    pdl_launch_dependents();
    pdl_wait();
    const size_t o = (size_t)b * p.st.cap;
    const int n = p.st.status[b] == HS_OK ? min(p.st.n_cand[b], EX_MAX_CAP) : 0;
    const int want = rerank_count(p, b);
    // candidates tid and tid + nthr; 0 = none (no value has order bits 0)
    unsigned int key[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int c = h * nthr + tid;
        key[h] = c < n ? float_order_bits(p.st.score[o + c] + 0.f) : 0u;
    }
    // offset of this sequence's tree: the trees ahead of it hold min(N, candidates) nodes each
    int part = 0;
    for (int bb = tid; bb < b; bb += nthr) part += rerank_count(p, bb);
    part = __reduce_add_sync(HS_FULL_MASK, part);
    if (lane == 0) s_warp[0][warp] = part;
    __syncthreads();
    const int off = __reduce_add_sync(HS_FULL_MASK, lane < nw ? s_warp[0][lane] : 0);
    // numbers of candidates whose flag is set ahead of this thread's two, in creation order, and in all
    auto ahead = [&](bool f0, bool f1, int (&a)[2]) -> int {
        const unsigned int b0 = __ballot_sync(HS_FULL_MASK, f0), b1 = __ballot_sync(HS_FULL_MASK, f1);
        __syncthreads();                           // (s_warp may still be read)
        if (lane == 0) { s_warp[0][warp] = __popc(b0); s_warp[1][warp] = __popc(b1); }
        __syncthreads();
        const int c0 = lane < nw ? s_warp[0][lane] : 0, c1 = lane < nw ? s_warp[1][lane] : 0;
        const int t0 = __reduce_add_sync(HS_FULL_MASK, c0), t1 = __reduce_add_sync(HS_FULL_MASK, c1);
        const unsigned int below = (1u << lane) - 1u;
        a[0] = __reduce_add_sync(HS_FULL_MASK, lane < warp ? c0 : 0) + __popc(b0 & below);
        a[1] = t0 + __reduce_add_sync(HS_FULL_MASK, lane < warp ? c1 : 0) + __popc(b1 & below);
        return t0 + t1;
    };
    // T = the want-th largest key: the largest T with at least `want` keys >= T
    unsigned int T = 0u;
    if (want < n) {
        for (int bit = 31; bit >= 0; --bit) {
            const unsigned int t = T | (1u << bit);
            int cnt = __syncthreads_count(key[0] >= t);
            if (n > nthr) cnt += __syncthreads_count(key[1] >= t);
            if (cnt >= want) T = t;
        }
    }
    int e[2], above = __syncthreads_count(key[0] > T);
    if (n > nthr) above += __syncthreads_count(key[1] > T);
    ahead(key[0] == T && key[0] != 0u, key[1] == T && key[1] != 0u, e);      // of the ties at T the first want - above stay
    const bool k0 = key[0] > T || (key[0] == T && key[0] != 0u && e[0] < want - above);
    const bool k1 = key[1] > T || (key[1] == T && key[1] != 0u && e[1] < want - above);
    int pos[2];
    ahead(k0, k1, pos);
    if (tid < n) s_new[tid] = k0 ? (short)pos[0] : (short)-1;
    if (nthr + tid < n) s_new[nthr + tid] = k1 ? (short)pos[1] : (short)-1;
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int c = h * nthr + tid;
        if (!(h ? k1 : k0)) continue;
        const int i = pos[h], par = p.st.parent[o + c];
        p.parent[off + i] = par >= 0 ? (int)s_new[par] : -1;   // (the kept set is closed under ancestors)
        p.token[off + i] = p.st.token[o + c];
        p.cand_id[off + i] = c;
        p.depth[off + i] = p.st.depth[o + c];
    }
    if (tid == 0) {
        p.node_off[b] = off;
        if (b == p.st.batch - 1) p.node_off[p.st.batch] = off + want;
    }
}

static bool state_ok(const hs_expand_state* s) {
    return s && s->batch >= 1 && s->batch <= HS_MAX_BATCH && s->top_k >= 1 && s->top_k <= HS_MAX_TOPK &&
           s->cap >= 1 + s->top_k && s->n_cand && s->parent && s->token && s->depth && s->logc && s->score &&
           s->frontier && s->n_frontier && s->status;
}

extern "C" hs_status hs_expand_init(hs_ctx* ctx, const hs_expand_state* st, hs_stream stream) {
    if (!ctx || !hs_on_device(ctx) || !state_ok(st)) return HS_ERR_INVALID_ARG;
    return hs_launch(expand_init_kernel, dim3((st->batch + 127) / 128), dim3(128), 0, (cudaStream_t)stream, ctx->pdl,
                     dim3(1, 1, 1), *st) == cudaSuccess ? HS_OK : HS_ERR_CUDA;
}

extern "C" hs_status hs_expand_level(hs_ctx* ctx, const hs_expand_state* st, const float* topk_val,
                                     const int32_t* topk_idx, const float* row_lse, int32_t topk_stride,
                                     hs_stream stream) {
    if (!ctx || !hs_on_device(ctx) || !state_ok(st) || !topk_val || !topk_idx || !row_lse) return HS_ERR_INVALID_ARG;
    if (topk_stride < st->top_k) return HS_ERR_INVALID_ARG;
    return hs_launch(expand_level_kernel, dim3(st->batch), dim3(EX_THREADS), 0, (cudaStream_t)stream, ctx->pdl,
                     dim3(1, 1, 1), *st, topk_val, topk_idx, row_lse, (int)topk_stride) == cudaSuccess ? HS_OK : HS_ERR_CUDA;
}

extern "C" hs_status hs_rerank(hs_ctx* ctx, const hs_expand_state* st, const int32_t* n_top, int32_t n_default,
                               int32_t* node_off, int32_t* parent, int32_t* token, int32_t* cand_id, int32_t* depth,
                               hs_stream stream) {
    if (!ctx || !hs_on_device(ctx) || !state_ok(st) || !node_off || !parent || !token || !cand_id || !depth)
        return HS_ERR_INVALID_ARG;
    if (st->cap > EX_MAX_CAP || (!n_top && n_default < 1)) return HS_ERR_SHAPE;
    RerankParams p;
    p.st = *st; p.n_top = n_top; p.n_default = n_default;
    p.node_off = node_off; p.parent = parent; p.token = token; p.cand_id = cand_id; p.depth = depth;
    const int threads = st->cap < RR_THREADS ? (st->cap + 31) / 32 * 32 : RR_THREADS;      // two candidates each
    return hs_launch(rerank_kernel, dim3(st->batch), dim3(threads), 0, (cudaStream_t)stream, ctx->pdl, dim3(1, 1, 1), p) ==
                   cudaSuccess ? HS_OK : HS_ERR_CUDA;
}
