// hs_accept_path: the row pass (one of two kernels) and, with draft logits, the walk.
//
// accept_rows_kernel   vocabulary pass over the target row of every kept node (arg-max with lowest
//                      index on ties; for sampling sequences also max and sum e^((x-max)/T)) and
//                      over the draft row of every kept internal node of a sampling sequence.
//                      A CTA per 32 KiB chunk of a row, all 16-byte loads in flight at once (launches
//                      with few rows); the chunks of a row merge in the shared memory of a thread-block
//                      cluster, or through partials and an arrival counter where the grid is too large
//                      for clusters to pay.
// accept_warp_kernel   the same pass for launches with many rows: every warp streams a share of the rows (accept_warps.cuh).
//                      Greedy sequences and sequences with deterministic proposals finish in the row
//                      pass: the CTA that completes a sequence's last target row walks its tree
//                      (greedy_walk, deterministic_walk).
// accept_walk_kernel   one thread-block cluster per sequence walks the tree from the root.
//                      Greedy (temperature 0): follow the child whose token is the arg-max.
//                      Sampling (Sec. 2.1): test siblings in index order with u < min(1, r/q); the
//                      residual after k rejections is max(p - c_k q, 0) / W_k with c_0 = 0, W_0 = 1,
//                      c_(k+1) = c_k + W_k, W_k = sum_v max(p_v - c_k q_v, 0), so a rejection costs
//                      one vocabulary-wide sum, split over the CTAs of the cluster and exchanged
//                      through distributed shared memory.  The bonus token is drawn by inverse CDF
//                      in token order, from the sums of the last rejection where there was one.  A node's
//                      probabilities are exponentiated once, into registers: a rejection after the first 2.4 k
//                      clocks instead of 4.5 k (two thirds of it shuffles and fp64 additions of three prefixes,
//                      the rest the exchange), a draw behind rejections 0.4 k instead of 6.8 k, the first sum of a
//                      node 4.6 - 6.2 k.  One tree, 64 heads, sampling: step 60.2 -> 56.1 us with the entropy pass of
//                      few rows (57.9 before this).
#include <cooperative_groups.h>
#include <math_constants.h>

#include "draw_cross.h"
#include "hs_common.cuh"
#include "hs_layout.h"
#include "hs_ptx.cuh"
#include "row_rounds.cuh"

namespace cg = cooperative_groups;

#define WALK_CLUSTER 16       // CTAs per sequence: 16 (larger than the portable 8: the launcher asks for it), or 8 for large batches
#define WALK_THREADS 512

// A bonus draw of a deterministic-proposal sequence that the CTAs of the launch share (in the workspace, one per sequence).
#define DET_SLICES 64
#define DET_MAX_BATCH 256     // sequences the sharing keeps counters for
struct DetJob {
    double sum[DET_SLICES];   // mass of each slice of the vocabulary
    int last[DET_SLICES];     // its last token of positive mass, -1
    const char* row;          // the target row of the node the walk ended on
    float pm, ips, invT;      // its maximum, 1 / sum, log2(e) / temperature
    int nrej;
    int rej[HS_MAX_NODES];    // tokens rejected there
};

struct RowOut {           // per kept node, in the workspace
    int* tgt_arg;         // arg-max token of the target row
    float2* tgt_ms;       // {max, sum e^((x-max)/T)} of the target row
    float2* drf_ms;       // same for the draft row (internal nodes of sampling sequences)
};

struct AcceptParams {
    const void* target;
    const void* draft;
    int64_t row_stride;
    int vocab, nvec, chunks, chunk_vecs, is_bf16, have_draft;
    int batch, n_nodes_total, target_layout, part_rows;
    const int* node_off;
    const int* token;
    hs_pruned_tree pr;
    const int* mode;
    const float* temperature;
    unsigned long long seed, offset;
    const float* uniforms;
    hs_accept_out out;
    RowOut ro;
    uint4* partials;      // [2][max_rows][chunks] {key lo, key hi, max, sum}
    int* row_cnt;
    int* seq_cnt;         // [batch] merged target rows of a sequence (zero between launches)
    DetJob* jobs;         // [batch], or NULL: every draw is made by the CTA that walked the tree
    int* det_cnt;         // [4][DET_MAX_BATCH] of a job: published, slices taken, slices finished, CTAs that have left (zero between launches)
    int shares;           // warp kernel: shares of the stream of rows
    int clustered;        // chunk kernel: the chunks of a row form a thread-block cluster and merge through shared memory
    int staged;           // the walk may stage row slices in shared memory by bulk copies (16-byte aligned rows)
    int* err;             // sticky device error word (a bounded wait that expired)
};

// Greedy acceptance of sequence b by one whole CTA (Sec. 5, temperature 0): from the root, move to the kept
// child whose token is the arg-max of the current node's target row until no child matches; the bonus
// token is the arg-max where the walk stops.  tgt_arg was written by other CTAs: read it past L1.
// The two walks below are run by the first HS_ROW_THREADS threads of a CTA (the whole CTA of the chunk kernel, eight of the
// sixteen warps of the warp kernel), which meet on a barrier of their own.
__device__ __forceinline__ void walk_sync() { named_bar_sync(2, HS_ROW_THREADS); }

// last b with off[b] <= k (skips empty sequences), by a whole warp
__device__ __forceinline__ int sequence_of(const int* off, int batch, int k, int lane) {
    int lo = 0, len = batch;
    while (len > 1) {
        const int step = (len + 31) / 32;
        const bool le = lane * step < len && off[lo + lane * step] <= k;
        const int n = __popc(__ballot_sync(HS_FULL_MASK, le));        // (off ascends: the lanes that agree are the first n)
        lo += (n - 1) * step;
        len = min(step, len - (n - 1) * step);
    }
    return lo;
}

struct WalkNode {         // kept node `threadIdx.x` of a sequence
    int par, tok, orig;   // parent among the kept nodes, token, drafted node id
};
__device__ __forceinline__ WalkNode load_walk_node(const AcceptParams& p, int koff, int nk, int nbase) {
    WalkNode n = {-1, -1, 0};
    if ((int)threadIdx.x < nk) {
        n.par = p.pr.new_parent[koff + threadIdx.x];
        n.orig = p.pr.keep_idx[koff + threadIdx.x];
        n.tok = p.token[nbase + n.orig];
    }
    return n;
}

__device__ void greedy_walk(const AcceptParams& p, int b, int koff, int nk, const WalkNode& node) {
    __shared__ int s_arg[HS_MAX_NODES], s_next[HS_MAX_NODES], s_orig[HS_MAX_NODES];
    const int tid = threadIdx.x, nthr = HS_ROW_THREADS;
    nk = min(nk, HS_MAX_NODES);
    const int cap = p.out.path_cap;
    // The rows' arg-maxima in one round trip; the walk itself then runs in shared memory: node j continues the path of its
    // parent iff its token is the parent's arg-max, and of several such children (duplicate tokens among siblings) the one
    // with the lowest index does.
    if (tid < nk) {
        s_arg[tid] = __ldcg(&p.ro.tgt_arg[koff + tid]);
        s_orig[tid] = node.orig;
        s_next[tid] = 0x7fffffff;
    }
    for (int j = tid; j < cap; j += nthr) {
        p.out.path_nodes[b * cap + j] = -1;
        p.out.path_compact[b * cap + j] = -1;
        p.out.path_tokens[b * cap + j] = -1;
    }
    walk_sync();
    if (tid > 0 && tid < nk && node.par >= 0 && node.par < tid && node.tok == s_arg[node.par]) atomicMin(&s_next[node.par], tid);
    walk_sync();
    if (tid == 0) {
        int cur = 0, len = 0;
        for (int step = 0; step < nk; ++step) {
            if (len < cap) {
                p.out.path_compact[b * cap + len] = cur;
                p.out.path_nodes[b * cap + len] = s_orig[cur];
            }
            const int nxt = s_next[cur];
            if (nxt == 0x7fffffff) break;
            if (len < cap) p.out.path_tokens[b * cap + len] = s_arg[cur];
            cur = nxt;
            ++len;
        }
        p.out.accept_len[b] = len;
        p.out.bonus_token[b] = s_arg[cur];
        p.out.terminal_rank[b] = p.pr.keep_rank[koff + cur];
        p.out.status[b] = HS_OK;
    }
}

__device__ __forceinline__ float load_logit(const void* base, int is_bf16, size_t off);

#include "accept_det.cuh"

// Few rows: a CTA per chunk of a row, all loads in flight at once.  Bound by its chain of latencies, so the chain is short: the
// entries of the pruned tree come in one round trip for a single sequence (two for a batch), what a walk needs of the tree is
// fetched beside the row, a thread takes packed maxima and only a warp that holds the chunk's maximum looks for its index, and
// the chunks of a row that form a cluster send their results to its first CTA and leave.
template <bool BF16>
__global__ void __launch_bounds__(HS_ROW_THREADS, 4) accept_rows_kernel(const __grid_constant__ AcceptParams p) {
    constexpr int VE = BF16 ? 8 : 4;
    constexpr int VPT = HS_ROW_VPT;
    constexpr int NW = HS_ROW_THREADS / 32;
    __shared__ float2 s_w[NW];                    // {max, sum} per warp
    __shared__ unsigned int s_arg;                // first token of the chunk with its maximum
    __shared__ __align__(16) uint4 s_cl[8];       // clustered launch, first CTA of a row: the chunks' results
    __shared__ unsigned long long s_bar;          //   and the barrier that counts them
    __shared__ int s_flag;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int chunk = blockIdx.x, k = blockIdx.y, which = blockIdx.z;   // which: 0 target, 1 draft
    if (tid == 0) {
        s_arg = 0x7fffffffu;
        s_flag = 0;
        if (p.clustered && chunk == 0) {
            mbar_init(smem_u32(&s_bar), 1);
            mbar_expect_tx(smem_u32(&s_bar), (unsigned int)(p.chunks - 1) * 16u);
            mbar_init_fence();
        }
    }
    __syncwarp();
    if (!p.have_draft) pdl_launch_dependents();      // (else behind the wait: the walk kernel relies on it)
    // First half of a cluster barrier: when it completes every CTA of the row's cluster runs, and its shared memory may
    // be written from outside.  (The CTAs of a cluster take every early exit below together: same row, same sequence.)
    if (p.clustered) cluster_arrive();
    pdl_wait();                            // the pruned tree and the logits come from upstream
    if (p.have_draft) pdl_launch_dependents();
    const int kept = p.pr.keep_off[p.batch], kidx = p.pr.keep_idx[k];
    const bool check = chunk == 0 && which == 0 && k < p.batch;
    const int e_keep = check ? p.pr.n_keep[k] : 1, e_status = check ? p.pr.status[k] : 0;
    const int b = sequence_of(p.pr.keep_off, p.batch, k, lane);
    const int koff = p.pr.keep_off[b], nk = p.pr.n_keep[b], md = p.mode[b], nbase = p.node_off[b];
    const float temp = p.temperature[b];
    // sequences that kept nothing (flagged upstream) get their empty result from CTA (0, b, 0)
    if (e_keep <= 0 || e_status != 0) {
        const int cap = p.out.path_cap;
        for (int j = tid; j < cap; j += HS_ROW_THREADS) {
            p.out.path_nodes[k * cap + j] = -1;
            p.out.path_compact[k * cap + j] = -1;
            p.out.path_tokens[k * cap + j] = -1;
        }
        if (tid == 0) {
            p.out.accept_len[k] = 0; p.out.bonus_token[k] = -1; p.out.terminal_rank[k] = -1;
            p.out.status[k] = e_status != 0 ? e_status : HS_ERR_BAD_TREE;
        }
    }
    if (k >= kept) return;
    const int i = k - koff;
    const bool sampling = md != HS_ACCEPT_GREEDY;          // the row's normaliser is needed
    if (which == 1) {
        if (md != HS_ACCEPT_REJECTION) return;
        int internal = 0;                         // does kept node i have a kept child?
        for (int j = i + 1 + tid; j < nk; j += HS_ROW_THREADS)
            internal |= (p.pr.new_parent[koff + j] == i);
        if (!__syncthreads_or(internal)) return;
    }
    const int row = which == 1 || p.target_layout == HS_ROWS_ORIGINAL ? nbase + kidx : k;
    const char* rowp = (const char*)(which == 1 ? p.draft : p.target) + (size_t)row * p.row_stride * (BF16 ? 2 : 4);
    const int v0 = chunk * p.chunk_vecs;
    const int v1 = min(v0 + p.chunk_vecs, p.nvec);

    uint4 d[VPT];
    const unsigned int ninf = BF16 ? 0xff80ff80u : 0xff800000u;
#pragma unroll
    for (int j = 0; j < VPT; ++j) {
        const int v = v0 + tid + j * HS_ROW_THREADS;
        d[j] = v < v1 ? ld_stream((const uint4*)rowp + v) : make_uint4(ninf, ninf, ninf, ninf);
    }
    // the walk's view of node `tid` (a greedy sequence is walked by one of its CTAs), fetched while the row is on its way
    WalkNode node;
    if (md == HS_ACCEPT_GREEDY && which == 0 && (chunk == 0 || !p.clustered)) node = load_walk_node(p, koff, nk, nbase);
    if (v1 == p.nvec && p.nvec * VE != p.vocab) {          // the row's last vector runs past vocab
#pragma unroll
        for (int j = 0; j < VPT; ++j)
            if (v0 + tid + j * HS_ROW_THREADS == p.nvec - 1) mask_tail<BF16>(d[j], p.nvec - 1, p.vocab);
    }
    static_assert(VPT == 8, "two rounds of four vectors");
    const uint4(&da)[4] = *reinterpret_cast<const uint4(*)[4]>(&d[0]);
    const uint4(&db)[4] = *reinterpret_cast<const uint4(*)[4]>(&d[4]);
    const float tmax = fmaxf(round_max<BF16>(da), round_max<BF16>(db));
    const float wm = order_bits_float(__reduce_max_sync(HS_FULL_MASK, float_order_bits(tmax)));
    const float invT = sampling ? LOG2E / temp : 0.f;
    float s = 0.f;
    if (sampling) {
        const float n = wm == -CUDART_INF_F ? 0.f : -wm * invT;
        const float2 l2 = make_float2(invT, invT), n2 = make_float2(n, n);
        float2 s2 = make_float2(0.f, 0.f);
        const unsigned int* x = reinterpret_cast<const unsigned int*>(&d[0]);
#pragma unroll
        for (int q = 0; q < (BF16 ? 4 * VPT : 2 * VPT); ++q) {
            const float2 t = fma2_ftz(BF16 ? make_float2(bf16_lo(x[q]), bf16_hi(x[q]))
                                           : make_float2(__uint_as_float(x[2 * q]), __uint_as_float(x[2 * q + 1])), l2, n2);
            s2 = add2_ftz(s2, make_float2(ex2f(t.x), ex2f(t.y)));
        }
        s = warp_sum(s2.x + s2.y);
    }
    if (lane == 0) s_w[warp] = make_float2(wm, s);
    __syncthreads();
    if (p.clustered) cluster_wait();
    const float2 ws = lane < NW ? s_w[lane] : make_float2(-CUDART_INF_F, 0.f);
    float M = warp_max(ws.x);
    if (wm == M && M > -CUDART_INF_F) {                    // this warp holds the chunk's maximum: the lowest index it has it at
        unsigned int at = 0x7fffffffu;
        if (tmax == M) {
#pragma unroll
            for (int j = VPT - 1; j >= 0; --j) {
                float x[8];
                unpack<BF16>(d[j], x);
#pragma unroll
                for (int e = VE - 1; e >= 0; --e)
                    if (x[e] == M) at = (unsigned int)((v0 + tid + j * HS_ROW_THREADS) * VE + e);
            }
        }
        at = __reduce_min_sync(HS_FULL_MASK, at);
        if (lane == 0) atomicMin(&s_arg, at);
    }
    __syncthreads();
    bool merges = false;                                   // (warp 0: it holds the row's result)
    if (warp == 0) {
        float S = sampling ? warp_sum(ws.x == -CUDART_INF_F ? 0.f : ws.y * ex2f((ws.x - M) * invT)) : 0.f;
        unsigned long long key = M > -CUDART_INF_F ? make_key(M, (int)s_arg) : 0ull;
        if (p.chunks == 1) {
            merges = true;
        } else if (p.clustered) {
            // the chunk's result goes into slot `chunk` of the first CTA of the row's cluster
            if (chunk != 0) {
                if (lane == 0)
                    st_async_v4(cluster_map_addr(smem_u32(&s_cl[chunk]), 0), (unsigned int)key, (unsigned int)(key >> 32),
                                __float_as_uint(M), __float_as_uint(S), cluster_map_addr(smem_u32(&s_bar), 0));
            } else {
                mbar_wait_cluster(smem_u32(&s_bar), 0u, p.err);
                merges = true;
            }
        } else {
            if (lane == 0) {
                p.partials[((size_t)which * p.part_rows + k) * p.chunks + chunk] =
                    make_uint4((unsigned int)key, (unsigned int)(key >> 32), __float_as_uint(M), __float_as_uint(S));
                // one release-acquire arrival at device scope: this thread's partial is visible to whoever arrives last,
                // and the last one sees all of them
                int* cnt = &p.row_cnt[which * HS_MAX_ROWS + k];
                int old;
                asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(old) : "l"(cnt) : "memory");
                merges = old == p.chunks - 1;
                if (merges) *cnt = 0;
            }
            merges = __shfl_sync(HS_FULL_MASK, merges, 0);
        }
        if (merges) {
            if (p.chunks > 1) {                            // (chunks <= 32, one lane per chunk)
                unsigned long long ck = 0ull;
                float cm = -CUDART_INF_F, cs = 0.f;
                if (lane < p.chunks) {
                    const uint4 q = p.clustered ? s_cl[lane] : __ldcg(&p.partials[((size_t)which * p.part_rows + k) * p.chunks + lane]);
                    ck = ((unsigned long long)q.y << 32) | q.x;
                    cm = __uint_as_float(q.z);
                    cs = __uint_as_float(q.w);
                    if (p.clustered && lane == 0) { ck = key; cm = M; cs = S; }
                }
                int src;
                key = warp_best_key(ck, src);
                M = warp_max(cm);
                if (sampling) S = warp_sum((cm == -CUDART_INF_F) ? 0.f : cs * ex2f((cm - M) * invT));
            }
            if (lane == 0) {
                s_flag = 1;
                if (which == 0) {
                    p.ro.tgt_arg[k] = key_index(key);
                    p.ro.tgt_ms[k] = make_float2(M, S);
                    if (md != HS_ACCEPT_REJECTION) {
                        int old;
                        asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(old) : "l"(&p.seq_cnt[b]) : "memory");
                        if (old == nk - 1) { s_flag = 2; p.seq_cnt[b] = 0; }   // the sequence's last target row: walk its tree
                    }
                } else {
                    p.ro.drf_ms[k] = make_float2(M, S);
                }
            }
        }
    }
    if (p.clustered && chunk != 0 && !(p.jobs && md == HS_ACCEPT_DETERMINISTIC && which == 0)) return;
    __syncthreads();
    const int flag = s_flag;
    if (flag && md == HS_ACCEPT_REJECTION && !p.have_draft && which == 0 && i == 0) {
        // rejection sampling needs the draft distribution: the caller passed none
        const int cap = p.out.path_cap;
        for (int j = tid; j < cap; j += HS_ROW_THREADS) {
            p.out.path_nodes[b * cap + j] = -1;
            p.out.path_compact[b * cap + j] = -1;
            p.out.path_tokens[b * cap + j] = -1;
        }
        if (tid == 0) {
            p.out.accept_len[b] = 0; p.out.bonus_token[b] = -1; p.out.terminal_rank[b] = -1;
            p.out.status[b] = HS_ERR_INVALID_ARG;
        }
    }
    if (which != 0 || md == HS_ACCEPT_REJECTION) return;
    // greedy sequences finish here; CTAs of a deterministic-proposal sequence stay to take slices of its bonus draw (where
    // the whole grid is resident)
    if (md == HS_ACCEPT_DETERMINISTIC) {
        if (flag == 2 || p.jobs) det_chunk_tail(p, b, nk, flag == 2);
    } else if (flag == 2) {
        greedy_walk(p, b, koff, nk, node);
    }
}

#include "accept_warps.cuh"

// Launches with fewer bytes of rows go to the chunk kernel, whose loads are all in flight at once.  us a call, chunk against warp kernel,
// greedy: 60 rows of 128256 bf16 (15 MiB) 8.3 : 11.1, 71 rows (17 MiB) 10.1 : 11.7, 92 (22 MiB) 12.6 : 12.3, 120 (29 MiB) 13.3 : 12.9, 180 of 64000
// (22 MiB) 12.0 : 12.4.  With draft logits, which are read for the inner nodes of rejection sequences only: one such sequence is decided by the
// same bytes (60 rows 20.0 : 20.4, alone 25.6 : 27.6).  In a batch the draft rows are counted like target rows, although 71 rows of two rejection
// sequences take 22.0 in either kernel: the host does not see the modes, and the bonus draw of a deterministic-proposal sequence is shared
// by the warp kernel at any size but by the chunk kernel only while its grid is resident (two such sequences, 71 rows: 55.2 : 28.0).
#define AW_MIN_BYTES ((size_t)20 << 20)

// ---- the walk ----------------------------------------------------------------------------------

__device__ __forceinline__ float load_logit(const void* base, int is_bf16, size_t off) {
    return is_bf16 ? __bfloat162float(((const __nv_bfloat16*)base)[off]) : ((const float*)base)[off];
}

// This CTA's slice of the current node's target row p and draft row q: vectors [v0, v0 + nv) of the row, read
// through pointers to shared memory (staged by bulk copies) or to the rows themselves.
struct RowSlice {
    const uint4* p;
    const uint4* q;       // NULL when only p is there
    int v0, nv;
};

// All-gather of one 64-bit value per CTA over the cluster of WC CTAs: warp 0 of every CTA stores its value into slot `rank`
// of the exchange buffer of all CTAs (posted stores through distributed shared memory, lane r to CTA r), one
// cluster barrier makes them visible, every CTA then reads its own copy.  The buffers alternate from one exchange to
// the next (s_x[xch & 1]), so one barrier per exchange is enough: a buffer is written again only two exchanges later,
// after a barrier that every CTA reaches with its reads done.  `v` must be valid in warp 0.
template <int WC>
__device__ __forceinline__ void cluster_allgather(unsigned long long v, unsigned long long (*s_x)[WALK_CLUSTER],
                                                  unsigned int& xch, unsigned int rank) {
    unsigned long long* buf = s_x[xch & 1u];
    ++xch;
    if (threadIdx.x < WC) {
        const unsigned int remote = cluster_map_addr(smem_u32(&buf[rank]), threadIdx.x);
        asm volatile("st.shared::cluster.b64 [%0], %1;" ::"r"(remote), "l"(v) : "memory");
    }
    __syncwarp();
    cluster_arrive();
    cluster_wait();
}
static_assert(WALK_THREADS / 32 == 16, "prefixes over the warps take 16 lanes");

// The probabilities of a thread's tokens at the node the walk stands on, target and draft.  A thread has a contiguous run of the vectors of its
// CTA's slice, taken in pieces of EL tokens; a run of one piece (up to 131072 bf16 logits over 16 CTAs of 512 threads) is exponentiated once
// per node and serves every rejection there and the final draw.
#define WALK_EL 16            // (32 spill)
struct Masses {
    float p[WALK_EL], q[WALK_EL];
    int w0, w1, pieces;       // the thread's vectors of the slice, pieces of its run
    int held;                 // piece in p, q; -1: none
};
struct RowScale {             // of a node: maxima, 1 / sums, log2(e) / temperature
    float pm, ips, qm, iqs, invT;
};
template <bool BF16>
__device__ __forceinline__ void fill_masses(Masses& m, int vocab, const RowSlice& rs, int piece, const RowScale& k) {
    constexpr int VE = BF16 ? 8 : 4;
#pragma unroll
    for (int i = 0; i < WALK_EL / VE; ++i) {
        const int v = m.w0 + piece * (WALK_EL / VE) + i;
#pragma unroll
        for (int e = 0; e < VE; ++e) m.p[i * VE + e] = m.q[i * VE + e] = 0.f;
        if (v >= m.w1) continue;
        float x[8];
        const int inside = vocab - (rs.v0 + v) * VE;             // tokens of the vocabulary in this vector (and behind it)
        unpack<BF16>(rs.p[v], x);
#pragma unroll
        for (int e = 0; e < VE; ++e)
            if (e < inside) m.p[i * VE + e] = exp2f((fmaxf(x[e], -1e30f) - k.pm) * k.invT) * k.ips;
        if (!rs.q) continue;
        unpack<BF16>(rs.q[v], x);
#pragma unroll
        for (int e = 0; e < VE; ++e)
            if (e < inside) m.q[i * VE + e] = exp2f((fmaxf(x[e], -1e30f) - k.qm) * k.invT) * k.iqs;
    }
}
// inclusive prefix over lanes 0 .. N - 1
template <int N>
__device__ __forceinline__ double warp_prefix_d(double v, int lane) {
#pragma unroll
    for (int o = 1; o < N; o <<= 1) {
        const double up = __shfl_up_sync(HS_FULL_MASK, v, o);
        if (lane >= o) v += up;
    }
    return v;
}

template <int WC>
__global__ void __launch_bounds__(WALK_THREADS, 1) accept_walk_kernel(const __grid_constant__ AcceptParams p) {
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ __align__(16) unsigned char s_rows[];    // staged: this CTA's slices of p and q, `per` vectors each
    __shared__ unsigned long long s_bar;
    __shared__ double s_scan[WALK_THREADS / 32];
    __shared__ unsigned long long s_x[2][WALK_CLUSTER];    // all-gather buffers of the cluster exchanges
    unsigned int xch = 0;                  // exchanges through s_x so far
    __shared__ int s_pick[2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = blockIdx.x / WC;
    const unsigned int rank = cluster.block_rank();
    pdl_launch_dependents();
    // Ahead of the dependency wait: all that does not come from the row pass.  (The row pass lets this kernel start only behind its
    // own wait, so the pruned tree and the caller's arrays are complete.)  Every candidate's logits under its parent's target and
    // draft row and its uniform, for all kept nodes at once: a thread per node, four dependent round trips of which
    // none is left on the path between the row pass and the walk (3 us of the 12 us of one sequence).
    static_assert(WALK_THREADS >= HS_MAX_NODES, "a thread per node");
    const int koff = p.pr.keep_off[b];
    const int nk = p.pr.n_keep[b];
    const int tree_status = p.pr.status[b];
    const int nbase = p.node_off[b];
    const int cap = p.out.path_cap;
    const bool sampling = p.mode[b] == HS_ACCEPT_REJECTION;
    const size_t esz = p.is_bf16 ? 2 : 4;
    const int nkc = tree_status == 0 ? min(nk, HS_MAX_NODES) : 0;
    const bool mine = sampling && tid < nkc;                  // this thread has node tid
    int par = -1, orig = 0, tok = 0;
    float lp = 0.f, lq = 0.f, u = 0.f, T = 1.f;
    if (sampling) T = p.temperature[b];
    if (mine) {
        par = p.pr.new_parent[koff + tid];
        orig = p.pr.keep_idx[koff + tid];
        tok = p.token[nbase + orig];
        if (par >= 0 && par < nkc) {
            const int porig = p.pr.keep_idx[koff + par];
            const int trow = p.target_layout == HS_ROWS_ORIGINAL ? nbase + porig : koff + par;
            lp = load_logit((const char*)p.target + (size_t)trow * p.row_stride * esz, p.is_bf16, tok);
            lq = load_logit((const char*)p.draft + (size_t)(nbase + porig) * p.row_stride * esz, p.is_bf16, tok);
        }
        u = p.uniforms ? p.uniforms[nbase + orig] : philox_uniform(p.seed, p.offset, b, orig, 0);
    }
    const float ufin = !sampling ? 0.f : p.uniforms ? p.uniforms[p.n_nodes_total + b] : philox_uniform(p.seed, p.offset, b, 0, 1);
    pdl_wait();                            // arg-max and normalisers come from the row pass

    if (!sampling && nk > 0 && tree_status == 0) return;      // greedy sequences were finished by the row pass
    if (rank == 0) {
        for (int j = tid; j < cap; j += WALK_THREADS) {
            p.out.path_nodes[b * cap + j] = -1;
            p.out.path_compact[b * cap + j] = -1;
            p.out.path_tokens[b * cap + j] = -1;
        }
    }
    if (nk <= 0 || tree_status != 0) {
        if (rank == 0 && tid == 0) {
            p.out.accept_len[b] = 0; p.out.bonus_token[b] = -1; p.out.terminal_rank[b] = -1;
            p.out.status[b] = tree_status != 0 ? tree_status : HS_ERR_BAD_TREE;
        }
        return;
    }
    // This CTA's slice of a row: vectors [v0, v0 + nv).  The rows of the node the walk stands on are brought into
    // shared memory once (one bulk copy each, only when a residual or the final draw needs them) and serve every
    // rejection at that node and the final draw.
    const int per = (p.nvec + WC - 1) / WC;
    RowSlice rs;
    rs.v0 = rank * per;
    rs.nv = max(min(rs.v0 + per, p.nvec) - rs.v0, 0);
    rs.p = nullptr; rs.q = nullptr;
    Masses m;
    const int ve = p.is_bf16 ? 8 : 4;
    {
        const int run = (rs.nv + WALK_THREADS - 1) / WALK_THREADS;
        m.w0 = min(tid * run, rs.nv); m.w1 = min(m.w0 + run, rs.nv);
        m.pieces = (run * ve + WALK_EL - 1) / WALK_EL;
        m.held = -1;
    }
    const unsigned int bar = smem_u32(&s_bar);
    if (tid == 0 && p.staged) { mbar_init(bar, 1); mbar_init_fence(); }
    unsigned int stage_n = 0;
    int staged_node = -1;
    bool staged_q = false;
    auto stage = [&](int node, const char* prow, const char* qrow) {      // qrow may be NULL: only p
        if (staged_node == node && (staged_q || qrow == nullptr)) {
            if (qrow == nullptr && rs.q != nullptr) { rs.q = nullptr; m.held = -1; }
            return;
        }
        staged_node = node; staged_q = qrow != nullptr;
        m.held = -1;
        if (!p.staged) {
            rs.p = (const uint4*)prow + rs.v0;
            rs.q = qrow ? (const uint4*)qrow + rs.v0 : nullptr;
            return;
        }
        __syncthreads();                   // nobody still reads the rows of the previous node
        if (tid == 0) {
            const unsigned int bytes = (unsigned int)rs.nv * 16u;
            mbar_expect_tx(bar, qrow ? 2u * bytes : bytes);
            if (bytes) {
                bulk_load(smem_u32(s_rows), (const uint4*)prow + rs.v0, bytes, bar);
                if (qrow) bulk_load(smem_u32(s_rows) + (unsigned int)per * 16u, (const uint4*)qrow + rs.v0, bytes, bar);
            }
        }
        mbar_wait(bar, stage_n & 1u, p.err);
        ++stage_n;
        rs.p = (const uint4*)s_rows;
        rs.q = qrow ? (const uint4*)s_rows + per : nullptr;
    };
    // Every candidate's probability under its parent's target and draft row, its uniform and the normalisers of its own rows, for all
    // kept nodes at once: one round trip for the normalisers; the walk below then runs from shared memory until a rejection needs a
    // vocabulary-wide residual sum.  Every CTA of the cluster fetches the same values and takes the same decisions.
    __shared__ int s_par[HS_MAX_NODES], s_tok[HS_MAX_NODES], s_orig[HS_MAX_NODES];
    __shared__ float s_pt[HS_MAX_NODES], s_qt[HS_MAX_NODES], s_u[HS_MAX_NODES];
    __shared__ float2 s_pms[HS_MAX_NODES];
    // Also per node: its first (lowest-index) kept child and whether that child, tested first (residual = p), is
    // accepted - the common step of the walk then costs two shared-memory reads.
    __shared__ int s_first[HS_MAX_NODES];
    __shared__ unsigned char s_acc0[HS_MAX_NODES];
    const float invT = LOG2E / T;
    float2 oms = make_float2(0.f, 1.f), pms0 = oms, qms0 = oms;
    const bool child = mine && par >= 0 && par < nkc;
    if (mine) {
        oms = p.ro.tgt_ms[koff + tid];
        s_first[tid] = 0x7fffffff;
    }
    if (child) { pms0 = p.ro.tgt_ms[koff + par]; qms0 = p.ro.drf_ms[koff + par]; }
    __syncthreads();
    if (mine) {
        float pt = 0.f, qt = 0.f;
        if (child) {
            pt = exp2f((fmaxf(lp, -1e30f) - pms0.x) * invT) * (1.f / pms0.y);
            qt = exp2f((fmaxf(lq, -1e30f) - qms0.x) * invT) * (1.f / qms0.y);
        }
        s_par[tid] = par; s_tok[tid] = tok; s_orig[tid] = orig;
        s_pms[tid] = oms;
        s_pt[tid] = pt; s_qt[tid] = qt;
        s_u[tid] = u;
        // (the same expressions as in the sibling loop below with c = 0, W = 1: the same decision, bit for bit)
        const float r0 = fmaxf(pt - 0.f * qt, 0.f) / 1.f;
        const float a0 = qt > 0.f ? fminf(1.f, r0 / qt) : 1.f;
        s_acc0[tid] = (par >= 0 && par < tid && u < a0) ? 1 : 0;
        if (par >= 0 && par < tid) atomicMin(&s_first[par], tid);
    }
    __syncthreads();
    int cur = 0, len = 0;
    bool drawn = false;
    {
        for (int step = 0; step < nkc; ++step) {
            if (rank == 0 && tid == 0 && len < cap) {
                p.out.path_compact[b * cap + len] = cur;
                p.out.path_nodes[b * cap + len] = s_orig[cur];
            }
            {
                const int j1 = s_first[cur];
                if (j1 != 0x7fffffff && s_acc0[j1]) {            // the first child is accepted: no residual is needed
                    if (rank == 0 && tid == 0 && len < cap) p.out.path_tokens[b * cap + len] = s_tok[j1];
                    cur = j1;
                    ++len;
                    continue;
                }
            }
            const int trow = p.target_layout == HS_ROWS_ORIGINAL ? nbase + s_orig[cur] : koff + cur;
            const int drow = nbase + s_orig[cur];
            const char* prow = (const char*)p.target + (size_t)trow * p.row_stride * esz;
            const char* qrow = (const char*)p.draft + (size_t)drow * p.row_stride * esz;
            RowScale k;
            k.pm = s_pms[cur].x; k.ips = 1.f / s_pms[cur].y; k.qm = 0.f; k.iqs = 0.f; k.invT = invT;
            float c = 0.f, c_next = 0.f;
            double W = 1.0;
            int accepted = -1;
            // the kept children of cur as bit masks (every warp finds them with four ballots instead of a serial scan)
            unsigned int kids[HS_MAX_NODES / 32];
#pragma unroll
            for (int w = 0; w < HS_MAX_NODES / 32; ++w) {
                const int j = w * 32 + (tid & 31);
                kids[w] = __ballot_sync(HS_FULL_MASK, j > cur && j < nkc && s_par[j] == cur);
            }
            // Siblings in index order; each rejection takes the residual's mass, and behind the last one the bonus token is drawn from the
            // residual, whose masses are then known already.  (One place in the code where masses are summed: what runs once is bound by
            // instruction fetch.)
            double mine = 0.0, incl = 0.0, wincl = 0.0, wv = 0.0, gincl = 0.0, gv = 0.0;
            int last_pos = -1;
            bool known = false;                                  // the sums above are those of the residual max(p - c q, 0)
            bool draw = false;
            for (;;) {
                int j = -1;
#pragma unroll
                for (int w = HS_MAX_NODES / 32 - 1; w >= 0; --w)
                    if (kids[w]) j = w * 32 + __ffs(kids[w]) - 1;
                draw = j < 0;
                if (!draw) {
#pragma unroll
                    for (int w = 0; w < HS_MAX_NODES / 32; ++w)
                        if (j >> 5 == w) kids[w] &= kids[w] - 1;
                    const float pt = s_pt[j], qt = s_qt[j];
                    const float r = fmaxf(pt - c * qt, 0.f) / (float)W;
                    const float a = qt > 0.f ? fminf(1.f, r / qt) : 1.f;
                    if (s_u[j] < a) { accepted = j; break; }
                    if (k.iqs == 0.f) {
                        const float2 qms = p.ro.drf_ms[koff + cur];
                        k.qm = qms.x; k.iqs = 1.f / qms.y;
                    }
                    c_next = c + (float)W;
                } else if (known) {
                    break;
                } else {
                    c_next = c;
                }
                stage(cur, prow, c_next > 0.f ? qrow : nullptr);
                // ---- masses of max(p - c_next q, 0): this thread's, ahead of it in the CTA, of the CTAs --------------------------------
                mine = 0.0;
                last_pos = -1;
                for (int ch = 0; ch < m.pieces; ++ch) {
                    if (m.held != ch) {
                        if (p.is_bf16) fill_masses<true>(m, p.vocab, rs, ch, k);
                        else fill_masses<false>(m, p.vocab, rs, ch, k);
                        m.held = ch;
                    }
                    double t[WALK_EL];
#pragma unroll
                    for (int e = 0; e < WALK_EL; ++e) {
                        const float f = fmaxf(m.p[e] - c_next * m.q[e], 0.f);
                        if (f > 0.f) last_pos = (rs.v0 + m.w0) * ve + ch * WALK_EL + e;
                        t[e] = (double)f;
                    }
#pragma unroll
                    for (int o = WALK_EL / 2; o > 0; o >>= 1)
#pragma unroll
                        for (int e = 0; e < o; ++e) t[e] += t[e + o];
                    mine += t[0];
                }
                if (tid == 0) { s_pick[0] = 0x7fffffff; s_pick[1] = -1; }
                incl = warp_prefix_d<32>(mine, lane);
                __syncthreads();                                 // (s_scan may still be read from the sum before)
                if (lane == 31) s_scan[warp] = incl;
                __syncthreads();
                wv = s_scan[lane & 15];
                wincl = warp_prefix_d<16>(wv, lane);
                const double* got = reinterpret_cast<const double*>(s_x[xch & 1u]);
                cluster_allgather<WC>((unsigned long long)__double_as_longlong(__shfl_sync(HS_FULL_MASK, wincl, 15)), s_x, xch, rank);
                gv = got[lane & (WC - 1)];
                gincl = warp_prefix_d<WC>(gv, lane);
                if (draw) break;
                const double W_next = __shfl_sync(HS_FULL_MASK, gincl, WC - 1);
                known = W_next > 0.0;
                if (known) {
                    c = c_next; W = W_next;
                } else {                                         // p == q: fall back to p, no more siblings
                    c = 0.f; W = 1.0;
#pragma unroll
                    for (int w = 0; w < HS_MAX_NODES / 32; ++w) kids[w] = 0u;
                }
            }
            if (accepted >= 0) {
                if (rank == 0 && tid == 0 && len < cap) p.out.path_tokens[b * cap + len] = s_tok[accepted];
                cur = accepted;
                ++len;
                continue;
            }
            // ---- inverse-CDF draw from max(p - c q, 0) in token order: smallest j whose running sum exceeds u * total; if rounding leaves
            // none, the last token with positive mass.  The slice with the crossing is the first whose running total exceeds the goal
            // (rounding leaves none: the last with mass); that CTA finds the token and writes it.
            drawn = true;
            const double goal = (double)ufin * __shfl_sync(HS_FULL_MASK, gincl, WC - 1);
            const double before = __shfl_sync(HS_FULL_MASK, gincl - gv, (int)rank), wbefore = __shfl_sync(HS_FULL_MASK, wincl - wv, warp);
            const unsigned int over = __ballot_sync(HS_FULL_MASK, lane < WC && gincl > goal);
            const unsigned int full = __ballot_sync(HS_FULL_MASK, lane < WC && gv > 0.0);
            const int owner = over ? __ffs(over) - 1 : (full ? 31 - __clz(full) : 0);
            if ((int)rank == owner) {
                double run = before + (wbefore + (incl - mine));
                if (run <= goal && run + mine > goal) {          // the crossing lies in this thread's run
                    bool found = false;
                    for (int ch = 0; ch < m.pieces && !found; ++ch) {
                        if (m.held != ch) {
                            if (p.is_bf16) fill_masses<true>(m, p.vocab, rs, ch, k);
                            else fill_masses<false>(m, p.vocab, rs, ch, k);
                            m.held = ch;
                        }
#pragma unroll
                        for (int e0 = 0; e0 < WALK_EL; e0 += 4) {
                            double t[4];
#pragma unroll
                            for (int e = 0; e < 4; ++e) t[e] = (double)fmaxf(m.p[e0 + e] - c * m.q[e0 + e], 0.f);
                            const int at = found ? -1 : crossing_of_four(t, goal, run);
                            if (at >= 0) { found = true; atomicMin(&s_pick[0], (rs.v0 + m.w0) * ve + ch * WALK_EL + e0 + at); }
                        }
                    }
                    if (!found && last_pos >= 0) atomicMin(&s_pick[0], last_pos);       // (rounding)
                }
                if (last_pos >= 0) atomicMax(&s_pick[1], last_pos);
                __syncthreads();
                if (tid == 0) p.out.bonus_token[b] = s_pick[0] != 0x7fffffff ? s_pick[0] : max(s_pick[1], 0);
            }
            break;
        }
    }
    // (every store into a CTA's exchange buffers precedes a barrier that CTA takes part in: it may leave now)
    if (rank == 0 && tid == 0) {
        p.out.accept_len[b] = len;
        if (!drawn) p.out.bonus_token[b] = -1;
        p.out.terminal_rank[b] = p.pr.keep_rank[koff + cur];
        p.out.status[b] = HS_OK;
    }
}

__global__ void philox_kernel(unsigned long long seed, unsigned long long offset, const int* b, const int* node,
                              const int* stream_id, int count, float* out) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) out[i] = philox_uniform(seed, offset, b[i], node[i], stream_id[i]);
}

hs_status hs_launch_philox(uint64_t seed, uint64_t offset, const int32_t* b, const int32_t* node,
                           const int32_t* stream_id, int32_t count, float* out, cudaStream_t stream) {
    philox_kernel<<<(count + 255) / 256, 256, 0, stream>>>(seed, offset, b, node, stream_id, count, out);
    return cudaGetLastError() == cudaSuccess ? HS_OK : HS_ERR_CUDA;
}

hs_status hs_launch_accept(hs_ctx* ctx, const hs_tree_batch* tree, const hs_pruned_tree* pruned,
                           const void* target_logits, int32_t target_layout, const void* draft_logits,
                           hs_dtype dtype, int64_t row_stride, int32_t vocab, const int32_t* mode,
                           const float* temperature, uint64_t seed, uint64_t offset, const float* uniforms,
                           const hs_accept_out* out, cudaStream_t stream) {
    AcceptParams p;
    const int ve = hs_vec_elems(dtype);
    p.target = target_logits;
    p.draft = draft_logits ? draft_logits : target_logits;   // only read by sampling sequences
    p.row_stride = row_stride;
    p.vocab = vocab;
    p.nvec = (vocab + ve - 1) / ve;
    p.chunks = hs_row_chunks(vocab, dtype);
    if (p.chunks > 32) return HS_ERR_SHAPE;
    p.chunk_vecs = (p.nvec + p.chunks - 1) / p.chunks;
    p.is_bf16 = dtype == HS_BF16;
    p.have_draft = draft_logits != nullptr;
    p.batch = tree->batch;
    p.n_nodes_total = tree->n_nodes_total;
    p.target_layout = target_layout;
    p.node_off = tree->node_off;
    p.token = tree->token;
    p.pr = *pruned;
    p.mode = mode;
    p.temperature = temperature;
    p.seed = seed;
    p.offset = offset;
    p.uniforms = uniforms;
    p.out = *out;
    int rows = tree->n_nodes_total;                // upper bound of kept nodes
    if (out->max_kept_rows > 0 && out->max_kept_rows < rows) rows = out->max_kept_rows;
    size_t o = 0;
    p.ro.tgt_arg = (int*)(ctx->scratch + o); o += hs_align_up((size_t)rows * sizeof(int), 256);
    p.ro.tgt_ms = (float2*)(ctx->scratch + o); o += hs_align_up((size_t)rows * sizeof(float2), 256);
    p.ro.drf_ms = (float2*)(ctx->scratch + o); o += hs_align_up((size_t)rows * sizeof(float2), 256);
    p.partials = (uint4*)(ctx->scratch + o);
    p.part_rows = rows;
    const bool streamed = ctx->row_pass == HS_ROW_PASS_STREAM ||
                          (ctx->row_pass == HS_ROW_PASS_AUTO && (size_t)rows * p.nvec * (p.have_draft && p.batch > 1 ? 32 : 16) >= AW_MIN_BYTES);
    // (chunk kernel: a partial per chunk of a row; warp kernel: two per share, one share per warp of the device - fewer
    // and longer ones in a workspace without room for that)
    const size_t room = ctx->scratch_bytes > o ? (ctx->scratch_bytes - o) / (2 * sizeof(uint4)) : 0;
    p.shares = (int)min((size_t)ctx->sm_count * AW_WARPS, room);
    o += streamed ? (size_t)2 * p.shares * sizeof(uint4) : (size_t)2 * rows * p.chunks * sizeof(uint4);
    if (o > ctx->scratch_bytes || (streamed && p.shares < ctx->sm_count)) return HS_ERR_WORKSPACE;
    p.row_cnt = ctx->counters + HS_CNT_ACC_ROW;
    p.seq_cnt = ctx->counters + HS_CNT_ACC_SEQ;
    p.err = ctx->counters + HS_CNT_ERROR;
    p.staged = 0;
    p.clustered = 0;
    p.jobs = nullptr;
    p.det_cnt = ctx->counters + HS_CNT_DET;
    o = hs_align_up(o, 256);
    DetJob* const jobs = p.batch <= DET_MAX_BATCH && o + p.batch * sizeof(DetJob) <= ctx->scratch_bytes ? (DetJob*)(ctx->scratch + o) : nullptr;
    // without draft logits every sequence must be greedy: no draft rows to scan and no sampling walk
    cudaError_t e;
    if (streamed) {
        // enough rows to be bound by memory traffic: every warp of the device streams a share of them
        p.jobs = jobs;
        const dim3 grid(ctx->sm_count), block(AW_THREADS), one(1, 1, 1);
        e = dtype == HS_BF16 ? hs_launch(accept_warp_kernel<true>, grid, block, 0, stream, ctx->pdl, one, p)
                             : hs_launch(accept_warp_kernel<false>, grid, block, 0, stream, ctx->pdl, one, p);
    } else {
        // up to eight chunks per row (the portable cluster size): the CTAs of a row are one cluster, and the row is
        // merged in the shared memory of its first CTA instead of through partials and a counter in global memory
        // - while the whole grid is resident at once (four CTAs per SM): with more CTAs the clusters wait for eight free
        // slots in one GPC and the pass gets slower than with independent CTAs
        p.clustered = p.chunks > 1 && p.chunks <= 8 &&
                      (size_t)p.chunks * rows * (p.have_draft ? 2 : 1) * 2 <= (size_t)7 * ctx->sm_count;
        if (p.clustered) p.jobs = jobs;               // (CTAs that stay to help must not keep others from starting)
        dim3 grid(p.chunks, rows, p.have_draft ? 2 : 1), cl(p.clustered ? p.chunks : 1, 1, 1);
        e = dtype == HS_BF16
            ? hs_launch(accept_rows_kernel<true>, grid, dim3(HS_ROW_THREADS), 0, stream, ctx->pdl, cl, p)
            : hs_launch(accept_rows_kernel<false>, grid, dim3(HS_ROW_THREADS), 0, stream, ctx->pdl, cl, p);
    }
    if (e != cudaSuccess) return HS_ERR_CUDA;
    if (!p.have_draft) return HS_OK;
    // Sixteen CTAs per sequence until the batch has three times as many sequences as clusters of that size run at once (sequences
    // in other modes leave at once, so a mixed batch needs a third to a half of them): then eight.  Budgeted batch of 32, 11 of
    // them sampling: 22.6 us with sixteen, 19 us with eight; ragged batch of 16, 8 of them sampling: 29 us and 31 us.
    if (!ctx->walk_ready) {                  // per device (= per context): more than 48 KiB of shared memory, 16-CTA clusters
        if (cudaFuncSetAttribute(accept_walk_kernel<WALK_CLUSTER>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024) != cudaSuccess ||
            cudaFuncSetAttribute(accept_walk_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024) != cudaSuccess ||
            cudaFuncSetAttribute(accept_walk_kernel<WALK_CLUSTER>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
            return HS_ERR_CUDA;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(WALK_CLUSTER * ctx->sm_count);
        cfg.blockDim = dim3(WALK_THREADS);
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = WALK_CLUSTER; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&ctx->walk_cap, accept_walk_kernel<WALK_CLUSTER>, &cfg) != cudaSuccess) {
            ctx->walk_cap = 0;
            (void)cudaGetLastError();
        }
        ctx->walk_ready = true;
    }
    const size_t esz = dtype == HS_BF16 ? 2 : 4;
    const int wc = p.batch <= 3 * ctx->walk_cap ? WALK_CLUSTER : 8;
    const size_t walk_smem = 2 * (size_t)((p.nvec + wc - 1) / wc) * 16;       // two row slices
    p.staged = ((uintptr_t)p.target % 16 == 0) && ((uintptr_t)p.draft % 16 == 0) && ((size_t)row_stride * esz % 16 == 0) &&
               walk_smem <= 160 * 1024;
    const dim3 wgrid(p.batch * wc), wcl(wc, 1, 1);
    e = wc == WALK_CLUSTER
        ? hs_launch(accept_walk_kernel<WALK_CLUSTER>, wgrid, dim3(WALK_THREADS), p.staged ? walk_smem : 0, stream, ctx->pdl, wcl, p)
        : hs_launch(accept_walk_kernel<8>, wgrid, dim3(WALK_THREADS), p.staged ? walk_smem : 0, stream, ctx->pdl, wcl, p);
    return e == cudaSuccess ? HS_OK : HS_ERR_CUDA;
}
