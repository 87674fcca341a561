// hs_entropy_quantify: two launches.
//
// quantify_cluster_kernel  Few rows (at most half as many as SMs): a row is cut into parts, one CTA each, that merge as a
//     thread-block cluster.
// quantify_warp_kernel     Many rows (row_warps.cuh): every warp of the device takes an equal share of the matrix on its own.
//     Both fold four 16-byte vectors per lane at a time: packed maximum, then sum e^(x-ref) and sum x e^(x-ref) with the
//     exponent's multiply-add and the two sums as packed fp32 pairs.  Top-K without sorting: maxima of disjoint sets (lanes,
//     half-warps) are distinct logits, so the K-th largest of 32 of them bounds the K-th largest logit of a part; the few
//     cells that reach the bound are read again and their logits ranked.  The parts of a row merge into max, log-sum-exp,
//     Shannon entropy, Top-K and the two Top-K entropies (Eq. 1 inner sum).
// tree_scores_kernel       One CTA per sequence: path confidence ln V_i (Sec. 2.2), cumulative meta-path
//     Top-K entropy Phi (Eq. 1) and the operational path P* (Sec. 4.1).  (The fused call launches the kernel
//     of stratify_prune.cu that runs the same tree stage and then prunes, in its place.)
//
// quantify_chunk_kernel (a CTA owns one chunk of one row, registers only) serves the allocation-free entry.
#include <math_constants.h>

#include <algorithm>
#include <mutex>

using std::max;
using std::min;

#include "hs_common.cuh"
#include "hs_layout.h"
#include "hs_ptx.cuh"
#include "row_rounds.cuh"
#include "tree_stage.cuh"

#define CAND_CAP 512

#define QS_THREADS 512                        // cluster kernel: sixteen warps
#define QS_ITEM_VECS 2048                     // vectors per item: 32 KiB, four per thread
#define QS_SLOTS 6                            // items a CTA has room for
#define QS_ITEM_BYTES (QS_ITEM_VECS * 16 + QS_THREADS * 4 + QS_THREADS)     // an item, every thread's maximum of it, its cells to read again
#define QS_SMEM_BYTES(items) ((items) * QS_ITEM_BYTES + 128)

struct QuantParams {
    const void* logits;
    int64_t row_stride;
    int vocab;
    int nvec;        // 16-byte vectors per row, the last one may be partial
    int chunks;      // chunk kernel: CTAs per row
    int chunk_vecs;  // chunk kernel: vectors per chunk
    int per;         // cluster kernel: vectors per part; warp kernel: places of the stream per share
    int split;       // cluster kernel: parts per row = cluster size
    int extra;       // warp kernel: places ahead of every row
    int rows;
    int batch;
    const int* node_off;
    const int* parent;
    const int* token;
    hs_quant_out out;
    float4* part_stats;             // {max, sum e, sum e*x, -} per partial
    unsigned long long* part_keys;  // HS_MAX_TOPK keys per partial
    int* row_cnt;
    int K, d_base, phi_mode, pstar_mode, entropy_mode, is_bf16;
    int inv_k;       // ceil(2^16 / K): i / K = i * inv_k >> 16 for i < 128
    int prefetch;    // the rows may be fetched before the dependency wait (the caller vouches that they are complete)
    int* err;        // sticky device error word (a bounded wait that expired)
};

// Rank candidates s_cand[0..n) by key (all distinct, 0 = empty) and write the K best to s_top (zeroed before).
__device__ __forceinline__ void rank_select(const unsigned long long* s_cand, int n, int K,
                                            unsigned long long* s_top, int tid, int nthr) {
    for (int t = tid; t < n; t += nthr) {
        unsigned long long k = s_cand[t];
        if (k == 0ull) continue;
        int rank = 0;
        for (int j = 0; j < n; ++j) rank += (s_cand[j] > k);
        if (rank < K) s_top[rank] = k;
    }
}

// The same by whole warps: warp w takes candidates w, w + nwarp, ...; the 32 lanes compare 32 others at a time.
__device__ __forceinline__ void rank_select_warps(const unsigned long long* s_cand, int n, int K,
                                                  unsigned long long* s_top, int warp, int lane, int nwarp) {
    for (int c = warp; c < n; c += nwarp) {
        const unsigned long long k = s_cand[c];
        if (k == 0ull) continue;
        int rank = 0;
        for (int j0 = 0; j0 < n && rank < K; j0 += 32) {
            const int j = j0 + lane;
            rank += __popc(__ballot_sync(HS_FULL_MASK, j < n && s_cand[j] > k));
        }
        if (rank < K && lane == 0) s_top[rank] = k;
    }
}

// barrier over the first `nthr` threads of the CTA (a multiple of 32); id 0 is __syncthreads' own
__device__ __forceinline__ void bar_sync(int id, int nthr) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthr) : "memory");
}

// Cold path of the Top-K: K rounds of "largest key below the previous winner" over vectors [v0, v1) of a row,
// read from global memory by `nthr` threads (barrier `bar`).  Exact for any number of ties; -inf logits are no
// candidates.  s_red: one slot per warp.
template <bool BF16>
__device__ __noinline__ void topk_by_rounds(const char* rowp, int v0, int v1, int vocab, int K,
                                            unsigned long long* s_top, unsigned long long* s_red,
                                            int tid, int nthr, int bar) {
    constexpr int VE = BF16 ? 8 : 4;
    const int lane = tid & 31, warp = tid >> 5, nwarp = nthr >> 5;
    unsigned long long last = ~0ull;
    for (int r = 0; r < K; ++r) {
        unsigned long long best = 0ull;
        for (int v = v0 + tid; v < v1; v += nthr) {
            uint4 dv = __ldg((const uint4*)(rowp) + v);
            float x[8];
            unpack<BF16>(dv, x);
#pragma unroll
            for (int e = 0; e < VE; ++e) {
                if (v * VE + e < vocab && x[e] > -CUDART_INF_F) {
                    unsigned long long k = make_key(x[e], v * VE + e);
                    if (k < last && k > best) best = k;
                }
            }
        }
        best = warp_max_u64(best);
        if (lane == 0) s_red[warp] = best;
        bar_sync(bar, nthr);
        best = s_red[0];
        for (int w = 1; w < nwarp; ++w) best = s_red[w] > best ? s_red[w] : best;
        if (tid == 0) s_top[r] = best;
        last = best;
        bar_sync(bar, nthr);
        if (best == 0ull) break;
    }
}

// One warp: the statistics of a whole row from its maximum M, {sum e^(x-R), sum x e^(x-R)} and its K best keys (`key`:
// lane i has the i-th, 0 = none): log-sum-exp, Shannon entropy, Top-K values and token ids, the entropy of the renormalised
// Top-K probabilities (Eq. 1 inner sum) and the truncated variant.
__device__ __forceinline__ void finalize_row(const QuantParams& p, int row, float M, float R, float S, float U,
                                             unsigned long long key, int lane) {
    const int K = p.K;
    const float lse = R + logf(S);
    const float H = lse - U / S;
    if (lane >= K) key = 0ull;
    const bool valid = key != 0ull;
    const float tv = valid ? key_value(key) : 0.f;
    const float t0 = __shfl_sync(HS_FULL_MASK, tv, 0);
    const float pv = valid ? expf(tv - lse) : 0.f;
    const float z = valid ? expf(tv - t0) : 0.f;
    float itr = valid ? -pv * (tv - lse) : 0.f, Z = z, zt = valid ? z * (tv - t0) : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {                           // three sums side by side
        itr += __shfl_xor_sync(HS_FULL_MASK, itr, o);
        Z += __shfl_xor_sync(HS_FULL_MASK, Z, o);
        zt += __shfl_xor_sync(HS_FULL_MASK, zt, o);
    }
    const float itk = logf(Z) - zt / Z;
    if (lane < K) {
        p.out.topk_val[(size_t)row * K + lane] = valid ? tv : -CUDART_INF_F;
        p.out.topk_idx[(size_t)row * K + lane] = valid ? key_index(key) : -1;
    }
    if (lane == 0) {
        p.out.row_max[row] = M;
        p.out.row_lse[row] = lse;
        p.out.h_full[row] = fmaxf(H, 0.f);
        p.out.i_topk[row] = fmaxf(itk, 0.f);
        p.out.i_trunc[row] = itr;
    }
}

// K-th largest of the warp's 32 values (one per lane), -inf if fewer than K are above -inf.  K rounds of a
// warp-wide maximum that retires one holder of the maximum per round (ties count one by one).
__device__ __forceinline__ float warp_kth_largest(float v, int K, int lane) {
    unsigned int ob = (v > -CUDART_INF_F) ? float_order_bits(v) : 0u;
    unsigned int mx = 0u;
    for (int i = 0; i < K; ++i) {
        mx = __reduce_max_sync(HS_FULL_MASK, ob);
        const unsigned int holders = __ballot_sync(HS_FULL_MASK, ob == mx);
        if (lane == __ffs(holders) - 1) ob = 0u;
    }
    return mx ? order_bits_float(mx) : -CUDART_INF_F;
}

#include "row_warps.cuh"

// ================================================================================================================
// The cluster kernel: few rows (at most half as many as SMs)
// ================================================================================================================
// Every row is cut into the same number of parts (at most eight, the portable cluster size), one CTA of 16 warps per part;
// the CTAs of a row are one thread-block cluster.  A part is at most QS_SLOTS items of 32 KiB, all of which are requested
// at once, a warp each, by bulk copies into shared memory of their own (with prefetch ahead of the dependency wait), so the pass is a chain
// of latencies, not a stream: items as they land, one bound for the Top-K of the part from the CTA's 32 half-warp maxima, the
// few cells that reach it read again from shared memory, eight at once, and from there one warp alone: candidates ranked by counting, the parts
// merged in the shared memory of the row's first CTA (asynchronous remote stores; the other CTAs leave at once).
// What it is bound by: 60 rows of 128256 bf16 take 14 k clocks behind the dependency wait (were 19 k), 7.5 k of them until the last
// item is reduced (128 KiB per SM), the rest dependent shared-memory reads and shuffles.  One thread that asked for all items with the CTA
// waiting behind it cost 2.5 k, items unrolled over the slots (34 KB of code instead of 82) and merges by all 16 warps
// between barriers the rest.  One greedy step of an 8B-shaped model 38.4 -> 36.2 us, of 32000 fp32 logits 30.1 -> 27.9.
// At most 72 registers per thread (and 64 where the logits are fp32: two CTAs of up to three items then share an SM, which clusters of five need,
// whose 28 do not find five SMs of a GPC each: ten levels of 28 rows of 85645 fp32 logits 141 us, with one CTA per SM 166): the CTA then fits into the register file beside a CTA of the kernel ahead that is still at work on
// the same SM (in a decode loop: the CTA that walks the accepted path of the step before).
// {ref, sum e, sum x e, max} of the first N lanes (N a power of two; lanes past the last one hold no values) as one, known to lanes 0 .. N - 1
template <int N>
__device__ __forceinline__ float4 merge_stats(float4 v) {
    float R = v.x, M = v.w;
#pragma unroll
    for (int o = N / 2; o > 0; o >>= 1) {
        R = fmaxf(R, __shfl_xor_sync(HS_FULL_MASK, R, o));
        M = fmaxf(M, __shfl_xor_sync(HS_FULL_MASK, M, o));
    }
    const float f = v.x == -CUDART_INF_F ? 0.f : ex2f((v.x - R) * LOG2E);
    float S = v.y * f, U = v.z * f;
#pragma unroll
    for (int o = N / 2; o > 0; o >>= 1) {
        S += __shfl_xor_sync(HS_FULL_MASK, S, o);
        U += __shfl_xor_sync(HS_FULL_MASK, U, o);
    }
    return make_float4(R, S, U, M);
}

template <bool BF16>
__global__ void __maxnreg__(BF16 ? 72 : 64) quantify_cluster_kernel(const __grid_constant__ QuantParams p) {
    constexpr int VE = BF16 ? 8 : 4;
    constexpr int NW = QS_THREADS / 32;
    extern __shared__ __align__(128) unsigned char s_dyn[];
    __shared__ unsigned long long s_full[QS_SLOTS], s_merge;
    __shared__ __align__(16) unsigned long long s_list[CAND_CAP];
    __shared__ unsigned long long s_top[HS_MAX_TOPK], s_red[NW];
    __shared__ __align__(16) float s_gm[32];
    __shared__ float4 s_wstat[NW];                               // {ref, sum e, sum x e, max} per warp
    __shared__ float4 s_stat;                                    //   and of the part
    __shared__ int s_cnt;
    __shared__ __align__(16) unsigned long long s_ck[8][HS_MAX_TOPK];   // first CTA of a row: the parts' Top-K keys
    __shared__ __align__(16) float4 s_cs[8];                            //   and their {ref, sum e, sum x e, max}

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int parts = p.split, row = blockIdx.x / parts, part = blockIdx.x - row * parts;
    const int sv0 = min(part * p.per, p.nvec), sv1 = min(sv0 + p.per, p.nvec);
    const int nit = (sv1 - sv0 + QS_ITEM_VECS - 1) / QS_ITEM_VECS;
    const char* rowp = (const char*)p.logits + (size_t)row * p.row_stride * (BF16 ? 2 : 4);
    const unsigned int slots0 = (smem_u32(s_dyn) + 127u) & ~127u;
    const uint4* slots = reinterpret_cast<const uint4*>(s_dyn + (slots0 - smem_u32(s_dyn)));
    float* s_cm = reinterpret_cast<float*>(s_dyn + (slots0 - smem_u32(s_dyn)) + nit * QS_ITEM_VECS * 16);      // [nit][QS_THREADS] maxima
    unsigned char* s_hit = reinterpret_cast<unsigned char*>(s_cm + nit * QS_THREADS) + warp * nit * 32;        // this warp's cells: item * 32 + lane
    const int K = p.K;

    if (tid == 0) {
        for (int s = 0; s < nit; ++s) mbar_init(smem_u32(&s_full[s]), 1);
        mbar_init(smem_u32(&s_merge), 1);
        if (part == 0 && parts > 1) mbar_expect_tx(smem_u32(&s_merge), (unsigned int)(parts - 1) * (16u + HS_MAX_TOPK * 8u));
        mbar_init_fence();
        s_cnt = 0;
    }
    if (tid < HS_MAX_TOPK) s_top[tid] = 0ull;
    __syncthreads();
    // First half of a cluster barrier: when it completes every CTA of the cluster runs with its barrier initialised, and its
    // shared memory may be written from outside.
    if (parts > 1) cluster_arrive();
    // The tree stage behind this kernel may start once every CTA has passed this point.  Without prefetch that is behind
    // the dependency wait, so whatever was written ahead of the call is complete by then and the tree stage may read its
    // inputs (not this kernel's results) without waiting.
    if (!p.prefetch) pdl_wait();
    pdl_launch_dependents();
    // A warp per item asks for it (one thread for all of them, with the CTA waiting behind it: 1 us).
    if (warp < nit && lane == 0) {
        const int len = min(QS_ITEM_VECS, sv1 - sv0 - warp * QS_ITEM_VECS);
        mbar_expect_tx(smem_u32(&s_full[warp]), (unsigned int)len * 16u);
        bulk_load(slots0 + (unsigned int)warp * (QS_ITEM_VECS * 16), rowp + (size_t)(sv0 + warp * QS_ITEM_VECS) * 16,
                  (unsigned int)len * 16u, smem_u32(&s_full[warp]));
    }
    __syncwarp();

    // ---- the part's items (a loop that stays one: its body unrolled over the slots is fetched once per item) ---------------
    const unsigned int ninf = BF16 ? 0xff80ff80u : 0xff800000u;
    float ref = -CUDART_INF_F, nref = 0.f, lm = -CUDART_INF_F;
    float2 s2 = make_float2(0.f, 0.f), u2 = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int it = 0; it < nit; ++it) {
        const int len = min(QS_ITEM_VECS, sv1 - sv0 - it * QS_ITEM_VECS);
        mbar_wait(smem_u32(&s_full[it]), 0u, p.err);
        __syncwarp();
        const uint4* st = slots + it * QS_ITEM_VECS;
        uint4 d[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int vl = tid + j * QS_THREADS;
            d[j] = vl < len ? st[vl] : make_uint4(ninf, ninf, ninf, ninf);
        }
        const int last = p.nvec - 1 - (sv0 + it * QS_ITEM_VECS);              // the row's last vector may run past vocab
        if (last < len && p.nvec * VE != p.vocab) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (tid + j * QS_THREADS == last) mask_tail<BF16>(d[j], p.nvec - 1, p.vocab);
        }
        float rm;
        fold_round<BF16>(d, ref, nref, s2, u2, rm);
        s_cm[it * QS_THREADS + tid] = rm;
        lm = fmaxf(lm, rm);
    }
    // ---- Top-K of the part: bound, candidates -------------------------------------------------------------------------
    {
        float hm = lm;
        hm = fmaxf(hm, __shfl_xor_sync(HS_FULL_MASK, hm, 1));
        hm = fmaxf(hm, __shfl_xor_sync(HS_FULL_MASK, hm, 2));
        hm = fmaxf(hm, __shfl_xor_sync(HS_FULL_MASK, hm, 4));
        hm = fmaxf(hm, __shfl_xor_sync(HS_FULL_MASK, hm, 8));
        if ((lane & 15) == 0) s_gm[warp * 2 + (lane >> 4)] = hm;
        const float wm = fmaxf(hm, __shfl_xor_sync(HS_FULL_MASK, hm, 16));
        const float ws = warp_sum(s2.x + s2.y), wu = warp_sum(u2.x + u2.y);
        if (lane == 0) s_wstat[warp] = make_float4(ref, ws, wu, wm);
    }
    __syncthreads();
    float tau;
    {
        const float w = s_gm[lane];
        int ge = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float4 f4 = reinterpret_cast<const float4*>(s_gm)[i];
            ge += (f4.x >= w) + (f4.y >= w) + (f4.z >= w) + (f4.w >= w);
        }
        // (maxima of disjoint sets are distinct logits)
        tau = order_bits_float(__reduce_max_sync(HS_FULL_MASK, float_order_bits(ge >= K ? w : -CUDART_INF_F)));
    }
    // The cells (a thread's 4 vectors of an item) that reach the bound are listed, then read again, a vector per lane: eight cells at once.
    int nhit = 0;
#pragma unroll 1
    for (int it = 0; it < nit; ++it) {
        const float cm = s_cm[it * QS_THREADS + tid];
        const bool hit = cm >= tau && cm > -CUDART_INF_F;
        const unsigned int b = __ballot_sync(HS_FULL_MASK, hit);
        if (hit) s_hit[nhit + __popc(b & ((1u << lane) - 1u))] = (unsigned char)(it * 32 + lane);
        nhit += __popc(b);
    }
    __syncwarp();
#pragma unroll 1
    for (int h = lane >> 2; h < nhit; h += 8) {
        const int cell = s_hit[h], vl = (cell >> 5) * QS_ITEM_VECS + warp * 32 + (cell & 31) + (lane & 3) * QS_THREADS, v = sv0 + vl;
        if (v >= sv1) continue;
        float x[8];
        unpack<BF16>(slots[vl], x);
        unsigned int m = 0u;
#pragma unroll
        for (int e = 0; e < VE; ++e) m |= (x[e] >= tau && x[e] > -CUDART_INF_F && v * VE + e < p.vocab) ? 1u << e : 0u;
        for (; m; m &= m - 1) {
            const int e = __ffs(m) - 1, sl = atomicAdd(&s_cnt, 1);
            const unsigned char* vp = reinterpret_cast<const unsigned char*>(slots + vl);
            const float xe = BF16 ? __uint_as_float((unsigned int)reinterpret_cast<const unsigned short*>(vp)[e] << 16)
                                  : reinterpret_cast<const float*>(vp)[e];
            if (sl < CAND_CAP) s_list[sl] = make_key(xe, v * VE + e);
        }
    }
    if (warp == NW - 1) {                                        // the warps' (ref, s, u, max) in a fixed order
        const float4 t = merge_stats<NW>(lane < NW ? s_wstat[lane] : make_float4(-CUDART_INF_F, 0.f, 0.f, -CUDART_INF_F));
        if (lane == 0) s_stat = t;
    }
    __syncthreads();                                             // all candidates are pushed
    const int ncand = s_cnt;
    if (ncand > 64) {
        if (ncand <= CAND_CAP) rank_select_warps(s_list, ncand, K, s_top, warp, lane, NW);
        else topk_by_rounds<BF16>(rowp, sv0, sv1, p.vocab, K, s_top, s_red, tid, QS_THREADS, 1);   // heavy ties
        __syncthreads();                                         // the Top-K is complete
    }
    // ---- the rest is one warp's -----------------------------------------------------------------------------------------
    // (and of one or three more in the first CTA of a row, which rank the keys of up to eight parts)
    const int nw = part == 0 && parts > 1 ? (parts * K + 31) / 32 : 1;
    if (warp >= nw) {
        if (parts > 1) cluster_wait();
        return;
    }
    if (warp == 0 && ncand <= 64) {                              // (the usual case: ranked by counting, two keys per shared-memory read)
        if (lane == 0) s_list[ncand] = 0ull;
        __syncwarp();
        for (int i = lane; i < ncand; i += 32) {
            const unsigned long long k = s_list[i];
            int rank = 0;
#pragma unroll 4
            for (int j = 0; j < ncand; j += 2) {
                const ulonglong2 two = *reinterpret_cast<const ulonglong2*>(&s_list[j]);
                rank += (two.x > k) + (two.y > k);
            }
            if (rank < K) s_top[rank] = k;
        }
        __syncwarp();
    }
    float4 st = s_stat;
    unsigned long long key = warp == 0 && lane < K ? s_top[lane] : 0ull;
    if (parts > 1) {
        cluster_wait();                                          // (the arrival above: every CTA of the cluster runs)
        if (part != 0) {
            // this part goes into slot `part` of the first CTA of the row's cluster (shared memory alone: the kernel ahead is not waited for, or
            // the first CTA's bounded wait would count its time too; that CTA waits for it, and the grid is not complete without)
            const unsigned int bar = cluster_map_addr(smem_u32(&s_merge), 0);
            if (lane < HS_MAX_TOPK / 2) {
                const unsigned long long a = s_top[2 * lane], b = s_top[2 * lane + 1];
                st_async_v4(cluster_map_addr(smem_u32(&s_ck[part][2 * lane]), 0), (unsigned int)a, (unsigned int)(a >> 32),
                            (unsigned int)b, (unsigned int)(b >> 32), bar);
            } else if (lane == HS_MAX_TOPK / 2) {
                st_async_v4(cluster_map_addr(smem_u32(&s_cs[part]), 0), __float_as_uint(st.x), __float_as_uint(st.y), __float_as_uint(st.z),
                            __float_as_uint(st.w), bar);
            }
            return;
        }
        if (warp == 0) {
            if (lane < HS_MAX_TOPK) s_ck[0][lane] = key;
            if (lane == 0) s_cs[0] = st;
        }
        mbar_wait_cluster(smem_u32(&s_merge), 0u, p.err);
        if (nw > 1) named_bar_sync(2, nw * 32);
        else __syncwarp();
        // the K best of the parts' lists (0 behind their ends), ranked by counting
        const int i = tid;
        if (i < parts * K) {
            const int q = i * p.inv_k >> 16;
            const unsigned long long k = s_ck[q][i - q * K];
            int rank = 0;
#pragma unroll 1
            for (int o = 0; o < parts; ++o)
#pragma unroll 4
                for (int j = 0; j < K; j += 2) {                 // (the lists have an even number of places)
                    const ulonglong2 two = *reinterpret_cast<const ulonglong2*>(&s_ck[o][j]);
                    rank += (two.x > k) + (two.y > k);
                }
            if (k != 0ull && rank < K) s_top[rank] = k;          // (warp 0 has read its own part's list)
        }
        if (nw > 1) named_bar_sync(2, nw * 32);
        else __syncwarp();
        if (warp != 0) return;
        if (lane < K) key = s_top[lane];
        st = merge_stats<16>(lane < parts ? s_cs[lane] : make_float4(-CUDART_INF_F, 0.f, 0.f, -CUDART_INF_F));
    }
    if (p.prefetch) pdl_wait();                                  // from here on results go to global memory
    finalize_row(p, row, st.w, st.x, st.y, st.z, key, lane);
}


// ================================================================================================================
// Tree stage: one CTA of 128 threads per sequence, one thread per node
// ================================================================================================================
__global__ void __launch_bounds__(HS_MAX_NODES) tree_scores_kernel(const QuantParams p) {
    __shared__ TreeStageSmem sm;
    pdl_launch_dependents();
    tree_stage_cta(p, blockIdx.x, sm);
}

static void fill_common(QuantParams& p, const hs_tree_batch* tree, const void* logits, hs_dtype dtype,
                        int64_t row_stride, int32_t vocab, const hs_policy* policy, const hs_quant_out* out) {
    const int ve = hs_vec_elems(dtype);
    p.logits = logits;
    p.row_stride = row_stride;
    p.vocab = vocab;
    p.nvec = (vocab + ve - 1) / ve;
    p.chunks = 0;
    p.chunk_vecs = 0;
    p.per = 0;
    p.split = 0;
    p.extra = 0;
    p.rows = tree->n_nodes_total;
    p.batch = tree->batch;
    p.node_off = tree->node_off;
    p.parent = tree->parent;
    p.token = tree->token;
    p.out = *out;
    p.K = policy->top_k;
    p.inv_k = (65536 + p.K - 1) / p.K;
    p.d_base = policy->d_base;
    p.phi_mode = policy->phi_mode;
    p.pstar_mode = policy->pstar_mode;
    p.entropy_mode = policy->entropy_mode;
    p.is_bf16 = dtype == HS_BF16;
    p.prefetch = 0;
    p.err = nullptr;
}

// Shares of the warp kernel: equal numbers of rounds, one share per warp of the device; a row in at most QW_MAX_SEGS of
// them, and no more shares than the workspace has partials for.
static hs_status launch_warps(hs_ctx* ctx, QuantParams& p, hs_dtype dtype, cudaStream_t stream) {
    if (!ctx->warps_ready) {
        if (cudaFuncSetAttribute(quantify_warp_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)QW_SMEM_BYTES) != cudaSuccess ||
            cudaFuncSetAttribute(quantify_warp_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)QW_SMEM_BYTES) != cudaSuccess)
            return HS_ERR_CUDA;
        ctx->warps_ready = true;
    }
    p.extra = QW_ROW_END;
    const long long rr = (p.nvec + ROUND_VECS - 1) / ROUND_VECS, total = (rr + p.extra) * p.rows;
    const long long room = (long long)((ctx->scratch_bytes - 256) / (2 * (sizeof(float4) + HS_MAX_TOPK * 8)));
    const long long shares = min((long long)ctx->sm_count * QW_WARPS, room);
    if (ctx->scratch_bytes < 512 || shares < ctx->sm_count / 2) return HS_ERR_WORKSPACE;
    const long long per = max((total + shares - 1) / shares, (rr + QW_MAX_SEGS - 3) / (QW_MAX_SEGS - 2));
    p.per = (int)per;
    const int used = (int)((total + per - 1) / per);
    p.part_stats = (float4*)ctx->scratch;
    p.part_keys = (unsigned long long*)(ctx->scratch + hs_align_up((size_t)2 * used * sizeof(float4), 256));
    const dim3 grid((used + QW_WARPS - 1) / QW_WARPS), one(1, 1, 1);
    cudaError_t e = dtype == HS_BF16
        ? hs_launch(quantify_warp_kernel<true>, grid, dim3(QW_THREADS), QW_SMEM_BYTES, stream, ctx->pdl, one, p)
        : hs_launch(quantify_warp_kernel<false>, grid, dim3(QW_THREADS), QW_SMEM_BYTES, stream, ctx->pdl, one, p);
    return e == cudaSuccess ? HS_OK : HS_ERR_CUDA;
}

hs_status hs_launch_quantify(hs_ctx* ctx, const hs_tree_batch* tree, const void* logits, hs_dtype dtype,
                             int64_t row_stride, int32_t vocab, const hs_policy* policy,
                             const hs_quant_out* out, cudaStream_t stream, bool with_tree_stage) {
    QuantParams p;
    fill_common(p, tree, logits, dtype, row_stride, vocab, policy, out);
    if (p.nvec > QS_ITEM_VECS * 64) return HS_ERR_SHAPE;            // vocabulary beyond 2^20 bf16 / 2^19 fp32 logits
    p.row_cnt = ctx->counters + HS_CNT_QUANT_ROW;
    p.err = ctx->counters + HS_CNT_ERROR;
    p.prefetch = (ctx->prefetch & HS_PREFETCH_LOGITS) != 0;
    // With at most half as many rows as SMs the rows are cut into parts, one CTA each (74 rows of 128256 bf16: 10.3 us,
    // the warp kernel 12.9 us); from there on a row would have an SM to itself (24 us at 75 rows).
    int parts = p.rows <= ctx->sm_count / 2 ? min(ctx->sm_count / p.rows, 8) : 0;
    while (parts > 1 && p.nvec / parts < 256) --parts;              // parts of at least 4 KiB
    const int pv = parts ? (p.nvec + parts - 1) / parts : 0;
    cudaError_t e;
    if (parts && pv <= QS_SLOTS * QS_ITEM_VECS) {
        // (The parts merge on chip and use none of it, but a workspace that was not sized for the batch stays refused: whether a call is
        // accepted does not depend on which kernel takes it.)
        if ((size_t)p.rows * parts * HS_ROW_PARTIAL_BYTES > ctx->scratch_bytes) return HS_ERR_WORKSPACE;
        if (!ctx->quant_ready) {
            if (cudaFuncSetAttribute(quantify_cluster_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, QS_SMEM_BYTES(QS_SLOTS)) != cudaSuccess ||
                cudaFuncSetAttribute(quantify_cluster_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, QS_SMEM_BYTES(QS_SLOTS)) != cudaSuccess)
                return HS_ERR_CUDA;
            ctx->quant_ready = true;
        }
        p.split = parts;
        p.per = pv;
        const size_t smem = QS_SMEM_BYTES((pv + QS_ITEM_VECS - 1) / QS_ITEM_VECS);
        e = dtype == HS_BF16
            ? hs_launch(quantify_cluster_kernel<true>, dim3(p.rows * parts), dim3(QS_THREADS), smem, stream, ctx->pdl, dim3(parts, 1, 1), p)
            : hs_launch(quantify_cluster_kernel<false>, dim3(p.rows * parts), dim3(QS_THREADS), smem, stream, ctx->pdl, dim3(parts, 1, 1), p);
        if (e != cudaSuccess) return HS_ERR_CUDA;
    } else {
        const hs_status st = launch_warps(ctx, p, dtype, stream);
        if (st != HS_OK) return st;
    }
    if (!with_tree_stage) return HS_OK;              // (the caller launches the kernel that also prunes)
    e = hs_launch(tree_scores_kernel, dim3(p.batch), dim3(HS_MAX_NODES), 0, stream, ctx->pdl, dim3(1, 1, 1), p);
    return e == cudaSuccess ? HS_OK : HS_ERR_CUDA;
}

// ================================================================================================================
// The chunk kernel: a CTA owns one chunk of one row (at most 256 * 8 vectors), everything in registers: 16-byte
// coalesced loads that are all issued before the first use, max / sum e^x / sum x e^x by warp shuffles, the chunk's
// Top-K from the K-th largest of 32 group maxima as the bound; the last chunk of a row to arrive merges the row.
// ================================================================================================================
template <bool BF16>
__global__ void __launch_bounds__(HS_ROW_THREADS, 2) quantify_chunk_kernel(const QuantParams p) {
    constexpr int VE = BF16 ? 8 : 4;
    constexpr int VPT = HS_ROW_VPT;
    __shared__ unsigned long long s_cand[CAND_CAP];
    __shared__ unsigned long long s_top[HS_MAX_TOPK];
    __shared__ unsigned long long s_red[8];
    __shared__ float s_gm[32];
    __shared__ float s_w[8][3];
    __shared__ int s_cnt;
    __shared__ int s_flag;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int chunk = blockIdx.x, row = blockIdx.y;
    const int K = p.K;
    const char* rowp = (const char*)p.logits + (size_t)row * p.row_stride * (BF16 ? 2 : 4);
    const int v0 = chunk * p.chunk_vecs;
    const int v1 = min(v0 + p.chunk_vecs, p.nvec);

    if (tid < HS_MAX_TOPK) s_top[tid] = 0ull;
    if (tid == 0) s_cnt = 0;

    const unsigned int ninf = BF16 ? 0xff80ff80u : 0xff800000u;
    uint4 d[VPT];
    pdl_launch_dependents();
    pdl_wait();
#pragma unroll
    for (int j = 0; j < VPT; ++j) {
        int v = v0 + tid + j * HS_ROW_THREADS;
        d[j] = (v < v1) ? __ldcs((const uint4*)(rowp) + v) : make_uint4(ninf, ninf, ninf, ninf);
    }
    // ---- maxima ---------------------------------------------------------------------------
    float vmax[VPT];
    float tmax = -CUDART_INF_F;
#pragma unroll
    for (int j = 0; j < VPT; ++j) {
        float x[8];
        unpack<BF16>(d[j], x);
        int v = v0 + tid + j * HS_ROW_THREADS;
        if (v == p.nvec - 1) {                       // the row's last vector may run past vocab
#pragma unroll
            for (int e = 0; e < VE; ++e)
                if (v * VE + e >= p.vocab) x[e] = -CUDART_INF_F;
        }
        float m = x[0];
#pragma unroll
        for (int e = 1; e < VE; ++e) m = fmaxf(m, x[e]);
        vmax[j] = m;
        tmax = fmaxf(tmax, m);
    }
    // ---- sums relative to the thread's own maximum ------------------------------------------
    const float nml = (tmax == -CUDART_INF_F) ? 0.f : -tmax * LOG2E;
    float s = 0.f, u = 0.f;
#pragma unroll
    for (int j = 0; j < VPT; ++j) {
        float x[8];
        unpack<BF16>(d[j], x);
        int v = v0 + tid + j * HS_ROW_THREADS;
        if (v == p.nvec - 1) {
#pragma unroll
            for (int e = 0; e < VE; ++e)
                if (v * VE + e >= p.vocab) x[e] = -CUDART_INF_F;
        }
#pragma unroll
        for (int e = 0; e < VE; ++e) {
            float xc = fmaxf(x[e], -1e30f);
            float ev = ex2f(fmaf(xc, LOG2E, nml));
            s += ev;
            u = fmaf(ev, xc, u);
        }
    }
    // ---- warp / block reduction of (max, s, u) ------------------------------------------------
    {
        float wm = warp_max(tmax);
        float f = (tmax == -CUDART_INF_F) ? 0.f : ex2f((tmax - wm) * LOG2E);
        float ws = warp_sum(s * f), wu = warp_sum(u * f);
        if (lane == 0) { s_w[warp][0] = wm; s_w[warp][1] = ws; s_w[warp][2] = wu; }
        float g = tmax;
        g = fmaxf(g, __shfl_xor_sync(HS_FULL_MASK, g, 1));
        g = fmaxf(g, __shfl_xor_sync(HS_FULL_MASK, g, 2));
        g = fmaxf(g, __shfl_xor_sync(HS_FULL_MASK, g, 4));
        if ((lane & 7) == 0) s_gm[warp * 4 + (lane >> 3)] = g;
    }
    __syncthreads();
    if (warp == 0) {       // the eight warps' (max, s, u): lanes 0..7 of warp 0, shuffle reductions
        const float wm = lane < 8 ? s_w[lane & 7][0] : -CUDART_INF_F;
        float M = wm;
        M = fmaxf(M, __shfl_xor_sync(HS_FULL_MASK, M, 1));
        M = fmaxf(M, __shfl_xor_sync(HS_FULL_MASK, M, 2));
        M = fmaxf(M, __shfl_xor_sync(HS_FULL_MASK, M, 4));
        const float f = (lane >= 8 || wm == -CUDART_INF_F) ? 0.f : ex2f((wm - M) * LOG2E);
        float S = s_w[lane & 7][1] * f, U = s_w[lane & 7][2] * f;
        // the serial order w = 0..7 of the sum is kept (the result does not depend on the launch shape)
        float St = 0.f, Ut = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            St += __shfl_sync(HS_FULL_MASK, S, w);
            Ut += __shfl_sync(HS_FULL_MASK, U, w);
        }
        if (lane == 0) p.part_stats[(size_t)row * p.chunks + chunk] = make_float4(M, St, Ut, 0.f);
    }
    // ---- Top-K of the chunk -------------------------------------------------------------------
    const float tau = warp_kth_largest(s_gm[lane], K, lane);   // K-th largest group maximum
    if (tmax >= tau && tmax > -CUDART_INF_F) {
#pragma unroll
        for (int j = 0; j < VPT; ++j) {
            if (vmax[j] >= tau) {
                float x[8];
                unpack<BF16>(d[j], x);
                int base = (v0 + tid + j * HS_ROW_THREADS) * VE;
#pragma unroll
                for (int e = 0; e < VE; ++e) {
                    if (x[e] >= tau && x[e] > -CUDART_INF_F && base + e < p.vocab) {
                        int slot = atomicAdd(&s_cnt, 1);
                        if (slot < CAND_CAP) s_cand[slot] = make_key(x[e], base + e);
                    }
                }
            }
        }
    }
    __syncthreads();
    const int ncand = s_cnt;
    if (ncand <= CAND_CAP) {
        rank_select(s_cand, ncand, K, s_top, tid, HS_ROW_THREADS);
    } else {
        // Heavy ties (e.g. a constant row): K rounds of "largest key below the previous one",
        // re-reading the chunk from global memory (cold path).
        topk_by_rounds<BF16>(rowp, v0, v1, p.vocab, K, s_top, s_red, tid, HS_ROW_THREADS, 0);
    }
    __syncthreads();
    if (tid < HS_MAX_TOPK)
        p.part_keys[((size_t)row * p.chunks + chunk) * HS_MAX_TOPK + tid] = (tid < K) ? s_top[tid] : 0ull;

    // ---- the last chunk of this row merges -----------------------------------------------
    // (the CTA's stores are ordered before thread 0's fence by the barrier, the fence before its arrival)
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        s_flag = (atomicAdd(&p.row_cnt[row], 1) == p.chunks - 1);
        __threadfence();
    }
    __syncthreads();
    if (!s_flag) return;
    const int nk = p.chunks * HS_MAX_TOPK;     // <= CAND_CAP, checked by the launcher
    for (int t = tid; t < nk; t += HS_ROW_THREADS)
        s_cand[t] = __ldcg(&p.part_keys[(size_t)row * p.chunks * HS_MAX_TOPK + t]);
    if (tid < HS_MAX_TOPK) s_top[tid] = 0ull;
    __syncthreads();
    rank_select(s_cand, nk, K, s_top, tid, HS_ROW_THREADS);
    __syncthreads();
    if (warp == 0) {
        float m = -CUDART_INF_F, cs = 0.f, cu = 0.f;
        if (lane < p.chunks) {
            float4 st = __ldcg(&p.part_stats[(size_t)row * p.chunks + lane]);
            m = st.x; cs = st.y; cu = st.z;
        }
        float M = warp_max(m);
        float f = (m == -CUDART_INF_F) ? 0.f : ex2f((m - M) * LOG2E);
        float S = warp_sum(cs * f), U = warp_sum(cu * f);
        finalize_row(p, row, M, M, S, U, lane < K ? s_top[lane] : 0ull, lane);
        if (lane == 0) p.row_cnt[row] = 0;                 // ready for the next launch
    }
}

// ---- hs_entropy_quantify_static: the same pass without any allocated workspace -------------------------------
//
// Some hosts of this library may not allocate device memory at all: a serving process that hands
// its whole memory budget to one arena at start-up, or code running under a capture / real-time
// rule that forbids cudaMalloc.  For them the chunk partials and arrival counters of the pass live
// in one fixed array that is part of the library image, so every GPU that loads the library carries
// HS_STATIC_SCRATCH_BYTES of it until the process exits.
#define HS_STATIC_MAX_CHUNKS 16
#define HS_STATIC_COUNTER_BYTES 2048    // HS_STATIC_MAX_ROWS ints (one arrival counter per row), rounded up
#define HS_STATIC_STATS_BYTES (HS_STATIC_MAX_ROWS * HS_STATIC_MAX_CHUNKS * 16)
#define HS_STATIC_KEYS_BYTES (HS_STATIC_MAX_ROWS * HS_STATIC_MAX_CHUNKS * HS_MAX_TOPK * 8)
#define HS_STATIC_SCRATCH_BYTES (HS_STATIC_COUNTER_BYTES + HS_STATIC_STATS_BYTES + HS_STATIC_KEYS_BYTES)
#define HS_STATIC_MAX_DEVICES 64

static __device__ __align__(256) unsigned char g_static_scratch[HS_STATIC_SCRATCH_BYTES];
// Device address of g_static_scratch on each device.  In host code the symbol itself is only a
// handle, never an address a kernel may use: the address is asked for once per device.
static unsigned char* g_static_addr[HS_STATIC_MAX_DEVICES];
static std::mutex g_static_mutex;

extern "C" hs_status hs_entropy_quantify_static(const hs_tree_batch* tree, const void* draft_logits, hs_dtype dtype,
                                                int64_t row_stride, int32_t vocab, const hs_policy* policy,
                                                const hs_quant_out* out, hs_stream stream_) {
    cudaStream_t stream = (cudaStream_t)stream_;
    if (!tree || !policy || !out || !draft_logits || ((uintptr_t)draft_logits & 15)) return HS_ERR_INVALID_ARG;
    if (dtype != HS_F32 && dtype != HS_BF16) return HS_ERR_INVALID_ARG;
    if (tree->batch < 1 || tree->n_nodes_total < tree->batch || !tree->node_off || !tree->parent || !tree->token)
        return HS_ERR_INVALID_ARG;
    const int ve = hs_vec_elems(dtype);
    if (vocab < 1 || row_stride < vocab || row_stride % ve != 0) return HS_ERR_INVALID_ARG;
    if (policy->top_k < 1 || policy->top_k > HS_MAX_TOPK || policy->d_base < 0 || policy->phi_mode < 0 ||
        policy->phi_mode > 1 || policy->pstar_mode < 0 || policy->pstar_mode > 1 || policy->entropy_mode < 0 ||
        policy->entropy_mode > 1)
        return HS_ERR_INVALID_ARG;
    if (!out->row_max || !out->row_lse || !out->h_full || !out->i_topk || !out->i_trunc || !out->topk_val ||
        !out->topk_idx || !out->logc || !out->score || !out->phi || !out->depth || !out->pstar_node ||
        !out->phi_star || !out->status)
        return HS_ERR_INVALID_ARG;
    const int chunks = hs_row_chunks(vocab, dtype);
    if (tree->n_nodes_total > HS_STATIC_MAX_ROWS || tree->batch > HS_STATIC_MAX_BATCH || chunks > HS_STATIC_MAX_CHUNKS)
        return HS_ERR_STATIC_LIMIT;

    int dev = -1;
    HS_CUDA_OK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= HS_STATIC_MAX_DEVICES) return HS_ERR_UNSUPPORTED;
    unsigned char* base;
    {
        std::lock_guard<std::mutex> lock(g_static_mutex);
        if (!g_static_addr[dev]) {              // first call on this device (it is the current one)
            void* sym = nullptr;
            if (cudaGetSymbolAddress(&sym, g_static_scratch) != cudaSuccess || !sym) return HS_ERR_CUDA;
            g_static_addr[dev] = (unsigned char*)sym;
        }
        base = g_static_addr[dev];
    }

    QuantParams p;
    fill_common(p, tree, draft_logits, dtype, row_stride, vocab, policy, out);
    p.chunks = chunks;
    p.chunk_vecs = (p.nvec + p.chunks - 1) / p.chunks;
    p.row_cnt = (int*)base;
    p.part_stats = (float4*)(base + HS_STATIC_COUNTER_BYTES);
    p.part_keys = (unsigned long long*)(base + HS_STATIC_COUNTER_BYTES + HS_STATIC_STATS_BYTES);
    // The array keeps whatever the previous call left: the arrival counters must start at zero.
    HS_CUDA_OK(cudaMemsetAsync(base, 0, HS_STATIC_COUNTER_BYTES, stream));
    dim3 grid(p.chunks, p.rows);
    if (dtype == HS_BF16) quantify_chunk_kernel<true><<<grid, HS_ROW_THREADS, 0, stream>>>(p);
    else quantify_chunk_kernel<false><<<grid, HS_ROW_THREADS, 0, stream>>>(p);
    if (cudaGetLastError() != cudaSuccess) return HS_ERR_CUDA;
    tree_scores_kernel<<<p.batch, HS_MAX_NODES, 0, stream>>>(p);      // (needs no scratch)
    return cudaGetLastError() == cudaSuccess ? HS_OK : HS_ERR_CUDA;
}
