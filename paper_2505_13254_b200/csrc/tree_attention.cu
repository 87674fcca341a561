// hs_tree_verify_attention (Sec. 2.2, tree-mask attention): one launch.
//
// CTA = (block of 128 query rows, KV split, sequence x kv-head).  The GQA group times the kept tree
// nodes forms the dense M dimension: query row r = node * G + g.  The KV prefix is cut into tiles of
// 64 keys that are shared out evenly over the splits; a CTA requests its first tiles by TMA
// (cp.async.bulk.tensor into 128-byte-swizzled shared memory, four stages, K and V on mbarriers of
// their own) before it waits for the kernel ahead of it in the stream if the caller vouches for the cache (it does not
// depend on the pruned tree).  The <= 128 tree keys belong to the last split; their rows may be indirect.  Behind
// prefix tiles the producer warp fetches them by tile::gather4 (plain loads by the softmax threads held up the
// longest split: 4096 tokens, 64 / 8 heads 19.6 us against 18.0, a ragged batch of 16 75.5 against 71).  S = Q K^T and
// O += P V run on the 5th-generation tensor cores (tcgen05.mma, accumulators in tensor memory) with fp32 accumulation; the softmax is the
// online (running max / running sum) form in base 2.  Prefix columns are fully visible, tree column j
// is visible to row r iff bit j of the ancestor mask of r's node is set.  The splits of one (query
// block, head) form a thread-block cluster: every CTA sends its partial (max, sum, O) from registers
// to the owner of each row by asynchronous stores through distributed shared memory;
// an owner merges its rows once all pieces have landed.  No partial ever goes to global memory and
// there is no second launch.
//
// Launches of more than one wave of such CTAs, and long prefixes, may go to tree_attn_duo.cuh, where two CTAs share an SM (see duo_splits).
#include <math_constants.h>

#include "attn_choice.h"
#include "hs_common.cuh"
#include "hs_layout.h"
#include "hs_ptx.cuh"

#define ATT_BM 128
#define ATT_BN 64
#define ATT_TILE_BYTES (ATT_BN * HS_HEAD_DIM * 2)   // 16 KiB: one K or V tile
#define ATT_STAGE_BYTES (2 * ATT_TILE_BYTES)
#define ATT_Q_BYTES (ATT_BM * HS_HEAD_DIM * 2)      // 32 KiB
#define ATT_PB_STRIDE (HS_HEAD_DIM * 2 + 16)        // bytes per row of a pushed partial: 128 bf16 of O / l, {max, sum}, padding
#define LOG2E 1.4426950408889634f
#define LN2 0.6931471805599453f

struct AttnParams {
    const __nv_bfloat16* q;
    const __nv_bfloat16* k_tree;
    const __nv_bfloat16* v_tree;
    __nv_bfloat16* out;
    float* lse_out;
    const int* n_keep;
    const int* keep_off;
    const int* keep_idx;
    const unsigned long long* anc_mask;
    const int* status;
    const int* node_off;
    const int* kv_off;
    int batch, hq, hkv, G, layout, nsplit, head_first, prefetch;
    int follow;               // of the instance that takes Q from tensor memory: FOLLOW at run time
    unsigned int inv_g;       // ceil(2^16 / G): r / G = r * inv_g >> 16 for the row numbers r < 2^11
    float scale_log2;
    int* err;
};

__device__ __forceinline__ unsigned int pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<unsigned int*>(&v);
}
// 4 x 4 transpose of 16-byte chunks over four lanes: lane q then holds chunk q of the four rows, and 64 bytes of a row leave in
// one instruction (a lane storing its own row touched 32 cache lines with every instruction).
__device__ __forceinline__ void quad_transpose(uint4 (&o)[4], int lane) {
    auto swap = [&](uint4& a, uint4& b, int m) {                  // a of the upper lane <-> b of the lower one
        const bool up = (lane & m) != 0;
        uint4 x = up ? a : b;
        x.x = __shfl_xor_sync(HS_FULL_MASK, x.x, m); x.y = __shfl_xor_sync(HS_FULL_MASK, x.y, m);
        x.z = __shfl_xor_sync(HS_FULL_MASK, x.z, m); x.w = __shfl_xor_sync(HS_FULL_MASK, x.w, m);
        if (up) a = x; else b = x;
    };
    swap(o[0], o[1], 1); swap(o[2], o[3], 1);
    swap(o[0], o[2], 2); swap(o[1], o[3], 2);
}
// acc += w * (eight bf16 values)
__device__ __forceinline__ void fma_bf16x8(float (&acc)[8], float w, uint4 v) {
    acc[0] = fmaf(w, bf16_lo(v.x), acc[0]); acc[1] = fmaf(w, bf16_hi(v.x), acc[1]);
    acc[2] = fmaf(w, bf16_lo(v.y), acc[2]); acc[3] = fmaf(w, bf16_hi(v.y), acc[3]);
    acc[4] = fmaf(w, bf16_lo(v.z), acc[4]); acc[5] = fmaf(w, bf16_hi(v.z), acc[5]);
    acc[6] = fmaf(w, bf16_lo(v.w), acc[6]); acc[7] = fmaf(w, bf16_hi(v.w), acc[7]);
}
// byte offset of (key row, 16-byte chunk 0..15 of the 128 d's) inside a swizzled 64x128 bf16 tile:
// two halves of 64 d's, rows of 128 bytes, chunk index XOR-ed with the row (the TMA 128-byte swizzle)
__device__ __forceinline__ unsigned int tile_off(int key, int chunk) {
    return (unsigned int)((chunk >> 3) * (ATT_TILE_BYTES / 2) + key * 128 + (((chunk & 7) ^ (key & 7)) << 4));
}
// same layout for the 128-row query tile
__device__ __forceinline__ unsigned int q_off(int row, int chunk) {
    return (unsigned int)((chunk >> 3) * (ATT_Q_BYTES / 2) + row * 128 + (((chunk & 7) ^ (row & 7)) << 4));
}

// prefix tiles of split `split`: the ceil(L / 64) tiles are shared out evenly, independent of the tree
__device__ __forceinline__ void prefix_range(int L, int nsplit, int split, int& t_prefix, int& t0, int& t1) {
    t_prefix = (L + ATT_BN - 1) / ATT_BN;
    const int per = (t_prefix + nsplit - 1) / nsplit;
    t0 = min(split * per, t_prefix);
    t1 = min(t0 + per, t_prefix);
}

// =====================================================================================================
// The kernel: S = Q K^T and O += P V by the 5th-generation tensor cores, accumulators in tensor
// memory.  Two softmax warpgroups run two independent online-softmax streams over the block's 128 query
// rows: warpgroup g takes the KV tiles i = g, g + 2, ... and keeps its own S buffer, P buffer, running
// (max, sum) and O accumulator; thread t of a warpgroup owns query row t (= tensor-memory lane t), so the
// softmax needs no shuffles and the two streams never wait for one another: while one exponentiates (the
// special-function unit), the other loads, masks and stores.  Three more warps give one elected thread each: the S issuer
// (S = Q K^T of tile i + 2 as soon as S of tile i is in registers; 8 instructions of K = 16, operands
// straight from the swizzled TMA tiles, Q and K are K-major; in long CTAs of some launches Q comes from tensor memory, where the
// softmax threads copy it while the first S are computed), the P V issuer (O_g += P V as soon as a P
// is written; V is the MN-major operand, the same swizzled tile as it arrived by TMA) and the TMA
// producer (a stage's K is refilled as soon as the S that read it is complete, its V once its P V is).
// A stream rescales its O in tensor memory only when a row's running maximum grows.  After the last
// tile the two streams are combined like two splits, in registers.
// =====================================================================================================
#define UM_THREADS 352                               // two softmax warpgroups + P V issuer, TMA producer, S issuer warps
#define UM_ROWS_THREADS 128
#define UM_SM_THREADS 256                            // softmax threads: row = tid & 127, stream = tid >> 7
#define UM_MAP_BYTES 1024                            // output-row map of the rows a CTA merges (<= 65 rows x 8 bytes)
#define UM_TMEM_COLS 512                             // S of stream g: columns 64 g ..; O: 128 + 128 g ..; P (bf16 pairs): 384 + 32 g ..; Q: 448 ..
#define UM_STAGES 4
// CTAs of more than ATT_Q_TILES tiles may take Q as the A operand from tensor memory (columns 448 ..) from tile UM_Q_FIRST on: see q_from_tensor_memory.
// From the third tile on instead of the ninth 4 trees of 60 nodes, 64 / 8 heads take 44.3 us for 42.9 at 4700 tokens, 140 for 124 at 16300; with the operand chosen per
// loop and not per instruction 45.2, 138: the issue of an S that leaves P V room between its instructions is part of the gain.
#define UM_Q_FIRST 8
static_assert(UM_Q_FIRST <= ATT_Q_TILES, "a CTA that takes Q from tensor memory reaches the tile that waits for it");
#define UM_WT_BYTES (66 * ATT_MAX_SPLIT * 4 + 64)    // split weights of the rows a CTA merges
#define UM_RECV_BYTES (ATT_PB_STRIDE * (ATT_BM + 2 * ATT_MAX_SPLIT))     // partials pushed by the splits of the cluster
#define UM_SMEM_BYTES (UM_STAGES * ATT_STAGE_BYTES + ATT_Q_BYTES + UM_MAP_BYTES + 1024 + 2048 + UM_WT_BYTES + UM_RECV_BYTES + 1024)

// FOLLOW: the exponents' reference follows every new row maximum over the second tile of each stream too (over the first four on long ranges): a score that was its
// row's maximum when its tile was taken has P = 2^0, which bf16 holds without error, and those are the weights that count most.  2-norm relative
// error against fp64, 10 x 60 nodes, 32 / 8 heads, plain, FOLLOW, tree_attn_duo_kernel: 1500 tokens 2.325e-3, 2.309e-3, 2.322e-3; 4096 tokens 2.3345e-3,
// 2.3195e-3, 2.3329e-3; 8192 tokens 2.339e-3, 2.332e-3, 2.334e-3.  Which launches take it, and what it costs: see wants_follow.
// QT: Q from tensor memory in CTAs of many tiles (see q_from_tensor_memory), FOLLOW at run time; other launches run an instance without that code.
template <bool FOLLOW, bool QT>
__global__ void __launch_bounds__(UM_THREADS, 1)
tree_attn_umma_kernel(const __grid_constant__ AttnParams p, const __grid_constant__ CUtensorMap tmK,
                      const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmKT,
                      const __grid_constant__ CUtensorMap tmVT) {
    extern __shared__ unsigned char smem_raw[];
    const int tid = threadIdx.x, warp = tid >> 5;
    // Sequences are taken longest prefix first (a ragged batch then ends on its short sequences, not on a long one
    // that started late): grid slot z / hkv holds the sequence of that rank by (length descending, index ascending).
    // kv_off is an array of the caller like any other: the ranking runs ahead of the dependency wait only where the caller
    // vouches for the cache and with it for its offsets.  (Both instructions come again below, without effect.)
    if (!p.prefetch) { pdl_launch_dependents(); pdl_wait(); }
    __shared__ int s_seq;
    int b = blockIdx.z / p.hkv;
    const int h = blockIdx.z % p.hkv;
    if (p.batch > 1 && p.batch <= UM_THREADS) {
        if (tid < p.batch) {
            const int len = p.kv_off[tid + 1] - p.kv_off[tid];
            int rank = 0;
            for (int j = 0; j < p.batch; ++j) {
                const int lj = p.kv_off[j + 1] - p.kv_off[j];
                rank += (lj > len || (lj == len && j < tid));
            }
            if (rank == b) s_seq = tid;
        }
        __syncthreads();
        b = s_seq;
    }
    const int split = blockIdx.y;
    const int m0 = blockIdx.x * ATT_BM;

    const unsigned int smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    unsigned char* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    const unsigned int sQ = smem_base + UM_STAGES * ATT_STAGE_BYTES;
    const unsigned int sM = sQ + ATT_Q_BYTES;                // row map, then barriers and exchange arrays
    // barriers: K-full[UM_STAGES], V-full[UM_STAGES], K-free[UM_STAGES], V-free[UM_STAGES], S-ready[2],
    // partials-received, all-MMAs-done, P-written[2], S-read[2]; then the tensor-memory base.  A parity wait can only tell the
    // current phase from the one before, so every barrier is laid out such that its next completion depends on the
    // thread that waits: a stage's barriers complete once per UM_STAGES tiles, S-ready and P-written alternate with
    // the tile's parity.
    const unsigned int bar0 = sM + UM_MAP_BYTES, bar_v = bar0 + UM_STAGES * 8, bar_ek = bar_v + UM_STAGES * 8,
                       bar_ev = bar_ek + UM_STAGES * 8;
    const unsigned int bar_s = bar_ev + UM_STAGES * 8, bar_r = bar_s + 16, bar_done = bar_r + 8,
                       bar_p = bar_done + 8, bar_sr = bar_p + 16, tslot = bar_sr + 16;
    unsigned char* gQ = smem_gen + UM_STAGES * ATT_STAGE_BYTES;
    unsigned char* gM = gQ + ATT_Q_BYTES;
    unsigned char* gR = gM + UM_MAP_BYTES + 1024 + 2048 + UM_WT_BYTES;      // partials received from the cluster
    volatile unsigned int* tslot_gen = reinterpret_cast<volatile unsigned int*>(gM + UM_MAP_BYTES + (4 * UM_STAGES + 8) * 8);
    float* s_mx = reinterpret_cast<float*>(gM + UM_MAP_BYTES + 1024);      // [2][128]: the streams' row maxima at the end
    float* s_lx = s_mx + 2 * ATT_BM;                                     // [2][128]: the streams' row sums

    // ---- with prefetch before the dependency wait: barriers, tensor memory, the first KV prefix tiles -----------------
    const int kv0 = p.kv_off[b];
    const int L = p.kv_off[b + 1] - kv0;
    int t_prefix, t0, t1;
    prefix_range(L, p.nsplit, split, t_prefix, t0, t1);
    const int np = t1 - t0;
    // one thread: K (V) of prefix tile i of this CTA into stage i % UM_STAGES; K and V complete on barriers of their own,
    // because a stage's K is free again (after S = Q K^T) two tiles before its V is (after O += P V)
    auto issue_kv = [&](int i, bool is_v) {
        const int stage = i % UM_STAGES;
        const unsigned int dst = smem_base + stage * ATT_STAGE_BYTES + (is_v ? ATT_TILE_BYTES : 0);
        const unsigned int bar = (is_v ? bar_v : bar0) + stage * 8;
        const CUtensorMap* tm = is_v ? &tmV : &tmK;
        const int tok = kv0 + (t0 + i) * ATT_BN;
        mbar_expect_tx(bar, ATT_TILE_BYTES);
        if (p.head_first) {
            tma_load_3d(dst, tm, 0, tok, h, bar);
            tma_load_3d(dst + ATT_TILE_BYTES / 2, tm, 64, tok, h, bar);
        } else {
            tma_load_3d(dst, tm, 0, h, tok, bar);
            tma_load_3d(dst + ATT_TILE_BYTES / 2, tm, 64, h, tok, bar);
        }
    };
    const int pre = min(np, UM_STAGES);
    if (warp == 9 && (tid & 31) < 2) tma_prefetch_desc((tid & 31) ? &tmVT : &tmKT);
    if (tid == 0) {
        for (int i = 0; i < 4 * UM_STAGES + 4; ++i) mbar_init(bar0 + i * 8, 1);
        mbar_init(bar_p, UM_ROWS_THREADS);               // P of a tile is written: one arrival per thread of the stream
        mbar_init(bar_p + 8, UM_ROWS_THREADS);
        mbar_init(bar_sr, UM_ROWS_THREADS);              // S of a tile is in registers: its buffer may take the next S
        mbar_init(bar_sr + 8, UM_ROWS_THREADS);
        if (p.nsplit > 1)                                // the partials of the rows this CTA will own: 128 bf16 and {max, sum} each
            mbar_expect_tx(bar_r, (unsigned int)(p.nsplit * (((split + 1) * ATT_BM + p.nsplit - 1) / p.nsplit - (split * ATT_BM + p.nsplit - 1) / p.nsplit) *
                                                 (HS_HEAD_DIM * 2 + 8)));
        mbar_init_fence();
        if (p.prefetch)                                  // the caller vouches for the cache: tiles requested ahead of the wait
            for (int i = 0; i < pre; ++i) { issue_kv(i, false); issue_kv(i, true); }
    }
    if (warp == 0) {
        tmem_alloc(tslot, UM_TMEM_COLS);
        tmem_relinquish();
    }
    pdl_launch_dependents();
    // First half of a cluster barrier: when it completes every CTA of the cluster runs with its barriers initialised, and its
    // shared memory may be written from outside.
    if (p.nsplit > 1) cluster_arrive();
    pdl_wait();                                      // the pruned tree, q, k_tree, v_tree come from upstream
    // the sequence's entries of the pruned tree in one round trip
    const int nk_b = p.n_keep[b], st_b = p.status[b], koff = p.keep_off[b];
    const int nbase = p.layout == HS_ROWS_ORIGINAL ? p.node_off[b] : 0;
    if (tid == 0 && !p.prefetch)
        for (int i = 0; i < pre; ++i) { issue_kv(i, false); issue_kv(i, true); }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const unsigned int tmem_base = *tslot_gen;
    const unsigned int lane_off = (unsigned int)((warp & 3) * 32) << 16;   // a warp reaches lanes 32 * (warp % 4) ...
    const int row = tid & (ATT_BM - 1), half = (tid >> 7) & 1;               // the thread's query row and stream
    const unsigned int tS = tmem_base, tO = tmem_base + 128, tP = tmem_base + 384, tQ = tmem_base + 448;   // (+ 64 / + 128 / + 32 columns for stream 1)

    const int nk = st_b == 0 ? nk_b : 0;
    const int M = nk * p.G;
    if (m0 >= M) {                                   // nothing to do (the same for every CTA of the cluster)
        if (tid == 0)
            for (int i = 0; i < pre; ++i) {              // no copy may outlive the CTA
                mbar_wait(bar0 + i * 8, 0u, p.err);
                mbar_wait(bar_v + i * 8, 0u, p.err);
            }
        __syncthreads();
        if (warp == 0) tmem_dealloc(tmem_base, UM_TMEM_COLS);
        if (p.nsplit > 1) cluster_wait();
        return;
    }
    // row of q / k_tree / v_tree of kept node `node` (times heads)
    auto kept_row_of = [&](int node) { return p.layout == HS_ROWS_ORIGINAL ? nbase + p.keep_idx[koff + node] : koff + node; };
    const int nt_tree = (split == p.nsplit - 1) ? (nk + ATT_BN - 1) / ATT_BN : 0;
    const int ntiles = np + nt_tree;

    // Tree tiles that open the pipeline (stages that no prefix tile uses): gathered rows by plain loads of the softmax threads, which
    // have nothing else to do yet (0.6 us less than tile::gather4).  1024 chunks of 16 bytes per matrix, swizzled stores.
    auto load_tree = [&](int i) {
        unsigned char* gK = smem_gen + i * ATT_STAGE_BYTES;
        unsigned char* gV = gK + ATT_TILE_BYTES;
        uint4 kvv[4], vvv[4];
        int row4[4];
#pragma unroll
        for (int it = 0; it < 4; ++it) {
            const int j = (i - np) * ATT_BN + ((tid + it * UM_SM_THREADS) >> 4);
            row4[it] = j < nk ? kept_row_of(j) : -1;
        }
#pragma unroll
        for (int it = 0; it < 4; ++it) {
            kvv[it] = make_uint4(0, 0, 0, 0);
            vvv[it] = make_uint4(0, 0, 0, 0);
            if (row4[it] >= 0) {
                const size_t off = ((size_t)row4[it] * p.hkv + h) * HS_HEAD_DIM + (tid & 15) * 8;
                kvv[it] = __ldg(reinterpret_cast<const uint4*>(p.k_tree + off));
                vvv[it] = __ldg(reinterpret_cast<const uint4*>(p.v_tree + off));
            }
        }
#pragma unroll
        for (int it = 0; it < 4; ++it) {
            const int c = tid + it * UM_SM_THREADS;
            *reinterpret_cast<uint4*>(gK + tile_off(c >> 4, c & 15)) = kvv[it];
            *reinterpret_cast<uint4*>(gV + tile_off(c >> 4, c & 15)) = vvv[it];
        }
    };
    // The later ones by the producer warp: four tree rows per lane of half a warp, for each of the two tree tiles.  Keys past the last one repeat it
    // (they are masked).
    int trow[2][4];
    if (warp == 9 && ntiles > np) {
#pragma unroll
        for (int k = 0; k < 8; ++k) trow[k >> 2][k & 3] = kept_row_of(min((k >> 2) * ATT_BN + (tid & 15) * 4 + (k & 3), nk - 1));
    }
    // K (V) of tree tile i (i >= np) into stage i % UM_STAGES; half a warp for each half of the columns
    auto gather_tree = [&](int i, bool is_v) {
        const int stage = i % UM_STAGES, lane = tid & 31;
        const unsigned int dst = smem_base + stage * ATT_STAGE_BYTES + (is_v ? ATT_TILE_BYTES : 0);
        const unsigned int bar = (is_v ? bar_v : bar0) + stage * 8;
        if (lane == 0) mbar_expect_tx(bar, ATT_TILE_BYTES);
        __syncwarp();
        const bool second = i > np;
        tma_gather4(dst + (lane >> 4) * (ATT_TILE_BYTES / 2) + (lane & 15) * 512, is_v ? &tmVT : &tmKT,
                    h * HS_HEAD_DIM + (lane >> 4) * 64, second ? trow[1][0] : trow[0][0], second ? trow[1][1] : trow[0][1],
                    second ? trow[1][2] : trow[0][2], second ? trow[1][3] : trow[0][3], bar);
    };

    // ---- query rows -> shared memory: 16 lanes per row (a thread fetching a row of its own touched 32 cache lines with
    // every load: 1 us of 2.3 us ahead of the first product) ------------------------------------------------------------
    if (warp < 8) {
        int qrow[8];
        uint4 qv[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int r = m0 + (tid >> 4) + 16 * i, node = (int)((unsigned int)r * p.inv_g >> 16);
            qrow[i] = r < M ? kept_row_of(node) * p.hq + h * p.G + (r - node * p.G) : -1;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
            qv[i] = qrow[i] >= 0 ? __ldg(reinterpret_cast<const uint4*>(p.q + (size_t)qrow[i] * HS_HEAD_DIM) + (tid & 15))
                                 : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int i = 0; i < 8; ++i) *reinterpret_cast<uint4*>(gQ + q_off((tid >> 4) + 16 * i, tid & 15)) = qv[i];
    }
    // this thread's own row: its ancestor mask and output row
    const int r = m0 + row;
    long long orow = -1;
    unsigned long long mk0 = 0ull, mk1 = 0ull;
    if (r < M && warp < 8) {
        const int node = (int)((unsigned int)r * p.inv_g >> 16);
        orow = (long long)kept_row_of(node) * p.hq + h * p.G + (r - node * p.G);
        mk0 = p.anc_mask[2 * (size_t)(koff + node)];
        mk1 = p.anc_mask[2 * (size_t)(koff + node) + 1];
    }
    if (warp < 8)
        for (int i = np; i < min(ntiles, UM_STAGES); ++i) load_tree(i);
    fence_proxy_async_smem();                        // generic stores -> visible to the tensor cores
    __syncthreads();

    const unsigned int idesc_qk = umma_idesc_bf16(ATT_BM, ATT_BN, false);
    const unsigned int idesc_pv = umma_idesc_bf16(ATT_BM, HS_HEAD_DIM, true);
    // Operand descriptors: the start-address field (16-byte units, low 14 bits) is the only part that varies, and no
    // shared-memory address reaches 2^18, so an offset is added to a descriptor built once.
    const unsigned long long dq0 = umma_desc_sw128(sQ, 16, 1024), dk0 = umma_desc_sw128(smem_base, 16, 1024);
    const unsigned long long dv0 = umma_desc_sw128(smem_base + ATT_TILE_BYTES, ATT_TILE_BYTES / 2, 1024);
    // the issuing warp: S = Q K^T of tile i into S buffer i & 1 (waits for K unless load_tree wrote it), then commit
    auto issue_qk = [&](int i, auto from_tmem) {
        const int stage = i % UM_STAGES;
        if (i < np || i >= UM_STAGES) mbar_wait(bar0 + stage * 8, (unsigned int)(i / UM_STAGES) & 1u, p.err);
        if (i >= 2) mbar_wait(bar_sr + (i & 1) * 8, (unsigned int)((i - 2) >> 1) & 1u, p.err);      // S of tile i - 2 is read
        __syncwarp();
        tc_fence_after_sync();
        if (!elect_one()) return;
        const unsigned long long dk = dk0 + (unsigned long long)(stage * (ATT_STAGE_BYTES >> 4));
        const unsigned int ts = tS + (i & 1) * ATT_BN;
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
            const unsigned int koffb = (ks >> 2) * (ATT_TILE_BYTES / 2) + (ks & 3) * 32;
            const unsigned int qoffb = (ks >> 2) * (ATT_Q_BYTES / 2) + (ks & 3) * 32;
            if (from_tmem(i)) umma_ts_bf16(ts, tQ + ks * 8, dk + (koffb >> 4), idesc_qk, ks > 0 ? 1u : 0u);
            else umma_ss_bf16(ts, dq0 + (qoffb >> 4), dk + (koffb >> 4), idesc_qk, ks > 0 ? 1u : 0u);
        }
        umma_commit(bar_s + (i & 1) * 8);
        if (i + UM_STAGES < ntiles) umma_commit(bar_ek + stage * 8);     // (the producer waits for it only then)
    };
    // O of stream i & 1 += P V of tile i (waits for its P, and for V likewise), then commit
    auto issue_pv = [&](int i) {
        const int stage = i % UM_STAGES;
        if (i < np || i >= UM_STAGES) mbar_wait(bar_v + stage * 8, (unsigned int)(i / UM_STAGES) & 1u, p.err);
        mbar_wait(bar_p + (i & 1) * 8, (unsigned int)(i >> 1) & 1u, p.err);   // P of tile i is written
        __syncwarp();
        tc_fence_after_sync();
        if (!elect_one()) return;
        const unsigned long long dv = dv0 + (unsigned long long)(stage * (ATT_STAGE_BYTES >> 4));
        const unsigned int tp = tP + (i & 1) * (ATT_BN / 2);
        const unsigned int to = tO + (i & 1) * HS_HEAD_DIM;
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)                       // 16 keys per instruction: two 8-key groups of V
            umma_ts_bf16(to, tp + kk * 8, dv + (kk * 2048 >> 4), idesc_pv, (i > 1 || kk > 0) ? 1u : 0u);
        umma_commit(bar_ev + stage * 8);
        // every S was read before the last P was written: all tensor-core work of this CTA is complete
        if (i == ntiles - 1) umma_commit(bar_done);
    };
    float mrun = -CUDART_INF_F, lrun = 0.f;
    const int nfollow = QT && !p.follow ? 0 : ntiles > 64 ? 8 : 4;

    // ---- KV tiles ------------------------------------------------------------------------------------------
    // The single-thread roles sit behind a branch on a warp-uniform value; all lanes run the loop and wait, and elect.sync chooses the
    // thread only for the instructions that one thread issues: the compiler then keeps loop counters, addresses and descriptors uniform.
    // (The issuing warps are what a tile waits for - with almost no arithmetic left in the softmax warps a tile took as long.  With the waits
    // inside the elected branch, timed in turn: 4 calls of 4 trees, 64 / 8 heads, 4470 - 4975 tokens 215 us, now 203; 32 calls of one tree,
    // 32 / 8 heads, 2048 tokens 380, now 366.)
    const int warp_u = __shfl_sync(HS_FULL_MASK, warp, 0);
    if (warp_u == 8) {
        // The P V issuer: O += P V of tile i as soon as its P is written.  It is short work on the streams' critical
        // path (a stream may not write P of tile i + 2 before it is complete), so it has a thread of its own that is
        // never held up behind the issue of an S.
#pragma unroll 1
        for (int i = 0; i < ntiles; ++i) {
            issue_pv(i);
            __syncwarp();
        }
    } else if (warp_u == 10) {
        // The S issuer: S of tile i + 2 as soon as the stream has S of tile i in registers, so a stream never waits
        // for its next S.
        auto ss = [](int) { return false; };                 // (from shared memory)
        if (!QT || ntiles <= ATT_Q_TILES) {
            if (ntiles > 0) issue_qk(0, ss);
            __syncwarp();
            if (ntiles > 1) issue_qk(1, ss);
            __syncwarp();
#pragma unroll 1
            for (int i = 2; i < ntiles; ++i) {
                issue_qk(i, ss);
                __syncwarp();
            }
        } else {
#pragma unroll 1
            for (int i = 0; i < ntiles; ++i) {
                if (i == UM_Q_FIRST) { named_bar_sync(3, UM_SM_THREADS + 32); tc_fence_after_sync(); }
                issue_qk(i, [](int t) { return t >= UM_Q_FIRST; });
                __syncwarp();
            }
        }
    } else if (warp_u == 9) {
        // The TMA producer, in the order in which the tensor pipe frees the stage halves: S runs four tiles ahead
        // of O += P V, so after the first K refills it is V of tile i + 4 (after P V of tile i), then K of tile i + 8
        // (after S of tile i + 4).
        auto refill = [&](int i, bool is_v, unsigned int bar, unsigned int parity) {
            if (i < np) {
                mbar_wait(bar, parity, p.err);
                __syncwarp();
                if (elect_one()) issue_kv(i, is_v);
            } else {
                mbar_wait(bar, parity, p.err);
                __syncwarp();
                gather_tree(i, is_v);
            }
            __syncwarp();
        };
#pragma unroll 1
        for (int t = UM_STAGES; t < min(ntiles, 2 * UM_STAGES); ++t) refill(t, false, bar_ek + (t % UM_STAGES) * 8, 0u);
#pragma unroll 1
        for (int i = 0; i + UM_STAGES < ntiles; ++i) {
            refill(i + UM_STAGES, true, bar_ev + (i % UM_STAGES) * 8, (unsigned int)(i / UM_STAGES) & 1u);
            if (i + 2 * UM_STAGES < ntiles)
                refill(i + 2 * UM_STAGES, false, bar_ek + (i % UM_STAGES) * 8, (unsigned int)(i / UM_STAGES + 1) & 1u);
        }
    }
    // Stream `half`: tiles half, half + 2, ...  As soon as S of tile i is in registers its buffer is handed back.  The
    // stream's P buffer and O were last used by O += P V of tile i - 2, which is waited for before they are touched
    // (its barrier's next completion is tile i + 2's, which needs this stream's P of tile i + 2).
    // What bounds a tile is the chain of a stream: 128 clocks for S, 140 for the maximum, 640 for the exponentials (530 with both streams at them), 30 for P,
    // and 123 for each answer of a barrier that is long complete.  So both barriers are asked ahead of other work and the answer is looked at
    // behind it, and the S issuer waits for K first: the slowest CTA of a launch, whose two streams are in step, takes 780 clocks a tile instead of
    // 910.  Us a call with Q from shared memory, without : with that, timed in turn: 4 trees of 60 nodes, 64 / 8 heads, 16300 tokens 141 : 130, 4700 47.1 : 44.4; 10 trees,
    // 32 / 8 heads, 4096 tokens 75.1 : 71.3; 16 trees 78.4 : 77.1; one tree of 2048 tokens 11.4 both ways.  (S of the next tile loaded ahead of P's store: 148
    // for the first; the streams' exponentials in turns: 142 .. 150.)
    unsigned int sr[64];                                     // the row's 64 scores
    if (QT && warp < 8 && ntiles > ATT_Q_TILES) {                    // Q into tensor memory while the first S are computed: half a row per thread
        uint4 qq[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) qq[c] = *reinterpret_cast<const uint4*>(gQ + q_off(row, half * 8 + c));
        tmem_st32(tQ + half * 32 + lane_off, reinterpret_cast<unsigned int*>(qq));
        tmem_wait_st();
        tc_fence_before_sync();
        asm volatile("bar.arrive 3, %0;" ::"r"(UM_SM_THREADS + 32) : "memory");
    }
    bool ok_s = false;                                       // S of the stream's next tile was complete when last asked
#pragma unroll 1
    for (int i = half; i < ntiles && warp < 8; i += 2) {
        if (!ok_s) mbar_wait(bar_s + half * 8, (unsigned int)(i >> 1) & 1u, p.err);      // S of tile i is complete
        __syncwarp();                                        // (each lane has waited by its own answer; warp-aligned loads follow)
        tc_fence_after_sync();
        tmem_ld32(tS + half * ATT_BN + lane_off, sr);
        tmem_ld32(tS + half * ATT_BN + 32 + lane_off, sr + 32);
        tmem_wait_ld();
        tc_fence_before_sync();
        mbar_arrive(bar_sr + half * 8);

        const bool is_tree = i >= np;
        const int col0 = is_tree ? (i - np) * ATT_BN : (t0 + i) * ATT_BN;
        const int nvis = (is_tree ? nk : L) - col0;          // columns of this tile inside the sequence / tree
        // The scores stay unscaled in registers (the scale is positive: it commutes with the maximum and folds into
        // the exponent's multiply-add). A prefix tile inside the sequence needs no mask at all.
        if (is_tree || nvis < ATT_BN) {
            // a tree tile of 64 keys lies inside one 64-bit word of the ancestor mask
            unsigned long long vis64 = nvis >= 64 ? ~0ull : ((1ull << max(nvis, 0)) - 1ull);
            if (is_tree) vis64 &= (col0 == 0 ? mk0 : mk1);
            const unsigned int vlo = (unsigned int)vis64, vhi = (unsigned int)(vis64 >> 32);
#pragma unroll
            for (int c = 0; c < 32; ++c) {
                if (!((vlo >> c) & 1u)) sr[c] = __float_as_uint(-CUDART_INF_F);
                if (!((vhi >> c) & 1u)) sr[32 + c] = __float_as_uint(-CUDART_INF_F);
            }
        }
        float mxa = -CUDART_INF_F, mxb = -CUDART_INF_F;
#pragma unroll
        for (int c = 0; c < 32; c += 2) {                    // three-input maxima: half the instructions
            mxa = max3(mxa, __uint_as_float(sr[c]), __uint_as_float(sr[c + 1]));
            mxb = max3(mxb, __uint_as_float(sr[32 + c]), __uint_as_float(sr[33 + c]));
        }
        const float mx = fmaxf(mxa, mxb) * p.scale_log2;
        // The reference the exponents are taken against only follows the row's maximum when that has grown by more
        // than 8 (a factor 256): until then P <= 256 instead of <= 1, which costs no precision (fp32 sums, bf16 keeps
        // its relative error, the final O / l is the same quotient), and O is rescaled a few times per row instead of
        // whenever any row of the warp sees a new maximum.
        const float mnew = (mx > mrun + (FOLLOW && i < nfollow ? 0.f : 8.f) || mrun == -CUDART_INF_F) ? fmaxf(mrun, mx) : mrun;
        const float muse = (mnew == -CUDART_INF_F) ? 0.f : mnew;
        const float corr = ex2_approx(mrun - muse);          // 1 when the maximum did not grow, 0 at the stream's first tile
        mrun = mnew;
        // the row's P of this tile, in registers first
        // (the exponent's multiply-add and the row sum run as packed fp32 pairs: half the instructions)
        const float2 sc2 = make_float2(p.scale_log2, p.scale_log2), nm2 = make_float2(-muse, -muse);
        float2 ls0 = make_float2(0.f, 0.f), ls1 = make_float2(0.f, 0.f);
        uint4 pk[8];
        bool ok_o = false;                                   // O += P V of tile i - 2 is complete
#pragma unroll
        for (int c8 = 0; c8 < 8; ++c8) {
            if (c8 == 4) ok_o = mbar_test_wait(bar_ev + ((i + 2) & (UM_STAGES - 1)) * 8, (unsigned int)((i + 2) / UM_STAGES - 1) & 1u);
            float2 pv[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float2 x = fma2_ftz(make_float2(__uint_as_float(sr[c8 * 8 + 2 * e]), __uint_as_float(sr[c8 * 8 + 2 * e + 1])), sc2, nm2);
                pv[e] = make_float2(ex2_approx(x.x), ex2_approx(x.y));
            }
            ls0 = add2_ftz(ls0, add2_ftz(pv[0], pv[1]));
            ls1 = add2_ftz(ls1, add2_ftz(pv[2], pv[3]));
            pk[c8].x = pack_bf16(pv[0].x, pv[0].y); pk[c8].y = pack_bf16(pv[1].x, pv[1].y);
            pk[c8].z = pack_bf16(pv[2].x, pv[2].y); pk[c8].w = pack_bf16(pv[3].x, pv[3].y);
        }
        const float2 ls = add2_ftz(ls0, ls1);
        lrun = fmaf(lrun, corr, ls.x + ls.y);
        if (i >= 2) {
            if (!ok_o) mbar_wait(bar_ev + ((i - 2) % UM_STAGES) * 8, (unsigned int)((i - 2) / UM_STAGES) & 1u, p.err);
            tc_fence_after_sync();
        }
        // rescale this stream's O (the load/store are warp-wide: a warp rescales if any of its rows needs it; the vote is where its lanes
        // meet again - a __syncwarp ahead of it as well makes 4 trees of 60 nodes, 64 / 8 heads, 4700 tokens 47.8 us instead of 43.0)
        if (i >= 2 && __any_sync(HS_FULL_MASK, corr != 1.f)) {
            // in pieces of 32 columns, a round trip each, where FOLLOW may rescale often (10 trees of 60 nodes, 32 / 8 heads, spread up to 8192 tokens, pieces of 16 : so
            // 65.7 : 62.3 us; 6000 tokens 52.8 : 50.7); the instance that serves the shortest steps rescales once or twice, and is 0.2 us shorter with 16
            constexpr int W = QT ? 32 : 16;
#pragma unroll 1
            for (int ch = 0; ch < HS_HEAD_DIM; ch += W) {
                unsigned int ov[W];
                const unsigned int at = tO + half * HS_HEAD_DIM + lane_off + ch;
                if constexpr (QT) tmem_ld32(at, ov); else tmem_ld16(at, ov);
                tmem_wait_ld();
#pragma unroll
                for (int c = 0; c < W; ++c) ov[c] = __float_as_uint(__uint_as_float(ov[c]) * corr);
                if constexpr (QT) tmem_st32(at, ov); else tmem_st16(at, ov);
            }
        }
        // P stays in tensor memory (the A operand of O += P V): this row's 64 bf16 values are 32 columns of its lane
        ok_s = mbar_test_wait(bar_s + half * 8, (unsigned int)((i + 2) >> 1) & 1u);
        tmem_st32(tP + half * (ATT_BN / 2) + lane_off, reinterpret_cast<unsigned int*>(pk));
        tmem_wait_st();
        tc_fence_before_sync();
        mbar_arrive(bar_p + half * 8);
    }
    if (ntiles > 0 && warp < 8) mbar_wait(bar_done, 0u, p.err);
    __syncwarp();                                        // the issuing and producer warps reconverge (warp-aligned barriers follow)
    tc_fence_after_sync();
    // the two streams of a row are combined like two splits: weights w0, w1 on the streams' O, one (max, sum)
    if (warp < 8) { s_mx[half * ATT_BM + row] = mrun; s_lx[half * ATT_BM + row] = lrun; }
    __syncthreads();
    float w0 = 0.f, w1 = 0.f;
    if (warp < 8) {
        const float m_a = s_mx[row], m_b = s_mx[ATT_BM + row];
        mrun = fmaxf(m_a, m_b);
        const float muse = (mrun == -CUDART_INF_F) ? 0.f : mrun;
        w0 = ex2_approx(m_a - muse);
        w1 = ex2_approx(m_b - muse);
        lrun = s_lx[row] * w0 + s_lx[ATT_BM + row] * w1;
    }
    // this thread's 32 columns [half * 64 + ch * 32, + 32) of the row's combined O (a stream without tiles has no O)
    auto load_o = [&](int ch, unsigned int* ov) {
        unsigned int oa[32], ob[32];
        if (ntiles > 0) tmem_ld32(tO + lane_off + half * 64 + ch * 32, oa);
        if (ntiles > 1) tmem_ld32(tO + HS_HEAD_DIM + lane_off + half * 64 + ch * 32, ob);
        tmem_wait_ld();
#pragma unroll
        for (int c = 0; c < 32; ++c) {
            float v = 0.f;
            if (ntiles > 0) v = __uint_as_float(oa[c]) * w0;
            if (ntiles > 1) v = fmaf(__uint_as_float(ob[c]), w1, v);
            ov[c] = __float_as_uint(v);
        }
    };

    // ---- epilogue ----------------------------------------------------------------------------------------------
    if (p.nsplit == 1) {
        const float inv = lrun > 0.f ? 1.f / lrun : 0.f;
#pragma unroll 1
        for (int ch = 0; ch < 2 && warp < 8; ++ch) {
            unsigned int ov[32];
            load_o(ch, ov);
            uint4 o[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                o[q].x = pack_bf16(__uint_as_float(ov[q * 8 + 0]) * inv, __uint_as_float(ov[q * 8 + 1]) * inv);
                o[q].y = pack_bf16(__uint_as_float(ov[q * 8 + 2]) * inv, __uint_as_float(ov[q * 8 + 3]) * inv);
                o[q].z = pack_bf16(__uint_as_float(ov[q * 8 + 4]) * inv, __uint_as_float(ov[q * 8 + 5]) * inv);
                o[q].w = pack_bf16(__uint_as_float(ov[q * 8 + 6]) * inv, __uint_as_float(ov[q * 8 + 7]) * inv);
            }
            const int lane = tid & 31;
            quad_transpose(o, lane);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int dst = __shfl_sync(HS_FULL_MASK, (int)orow, (lane & ~3) + i);
                if (dst >= 0)
                    *(reinterpret_cast<uint4*>(p.out + (size_t)dst * HS_HEAD_DIM + half * 64 + ch * 32) + (lane & 3)) = o[i];
            }
        }
        if (orow >= 0 && p.lse_out && half == 0) p.lse_out[orow] = (mrun + log2f(lrun)) * LN2;
    } else {
        // ---- merge across the splits of the cluster through distributed shared memory ----------------------------
        // Row rl of the block is merged by CTA owner(rl) = rl * ns / 128.  Every thread sends its part of its row, {O / l as
        // bf16, max, sum}, straight from registers into the owner's receive area (which no tile ever uses) by asynchronous
        // remote stores that signal the owner's mbarrier; an owner merges once all ns pieces have landed: per row the
        // splits' weights 2^(max_s - max) l_s / sum once, then out = sum_s weight_s (O_s / l_s).  (A normalised
        // partial is a convex combination of V rows, so bf16 keeps it to 2^-9 of the values' magnitude: the output
        // is bf16 anyway.)  A sender may leave at once: nothing reads its shared memory.  (Staging the rows, a cluster
        // barrier and bulk copies cost 1.5 us more.)
        const int ns = p.nsplit;
        unsigned char* po = gR;                                                      // [ns][rows_max] rows of ATT_PB_STRIDE bytes
        const unsigned int s_recv = smem_u32(gR);
        const int rows_max = (ATT_BM + ns - 1) / ns + 1;
        const int r_lo = (split * ATT_BM + ns - 1) / ns, r_hi = ((split + 1) * ATT_BM + ns - 1) / ns;   // rows this CTA owns
        long long* s_og = reinterpret_cast<long long*>(gM);               // output row of each owned row (or -1)
        float* s_wt = reinterpret_cast<float*>(gM + UM_MAP_BYTES + 1024 + 2048);  // [rows owned][ATT_MAX_SPLIT] weights
        cluster_wait();                                      // (the arrival at the start, long complete)
        if (warp < 8) {
            const int owner = row * ns / ATT_BM, o_lo = (owner * ATT_BM + ns - 1) / ns;
            const unsigned int dst = cluster_map_addr(s_recv + (unsigned int)(split * rows_max + row - o_lo) * ATT_PB_STRIDE, owner);
            const unsigned int rbar = cluster_map_addr(bar_r, owner);
            if (half == 0) st_async_v2(dst + HS_HEAD_DIM * 2, __float_as_uint(mrun), __float_as_uint(lrun), rbar);
            const float inv = lrun > 0.f ? 1.f / lrun : 0.f;
#pragma unroll 1
            for (int ch = 0; ch < 2; ++ch) {
                unsigned int ov[32];
                load_o(ch, ov);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    st_async_v4(dst + (half * 64 + ch * 32 + q * 8) * 2,
                                pack_bf16(__uint_as_float(ov[q * 8 + 0]) * inv, __uint_as_float(ov[q * 8 + 1]) * inv),
                                pack_bf16(__uint_as_float(ov[q * 8 + 2]) * inv, __uint_as_float(ov[q * 8 + 3]) * inv),
                                pack_bf16(__uint_as_float(ov[q * 8 + 4]) * inv, __uint_as_float(ov[q * 8 + 5]) * inv),
                                pack_bf16(__uint_as_float(ov[q * 8 + 6]) * inv, __uint_as_float(ov[q * 8 + 7]) * inv), rbar);
            }
        }
        int og_mine = -1;
        if (tid < r_hi - r_lo) {
            const int rg = m0 + r_lo + tid, node = (int)((unsigned int)rg * p.inv_g >> 16);
            if (rg < M) og_mine = kept_row_of(node) * p.hq + h * p.G + (rg - node * p.G);
            s_og[tid] = og_mine;
        }
        mbar_wait_cluster(bar_r, 0u, p.err);                         // all ns pieces of this CTA's rows have landed
        // the splits' weights of every owned row, once
        if (tid < r_hi - r_lo) {
            float2 ml[ATT_MAX_SPLIT];
            float Mx = -CUDART_INF_F;
#pragma unroll
            for (int s2 = 0; s2 < ATT_MAX_SPLIT; ++s2) {
                ml[s2] = make_float2(-CUDART_INF_F, 0.f);
                if (s2 < ns) ml[s2] = *reinterpret_cast<const float2*>(po + (size_t)(s2 * rows_max + tid) * ATT_PB_STRIDE + HS_HEAD_DIM * 2);
                Mx = fmaxf(Mx, ml[s2].x);
            }
            float w[ATT_MAX_SPLIT], lsum = 0.f;
#pragma unroll
            for (int s2 = 0; s2 < ATT_MAX_SPLIT; ++s2) {
                w[s2] = (ml[s2].x == -CUDART_INF_F) ? 0.f : ex2_approx(ml[s2].x - Mx) * ml[s2].y;
                lsum += w[s2];
            }
            const float inv = lsum > 0.f ? 1.f / lsum : 0.f;
#pragma unroll
            for (int s2 = 0; s2 < ATT_MAX_SPLIT; ++s2) s_wt[tid * ATT_MAX_SPLIT + s2] = w[s2] * inv;
            if (og_mine >= 0 && p.lse_out) p.lse_out[og_mine] = (Mx + log2f(lsum)) * LN2;
        }
        __syncwarp();
        if (tid < UM_SM_THREADS)                             // the softmax threads: the weights are written
            asm volatile("bar.sync 2, %0;" ::"r"(UM_SM_THREADS) : "memory");
        // items = (row, 16-byte column group of 8); every item combines one group of each split, all from local shared memory
        for (int it = tid; it < (r_hi - r_lo) * 16 && tid < UM_SM_THREADS; it += UM_SM_THREADS) {
            const int rl = it >> 4, c8 = it & 15;
            float acc[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[e] = 0.f;
#pragma unroll
            for (int s2 = 0; s2 < ATT_MAX_SPLIT; ++s2) {
                if (s2 < ns) {
                    const float w = s_wt[rl * ATT_MAX_SPLIT + s2];
                    fma_bf16x8(acc, w, *reinterpret_cast<const uint4*>(po + (size_t)(s2 * rows_max + rl) * ATT_PB_STRIDE + c8 * 16));
                }
            }
            const long long og = s_og[rl];
            if (og >= 0) {
                uint4 packed;
                packed.x = pack_bf16(acc[0], acc[1]); packed.y = pack_bf16(acc[2], acc[3]);
                packed.z = pack_bf16(acc[4], acc[5]); packed.w = pack_bf16(acc[6], acc[7]);
                *reinterpret_cast<uint4*>(p.out + (size_t)og * HS_HEAD_DIM + c8 * 8) = packed;
            }
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    if (warp == 0) tmem_dealloc(tmem_base, UM_TMEM_COLS);
}
#include "tree_attn_duo.cuh"

// ---- host side -----------------------------------------------------------------------------------------------------
typedef CUresult (*encode_tiled_fn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                    const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                    CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static bool encode(hs_ctx* ctx, CUtensorMap* tm, int rank, const void* base, const cuuint64_t* gdim, const cuuint64_t* gstr,
                   const cuuint32_t* box) {
    const cuuint32_t estr[3] = {1, 1, 1};
    return ((encode_tiled_fn)ctx->encode_tiled)(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, const_cast<void*>(base), gdim, gstr,
                                                box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                                CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
static bool make_kv_map(hs_ctx* ctx, CUtensorMap* tm, const void* base, const hs_attn_desc* d, bool head_first) {
    const cuuint64_t tok = (cuuint64_t)d->kv_total, heads = (cuuint64_t)d->hkv;
    const cuuint64_t ts = (cuuint64_t)d->kv_token_stride * 2, hs = (cuuint64_t)d->kv_head_stride * 2;
    // (d, token, head) if the token stride is the smaller one, else (d, head, token)
    const cuuint64_t gdim[3] = {HS_HEAD_DIM, head_first ? tok : heads, head_first ? heads : tok};
    const cuuint64_t gstr[2] = {head_first ? ts : hs, head_first ? hs : ts};
    const cuuint32_t box[3] = {64, head_first ? (cuuint32_t)ATT_BN : 1u, head_first ? 1u : (cuuint32_t)ATT_BN};
    return encode(ctx, tm, 3, base, gdim, gstr, box);
}
// rows of `width` elements, gathered one by one (box one row high)
static bool make_row_map(hs_ctx* ctx, CUtensorMap* tm, const void* base, size_t rows, size_t width) {
    const cuuint64_t gdim[2] = {(cuuint64_t)width, (cuuint64_t)rows}, gstr[1] = {(cuuint64_t)width * 2};
    const cuuint32_t box[2] = {64, 1};
    return encode(ctx, tm, 2, base, gdim, gstr, box);
}

template <typename Kernel>
static void query_cluster_caps(Kernel kernel, int threads, size_t smem, int sm_count, int* cap) {
    for (int sz = 1; sz <= ATT_MAX_SPLIT; ++sz) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(1, sz, sm_count);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = smem;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 1; at[0].val.clusterDim.y = sz; at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int nclusters = 0;
        if (cudaOccupancyMaxActiveClusters(&nclusters, kernel, &cfg) == cudaSuccess) cap[sz] = nclusters * sz;
        else { cap[sz] = 0; (void)cudaGetLastError(); }
    }
}

hs_status hs_launch_attention(hs_ctx* ctx, const hs_pruned_tree* pruned, const hs_attn_desc* d, const void* q,
                              const void* k_tree, const void* v_tree, const void* k_cache, const void* v_cache,
                              void* out, float* lse_out, cudaStream_t stream) {
    int* cap_umma = ctx->attn_cap;                   // CTAs that run at once in clusters of s (per device = per context)
    if (!ctx->attn_ready) {
        for (const auto kernel : {tree_attn_umma_kernel<false, false>, tree_attn_umma_kernel<true, false>, tree_attn_umma_kernel<true, true>})
            if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, UM_SMEM_BYTES) != cudaSuccess) return HS_ERR_CUDA;
        if (cudaFuncSetAttribute(tree_attn_duo_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, AD_SMEM_BYTES) != cudaSuccess)
            return HS_ERR_CUDA;
        query_cluster_caps(tree_attn_umma_kernel<false, false>, UM_THREADS, UM_SMEM_BYTES, ctx->sm_count, cap_umma);
        ctx->attn_ready = true;
    }
    AttnParams p;
    p.q = (const __nv_bfloat16*)q;
    p.k_tree = (const __nv_bfloat16*)k_tree;
    p.v_tree = (const __nv_bfloat16*)v_tree;
    p.out = (__nv_bfloat16*)out;
    p.lse_out = lse_out;
    p.n_keep = pruned->n_keep;
    p.keep_off = pruned->keep_off;
    p.keep_idx = pruned->keep_idx;
    p.anc_mask = (const unsigned long long*)pruned->anc_mask;
    p.status = pruned->status;
    p.node_off = d->node_off;
    p.kv_off = d->kv_off;
    p.batch = d->batch;
    p.hq = d->hq;
    p.hkv = d->hkv;
    p.G = d->hq / d->hkv;
    p.inv_g = (65536u + p.G - 1) / p.G;
    p.layout = d->layout;
    p.head_first = d->kv_head_stride > d->kv_token_stride;
    p.scale_log2 = d->sm_scale * LOG2E;
    p.err = ctx->counters + HS_CNT_ERROR;
    p.prefetch = (ctx->prefetch & HS_PREFETCH_KV) != 0;
    const int pairs = d->batch * d->hkv, rows = p.G * d->max_nodes;

    CUtensorMap tmK, tmV;
    memset(&tmK, 0, sizeof(tmK));
    memset(&tmV, 0, sizeof(tmV));
    const int mblocks = (rows + ATT_BM - 1) / ATT_BM;
    const int prefix_tiles = (d->max_kv_len + ATT_BN - 1) / ATT_BN;
    const AttnChoice how = attn_choice(pairs * mblocks, mblocks, ctx->sm_count, prefix_tiles, cap_umma);
    p.nsplit = how.splits;
    p.follow = how.follow;
    if (d->kv_total > 0) {
        if (!make_kv_map(ctx, &tmK, k_cache, d, p.head_first) || !make_kv_map(ctx, &tmV, v_cache, d, p.head_first))
            return HS_ERR_CUDA;
    }
    const dim3 grid(mblocks, p.nsplit, pairs), cl(1, p.nsplit, 1);
    cudaError_t e;
    // Rows by drafted node id may lie anywhere in the batch's rows, behind sequences that are skipped as well: past max_rows, which bounds
    // the kept ones, but never past what a batch may hold.  (The maps only have to cover the rows that are asked for.)
    const size_t n = HS_MAX_ROWS;
    const size_t w = (size_t)d->hkv * HS_HEAD_DIM;
    CUtensorMap tmQ, tmKT, tmVT;
    if (!make_row_map(ctx, &tmKT, k_tree, n, w) || !make_row_map(ctx, &tmVT, v_tree, n, w)) return HS_ERR_CUDA;
    if (how.duo) {
        if (!make_row_map(ctx, &tmQ, q, n * d->hq, HS_HEAD_DIM)) return HS_ERR_CUDA;
        e = hs_launch(tree_attn_duo_kernel, grid, dim3(AD_THREADS), AD_SMEM_BYTES, stream, ctx->pdl, cl, p, tmK, tmV, tmQ, tmKT, tmVT);
    } else {
        const int tree_tiles = (d->max_nodes + ATT_BN - 1) / ATT_BN;
        const auto kernel = q_from_tensor_memory(pairs * mblocks, mblocks, ctx->sm_count, prefix_tiles, tree_tiles, how) ? tree_attn_umma_kernel<true, true>
                            : how.follow ? tree_attn_umma_kernel<true, false> : tree_attn_umma_kernel<false, false>;
        e = hs_launch(kernel, grid, dim3(UM_THREADS), UM_SMEM_BYTES, stream, ctx->pdl, cl, p, tmK, tmV, tmKT, tmVT);
    }
    return e == cudaSuccess ? HS_OK : HS_ERR_CUDA;
}
