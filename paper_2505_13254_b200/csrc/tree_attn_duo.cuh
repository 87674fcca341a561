// The attention kernel for launches of more than one wave of CTAs and for the longest prefixes in pairs of splits.  Included by tree_attention.cu, whose header
// describes the problem.
//
// TWO CTAs share an SM (half of its tensor memory, 99 KiB of shared memory each): while one starts (dependent loads of the pruned
// tree, Q, first tiles: about 10 us ahead of and behind its tiles together) or merges, the other one computes.  tree_attn_umma_kernel
// has a whole SM to itself, less latency for one CTA and nothing to fill such gaps with.  A CTA has 128 query rows and ONE stream
// over tiles of 64 keys: S is double-buffered, P (bf16) overwrites the S it came from, so the tensor-core order is S(i), P V(i),
// S(i + 2) from one issuing thread.  Two threads share a row (32 keys of a tile each).  One producer warp: prefix tiles by tiled
// copies, the indirectly indexed rows of Q and of the tree tokens by tile::gather4.
// Bound by the chain of a tile (S, load, maximum, exponentials, P V): 0.68 us for one CTA, 1.06 us for two at once, against 0.77 to 1.0 us
// for two tiles of tree_attn_umma_kernel, but nothing of a start or an end is left uncovered.  16 trees of 60 nodes, 32 / 8 heads, 512 tokens 19.4 us against 22.1; 32 trees 38.2
// against 48.1 (which launches come here, and what it costs at long prefixes: see duo_splits).  With tiles of 128 keys S and P leave room for one buffer only: 4 x 62 nodes,
// 64 / 8 heads, 32768 tokens 366 us instead of 302.
#pragma once

#define AD_HALF_BYTES (ATT_TILE_BYTES / 2)          // columns 0..63 / 64..127 of a K or V tile (rows of 128 bytes, 128-byte swizzle)
#define AD_SM_THREADS 256                           // softmax threads
#define AD_MMA_WARP 8
#define AD_TMA_WARP 9
#define AD_THREADS 320
#define AD_MISC_BYTES 3072                          // barriers and small arrays ahead of the tiles
#define AD_SLOTS 4                                  // ring of K and V tiles
#define AD_SMEM_BYTES (AD_MISC_BYTES + ATT_Q_BYTES + AD_SLOTS * ATT_TILE_BYTES)
#define AD_TMEM_COLS 256                            // S / P of tile i: columns 64 (i & 1) ..; O: 128 ..
// Tiles after the first over which the exponents' reference follows every new row maximum.  One stream per row has one exact P where the two
// streams of tree_attn_umma_kernel have two, so its error against fp64 was larger (2-norm relative, 16 x 50..60 nodes, 256..512 tokens:
// 2.296e-3 against 2.251e-3; 12 x 37..46, 1200 tokens: 2.339e-3 against 2.325e-3).  Followed over one tile 2.261e-3 and 2.330e-3, over two
// 2.230e-3 and 2.319e-3, over three 2.202e-3 and 2.313e-3; each costs 0.5 us of 18.7 and of 29.8 (one more rescale of O).
#define AD_FOLLOW 2
// Merge of the splits, in the memory of the query tile and the ring: (max, sum) of the warps, weights and output rows of the rows owned,
// then the partials received, 128 fp32 of O / l and {max, sum} per row.  (As bf16 a split launch rounded O twice: 2.876e-3 from fp64 at
// 4 x 62 nodes, 64 / 8 heads, 32768 tokens, now 2.339e-3, for 2.5 us of 276.)
#define AD_PART_BYTES (HS_HEAD_DIM * 4 + 8)
#define AD_PB_STRIDE (HS_HEAD_DIM * 4 + 16)
#define AD_END_BYTES 4608
static_assert(AD_END_BYTES % 16 == 0 && AD_END_BYTES >= 2048 + 68 * ATT_MAX_SPLIT * 4 + 68 * 4 &&
              AD_END_BYTES + (ATT_BM + 2 * ATT_MAX_SPLIT) * AD_PB_STRIDE <= ATT_Q_BYTES + AD_SLOTS * ATT_TILE_BYTES, "partials behind the small arrays");

// The two warps that share 32 rows meet on barriers 1 .. 4.  (Constant numbers: with a number in a register the kernel would claim all
// 16 of a CTA and only one CTA would fit on an SM.)  What one of them has read from tensor memory ahead of the barrier the other may
// overwrite behind it (S by P), which needs tcgen05's own fences on both sides.
__device__ __forceinline__ void pair_sync(int quad) {
    tc_fence_before_sync();
    if (quad == 0) named_bar_sync(1, 64);
    else if (quad == 1) named_bar_sync(2, 64);
    else if (quad == 2) named_bar_sync(3, 64);
    else named_bar_sync(4, 64);
    tc_fence_after_sync();
}

__global__ void __launch_bounds__(AD_THREADS, 2)
tree_attn_duo_kernel(const __grid_constant__ AttnParams p, const __grid_constant__ CUtensorMap tmK,
                      const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmQ,
                      const __grid_constant__ CUtensorMap tmKT, const __grid_constant__ CUtensorMap tmVT) {
    extern __shared__ __align__(1024) unsigned char smem[];
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(HS_FULL_MASK, tid >> 5, 0);
    const unsigned int sbase = smem_u32(smem);
    // barriers: slot full[4], slot empty[4], S ready[2], P written[2], Q full, P V of a tile done, partials received, last P V done
    const unsigned int bar_full = sbase, bar_empty = bar_full + 8 * AD_SLOTS, bar_s = bar_empty + 8 * AD_SLOTS,
                       bar_p = bar_s + 16, bar_qfull = bar_p + 16, bar_o = bar_qfull + 8, bar_r = bar_o + 8, bar_done = bar_r + 8;
    volatile unsigned int* s_tmem = reinterpret_cast<volatile unsigned int*>(smem + 256);
    int* s_seq = reinterpret_cast<int*>(smem + 264);
    float* s_pair = reinterpret_cast<float*>(smem + 512);      // [4 quads][2 parities][2 halves][32 rows]
    const unsigned int sQ = sbase + AD_MISC_BYTES, sR = sQ + ATT_Q_BYTES;      // query tile, the ring

    // kv_off is an array of the caller like any other: it is read ahead of the dependency wait only where the caller vouches for the
    // cache and with it for its offsets.  (Both instructions come again below, without effect.)
    if (!p.prefetch) { pdl_launch_dependents(); pdl_wait(); }
    // sequences are taken longest prefix first (see tree_attn_umma_kernel)
    int b = blockIdx.z / p.hkv;
    const int h = blockIdx.z % p.hkv;
    if (p.batch > 1 && p.batch <= AD_THREADS) {
        if (tid < p.batch) {
            const int len = p.kv_off[tid + 1] - p.kv_off[tid];
            int rank = 0;
            for (int j = 0; j < p.batch; ++j) {
                const int lj = p.kv_off[j + 1] - p.kv_off[j];
                rank += (lj > len || (lj == len && j < tid));
            }
            if (rank == b) *s_seq = tid;
        }
        __syncthreads();
        b = *s_seq;
    }
    const int split = blockIdx.y, m0 = blockIdx.x * ATT_BM;
    const int kv0 = p.kv_off[b], L = p.kv_off[b + 1] - kv0;
    // units of work: the prefix tiles, then the tree tokens (one or two tiles); t0 .. t0 + nunit of them
    const int T = (L + ATT_BN - 1) / ATT_BN + 1;
    const int per = (T + p.nsplit - 1) / p.nsplit;
    const int t0 = min(split * per, T), nunit = min(t0 + per, T) - t0;
    const int np = max(min(nunit, T - 1 - t0), 0);               // prefix tiles of this CTA

    // rows of the block that this CTA will merge
    auto owned = [&](int s, int& lo, int& hi) {
        lo = (s * ATT_BM + p.nsplit - 1) / p.nsplit;
        hi = ((s + 1) * ATT_BM + p.nsplit - 1) / p.nsplit;
    };
    if (tid == 0) {
        for (int i = 0; i < 2 * AD_SLOTS; ++i) mbar_init(bar_full + i * 8, 1);
        mbar_init(bar_s, 1); mbar_init(bar_s + 8, 1);
        mbar_init(bar_p, 8); mbar_init(bar_p + 8, 8);                          // one arrival per warp of the stream
        for (int i = 0; i < 4; ++i) mbar_init(bar_qfull + i * 8, 1);
        mbar_init_fence();
    }
    if (warp == AD_TMA_WARP && lane < 5)
        tma_prefetch_desc(lane == 0 ? &tmK : lane == 1 ? &tmV : lane == 2 ? &tmQ : lane == 3 ? &tmKT : &tmVT);
    if (warp == AD_MMA_WARP) {
        tmem_alloc(smem_u32((const void*)s_tmem), AD_TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    pdl_launch_dependents();
    const unsigned int tmem = *s_tmem;

    // ---- producer pieces (one warp) -----------------------------------------------------------------------------
    // Tiles go through the ring in the order in which the tensor cores take them: K0, K1, then V(i), K(i + 2).
    int pslot = 0;                                             // next slot to fill, parity its `empty` barrier is waited with
    unsigned int ppar = 1u;
    // K (V) of prefix tile i of this CTA into the next slot; called by one lane
    auto load_prefix = [&](int i, bool is_v) {
        const unsigned int dst = sR + pslot * ATT_TILE_BYTES, bar = bar_full + pslot * 8;
        mbar_wait(bar_empty + pslot * 8, ppar, p.err);
        mbar_expect_tx(bar, ATT_TILE_BYTES);
        const CUtensorMap* tm = is_v ? &tmV : &tmK;
        const int tok = kv0 + (t0 + i) * ATT_BN;
        if (p.head_first) {
            tma_load_3d(dst, tm, 0, tok, h, bar);
            tma_load_3d(dst + AD_HALF_BYTES, tm, 64, tok, h, bar);
        } else {
            tma_load_3d(dst, tm, 0, h, tok, bar);
            tma_load_3d(dst + AD_HALF_BYTES, tm, 64, h, tok, bar);
        }
    };
    auto advance_slot = [&]() { if (++pslot == AD_SLOTS) { pslot = 0; ppar ^= 1u; } };
    // place `pos` of the ring's order for ntile tiles -> tile and K or V
    auto place = [&](int pos, int ntile, int& i, bool& is_v) {
        is_v = pos >= 2 && ((pos & 1) == 0 || pos == 2 * ntile - 1);
        i = !is_v ? (pos + 1) / 2 : (pos & 1) ? ntile - 1 : pos / 2 - 1;
        if (ntile == 1) { is_v = pos == 1; i = 0; }
    };
    int issued = 0;                                            // places filled ahead of the dependency wait
    if (warp == AD_TMA_WARP && p.prefetch) {
        // (with three prefix tiles the first four places hold K0, K1, V0, K2 whatever else there is)
        issued = np >= 3 ? AD_SLOTS : np == 2 ? 3 : 0;
        for (int n = 0; n < issued; ++n) {
            int i; bool is_v;
            place(n, 1 << 20, i, is_v);
            if (lane == 0) load_prefix(i, is_v);
            advance_slot();
        }
    }
    pdl_wait();                                                // the pruned tree, q, k_tree, v_tree come from upstream
    const int nk_b = p.n_keep[b], st_b = p.status[b], koff = p.keep_off[b];
    const int nbase = p.layout == HS_ROWS_ORIGINAL ? p.node_off[b] : 0;
    const int nk = st_b == 0 ? nk_b : 0, M = nk * p.G;
    if (m0 >= M) {                                             // nothing to do (the same for every CTA of the cluster)
        if (warp == AD_TMA_WARP && lane == 0)
            for (int i = 0; i < issued; ++i) mbar_wait(bar_full + i * 8, 0u, p.err);   // no copy may outlive the CTA
        __syncthreads();
        if (warp == AD_MMA_WARP) tmem_dealloc(tmem, AD_TMEM_COLS);
        return;
    }
    const int ntile = nunit > np ? np + (nk + ATT_BN - 1) / ATT_BN : np;
    auto kept_row_of = [&](int node) { return p.layout == HS_ROWS_ORIGINAL ? nbase + p.keep_idx[koff + node] : koff + node; };
    auto query_row = [&](int r) {                              // row of q / out that holds query row r
        const int node = (int)((unsigned int)r * p.inv_g >> 16);
        return kept_row_of(node) * p.hq + h * p.G + (r - node * p.G);
    };

    if (warp == AD_TMA_WARP) {
        // ---- the producer warp ----------------------------------------------------------------------------------
        if (ntile > 0) {
            // query rows: four per lane (rows past the last one repeat it; nobody reads their results)
            if (lane == 0) mbar_expect_tx(bar_qfull, ATT_Q_BYTES);
            __syncwarp();
            {
                int r[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) r[i] = query_row(min(m0 + lane * 4 + i, M - 1));
                const unsigned int dst = sQ + lane * 512;
                tma_gather4(dst, &tmQ, 0, r[0], r[1], r[2], r[3], bar_qfull);
                tma_gather4(dst + ATT_Q_BYTES / 2, &tmQ, 64, r[0], r[1], r[2], r[3], bar_qfull);
            }
            for (int n = issued; n < 2 * ntile; ++n) {
                int i; bool is_v;
                place(n, ntile, i, is_v);
                if (i < np) {
                    if (lane == 0) load_prefix(i, is_v);
                } else {
                    // tree tokens: four keys per lane of half a warp (keys past the last one repeat it; they are masked)
                    int r[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) r[k] = kept_row_of(min((i - np) * ATT_BN + (lane & 15) * 4 + k, nk - 1));
                    const unsigned int dst = sR + pslot * ATT_TILE_BYTES + (lane >> 4) * AD_HALF_BYTES + (lane & 15) * 512;
                    const unsigned int bar = bar_full + pslot * 8;
                    mbar_wait(bar_empty + pslot * 8, ppar, p.err);
                    __syncwarp();
                    if (lane == 0) mbar_expect_tx(bar, ATT_TILE_BYTES);
                    __syncwarp();
                    tma_gather4(dst, is_v ? &tmVT : &tmKT, h * HS_HEAD_DIM + (lane >> 4) * 64, r[0], r[1], r[2], r[3], bar);
                }
                advance_slot();
                __syncwarp();
            }
        }
        __syncwarp();
    } else if (warp == AD_MMA_WARP) {
        // ---- the issuing warp: all lanes wait, one elected thread issues, all loop state warp-uniform -------------------
        // (with the waits inside the elected branch 16 trees of 40..60 nodes, 900..1000 tokens took 26.9 us a call, now 25.9)
        const unsigned int idesc_qk = umma_idesc_bf16(ATT_BM, ATT_BN, false);
        const unsigned int idesc_pv = umma_idesc_bf16(ATT_BM, HS_HEAD_DIM, true);
        const unsigned long long dq0 = umma_desc_sw128(sQ, 16, 1024), dk0 = umma_desc_sw128(sR, 16, 1024);
        const unsigned long long dv0 = umma_desc_sw128(sR, AD_HALF_BYTES, 1024);
        int slot = 0;                                          // slot of the next K or V tile and its full parity
        unsigned int par = 0u;
        auto issue_s = [&](int i) {
            mbar_wait(bar_full + slot * 8, par, p.err);
            __syncwarp();
            tc_fence_after_sync();
            if (elect_one()) {
                const unsigned long long dk = dk0 + (unsigned long long)(slot * (ATT_TILE_BYTES >> 4));
                const unsigned int ts = tmem + (i & 1) * ATT_BN;
#pragma unroll
                for (int ks = 0; ks < 8; ++ks)
                    umma_ss_bf16(ts, dq0 + (((ks >> 2) * (ATT_Q_BYTES / 2) + (ks & 3) * 32) >> 4),
                                 dk + (((ks >> 2) * AD_HALF_BYTES + (ks & 3) * 32) >> 4), idesc_qk, ks > 0 ? 1u : 0u);
                umma_commit(bar_s + (i & 1) * 8);
                umma_commit(bar_empty + slot * 8);
            }
            __syncwarp();
            if (++slot == AD_SLOTS) { slot = 0; par ^= 1u; }
        };
        if (ntile > 0) {
            mbar_wait(bar_qfull, 0u, p.err);
            __syncwarp();
            issue_s(0);
            if (ntile > 1) issue_s(1);
        }
#pragma unroll 1
        for (int i = 0; i < ntile; ++i) {
            mbar_wait(bar_full + slot * 8, par, p.err);
            mbar_wait(bar_p + (i & 1) * 8, (unsigned int)(i >> 1) & 1u, p.err);
            __syncwarp();
            tc_fence_after_sync();
            if (elect_one()) {
                const unsigned long long dv = dv0 + (unsigned long long)(slot * (ATT_TILE_BYTES >> 4));
                const unsigned int tp = tmem + (i & 1) * ATT_BN, to = tmem + 2 * ATT_BN;
                // 16 keys per instruction; none for keys behind the end of the prefix or of the tree
                const int nkk = ((i < np ? L - (t0 + i) * ATT_BN : nk - (i - np) * ATT_BN) + 15) >> 4;
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                    if (kk < nkk) umma_ts_bf16(to, tp + kk * 8, dv + (kk * 2048 >> 4), idesc_pv, (i > 0 || kk > 0) ? 1u : 0u);
                umma_commit(bar_empty + slot * 8);
                umma_commit(bar_o);
                if (i == ntile - 1) umma_commit(bar_done);
            }
            __syncwarp();
            if (++slot == AD_SLOTS) { slot = 0; par ^= 1u; }
            if (i + 2 < ntile) issue_s(i + 2);
        }
    }
    // ---- softmax warps: (half, quad) has rows 32 quad .. + 31 and keys 32 half .. + 31 of every tile -----------------------
    const int half = (warp >> 2) & 1, quad = warp & 3;         // (meaningful for warps 0 .. 7)
    const int row = quad * 32 + lane;
    const unsigned int lane_off = (unsigned int)(quad * 32) << 16;
    float mrun = -CUDART_INF_F, lrun = 0.f;
    if (warp < AD_MMA_WARP) {
        const unsigned int tO = tmem + lane_off + 2 * ATT_BN;
        const int r = m0 + row;
        const bool live = __any_sync(HS_FULL_MASK, r < M);     // the warp has a row with a result
        // the row's ancestors among this thread's keys of the two tree tiles
        unsigned int mk0 = 0u, mk1 = 0u;
        if (r < M) {
            const unsigned long long* am = p.anc_mask + 2 * (size_t)(koff + (int)((unsigned int)r * p.inv_g >> 16));
            mk0 = (unsigned int)(am[0] >> (32 * half));
            mk1 = (unsigned int)(am[1] >> (32 * half));
        }
#pragma unroll 1
        for (int i = 0; i < ntile; ++i) {
            const unsigned int tS = tmem + lane_off + (i & 1) * ATT_BN;
            mbar_wait(bar_s + (i & 1) * 8, (unsigned int)(i >> 1) & 1u, p.err);      // S of this tile is complete
            __syncwarp();                                      // (warp-aligned instructions follow)
            tc_fence_after_sync();
            if (!live) {
                if (lane == 0) mbar_arrive(bar_p + (i & 1) * 8);
                __syncwarp();
                continue;
            }
            unsigned int sr[32];                               // this thread's scores
            tmem_ld32(tS + half * 32, sr);
            tmem_wait_ld();
            const bool is_tree = i >= np;
            const int nvis = (is_tree ? nk - (i - np) * ATT_BN : L - (t0 + i) * ATT_BN) - half * 32;     // columns inside the sequence / tree
            // The scores stay unscaled in registers (the scale is positive: it commutes with the maximum and folds into the
            // exponent's multiply-add).  A prefix tile inside the sequence needs no mask at all.
            if (is_tree || nvis < 32) {
                unsigned int v = nvis >= 32 ? ~0u : ((1u << max(nvis, 0)) - 1u);
                if (is_tree) v &= i == np ? mk0 : mk1;
#pragma unroll
                for (int c = 0; c < 32; ++c)
                    if (!((v >> c) & 1u)) sr[c] = __float_as_uint(-CUDART_INF_F);
            }
            float mx2[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {                      // three-input maxima, two independent chains
                mx2[q] = fmaxf(__uint_as_float(sr[q * 16]), __uint_as_float(sr[q * 16 + 1]));
#pragma unroll
                for (int c = 2; c < 16; c += 2)
                    mx2[q] = max3(mx2[q], __uint_as_float(sr[q * 16 + c]), __uint_as_float(sr[q * 16 + c + 1]));
            }
            // The row's maximum over both halves.  (The barrier also says that the other half's scores are in registers: P may
            // overwrite them.)
            const float own = fmaxf(mx2[0], mx2[1]) * p.scale_log2;
            float* xf = s_pair + (quad * 2 + (i & 1)) * 64;
            xf[half * 32 + lane] = own;
            pair_sync(quad);
            const float mx = fmaxf(own, xf[(half ^ 1) * 32 + lane]);
            // The reference follows the maximum only when that has grown by more than 8 (see tree_attn_umma_kernel) - but closely over
            // the first AD_FOLLOW + 1 tiles: a score that was the maximum when its tile was taken has P = 2^0, which bf16 holds without error,
            // and those are the weights that count most.
            const float mnew = (mx > mrun + (i <= AD_FOLLOW ? 0.f : 8.f) || mrun == -CUDART_INF_F) ? fmaxf(mrun, mx) : mrun;
            const float muse = (mnew == -CUDART_INF_F) ? 0.f : mnew;
            const float corr = ex2_approx(mrun - muse);        // 1 when the reference stays, 0 at the first tile
            mrun = mnew;
            if (i > 0 && __any_sync(HS_FULL_MASK, corr != 1.f)) {        // (the accesses are warp-wide; 64 columns per half)
                mbar_wait(bar_o, (unsigned int)(i - 1) & 1u, p.err);     // O is at rest (its next completion needs this tile's P)
                __syncwarp();
                tc_fence_after_sync();
#pragma unroll 1
                for (int ch = 0; ch < 4; ++ch) {
                    unsigned int ov[16];
                    tmem_ld16(tO + half * 64 + ch * 16, ov);
                    tmem_wait_ld();
#pragma unroll
                    for (int c = 0; c < 16; ++c) ov[c] = __float_as_uint(__uint_as_float(ov[c]) * corr);
                    tmem_st16(tO + half * 64 + ch * 16, ov);
                }
            }
            // P over S
            const float2 sc2 = make_float2(p.scale_log2, p.scale_log2), nm2 = make_float2(-muse, -muse);
            float2 ls0 = make_float2(0.f, 0.f), ls1 = make_float2(0.f, 0.f);
            unsigned int pk[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                const float2 x = fma2_ftz(make_float2(__uint_as_float(sr[2 * e]), __uint_as_float(sr[2 * e + 1])), sc2, nm2);
                const float2 e2 = make_float2(ex2_approx(x.x), ex2_approx(x.y));
                if (e & 1) ls1 = add2_ftz(ls1, e2); else ls0 = add2_ftz(ls0, e2);
                pk[e] = pack_bf16(e2.x, e2.y);
            }
            tmem_st16(tS + half * 16, pk);
            const float2 ls = add2_ftz(ls0, ls1);
            lrun = fmaf(lrun, corr, ls.x + ls.y);
            tmem_wait_st();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_p + (i & 1) * 8);
        }
        // Every tile has been used and the last P V is complete: Q and the ring are free.
        if (ntile > 0) mbar_wait(bar_done, 0u, p.err);
        __syncwarp();
        tc_fence_after_sync();
    }
    const int ns = p.nsplit;
    const int rows_max = (ATT_BM + ns - 1) / ns + 1;
    int r_lo, r_hi;
    owned(split, r_lo, r_hi);
    if (ns > 1) {
        if (tid == 0) mbar_expect_tx(bar_r, (unsigned int)(ns * (r_hi - r_lo) * AD_PART_BYTES));
        __syncwarp();
        cluster_arrive();                                      // partials may now arrive in this CTA's tiles
    }

    // ---- end: the parts of a row held by several threads are combined; all of this in the query tile's memory -----------------
    float2* s_ml = reinterpret_cast<float2*>(smem + AD_MISC_BYTES);                  // [8 warps][32] (max, sum)
    float* s_wt = reinterpret_cast<float*>(smem + AD_MISC_BYTES + 2048);             // [rows owned <= 65][ATT_MAX_SPLIT] weights
    int* s_og = reinterpret_cast<int*>(smem + AD_MISC_BYTES + 2048 + 68 * ATT_MAX_SPLIT * 4);   // [rows owned] output row or -1
    const unsigned char* gP = smem + AD_MISC_BYTES + AD_END_BYTES;                              // [ns][rows_max] partials received
    if (warp < AD_MMA_WARP) {
        s_ml[warp * 32 + lane] = make_float2(mrun, lrun);
        named_bar_sync(5, AD_SM_THREADS);
        lrun += s_ml[(warp ^ 4) * 32 + lane].y;                // (the halves of a row have one reference)
        const float inv = lrun > 0.f ? 1.f / lrun : 0.f;
        // 32 columns at a time of this thread's 64 of the normalised O row
        auto load_piece = [&](int ch, float (&o)[32]) {
            unsigned int oa[32];
#pragma unroll
            for (int c = 0; c < 32; ++c) oa[c] = 0u;           // (an accumulator without tiles holds anything)
            if (ntile > 0) tmem_ld32(tmem + lane_off + 2 * ATT_BN + half * 64 + ch * 32, oa);
            tmem_wait_ld();
#pragma unroll
            for (int c = 0; c < 32; ++c) o[c] = __uint_as_float(oa[c]) * inv;
        };
        const int col0 = half * 64;
        const bool has_ml = half == 0;                   // this thread speaks for the row's (max, sum)
        if (ns == 1) {
            const int orow = m0 + row < M ? query_row(m0 + row) : -1;
#pragma unroll 1
            for (int ch = 0; ch < 2; ++ch) {
                float of[32];
                load_piece(ch, of);
                uint4 o[4];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    o[q] = make_uint4(pack_bf16(of[q * 8], of[q * 8 + 1]), pack_bf16(of[q * 8 + 2], of[q * 8 + 3]),
                                      pack_bf16(of[q * 8 + 4], of[q * 8 + 5]), pack_bf16(of[q * 8 + 6], of[q * 8 + 7]));
                quad_transpose(o, lane);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int dst = __shfl_sync(HS_FULL_MASK, orow, (lane & ~3) + i);
                    if (dst >= 0)
                        *(reinterpret_cast<uint4*>(p.out + (size_t)dst * HS_HEAD_DIM + col0 + ch * 32) + (lane & 3)) = o[i];
                }
            }
            if (orow >= 0 && p.lse_out && has_ml) p.lse_out[orow] = (mrun + log2f(lrun)) * LN2;
        } else {
            // rows of the block that this CTA owns: the merge needs their output rows
            if (tid < r_hi - r_lo) s_og[tid] = m0 + r_lo + tid < M ? query_row(m0 + r_lo + tid) : -1;
            __syncwarp();
            cluster_wait();                                    // every CTA of the cluster has used its tiles
            const int owner = row * ns / ATT_BM;
            int o_lo, o_hi;
            owned(owner, o_lo, o_hi);
            const unsigned int dst = cluster_map_addr(sbase + AD_MISC_BYTES + AD_END_BYTES + (unsigned int)(split * rows_max + row - o_lo) * AD_PB_STRIDE, owner);
            const unsigned int rbar = cluster_map_addr(bar_r, owner);
            if (has_ml) st_async_v2(dst + HS_HEAD_DIM * 4, __float_as_uint(mrun), __float_as_uint(lrun), rbar);
            __syncwarp();
#pragma unroll 1
            for (int ch = 0; ch < 2; ++ch) {
                float o[32];
                load_piece(ch, o);
#pragma unroll
                for (int i = 0; i < 32; i += 4)
                    st_async_v4(dst + (col0 + ch * 32 + i) * 4, __float_as_uint(o[i]), __float_as_uint(o[i + 1]), __float_as_uint(o[i + 2]),
                                __float_as_uint(o[i + 3]), rbar);
            }
            mbar_wait_cluster(bar_r, 0u, p.err);               // all ns pieces of this CTA's rows have landed
            // the ranges' weights of every owned row, once
            if (tid < r_hi - r_lo) {
                float2 ml[ATT_MAX_SPLIT];
                float Mx = -CUDART_INF_F;
#pragma unroll
                for (int s2 = 0; s2 < ATT_MAX_SPLIT; ++s2) {
                    ml[s2] = make_float2(-CUDART_INF_F, 0.f);
                    if (s2 < ns) ml[s2] = *reinterpret_cast<const float2*>(gP + (size_t)(s2 * rows_max + tid) * AD_PB_STRIDE + HS_HEAD_DIM * 4);
                    Mx = fmaxf(Mx, ml[s2].x);
                }
                float w[ATT_MAX_SPLIT], lsum = 0.f;
#pragma unroll
                for (int s2 = 0; s2 < ATT_MAX_SPLIT; ++s2) {
                    w[s2] = (ml[s2].x == -CUDART_INF_F) ? 0.f : ex2_approx(ml[s2].x - Mx) * ml[s2].y;
                    lsum += w[s2];
                }
                const float isum = lsum > 0.f ? 1.f / lsum : 0.f;
#pragma unroll
                for (int s2 = 0; s2 < ATT_MAX_SPLIT; ++s2) s_wt[tid * ATT_MAX_SPLIT + s2] = w[s2] * isum;
                if (s_og[tid] >= 0 && p.lse_out) p.lse_out[s_og[tid]] = (Mx + log2f(lsum)) * LN2;
            }
            __syncwarp();
            named_bar_sync(5, AD_SM_THREADS);                  // the weights are written
            // items = (row, column group of 8), each over all ranges from local shared memory
            for (int it = tid; it < (r_hi - r_lo) * 16; it += AD_SM_THREADS) {
                const int rl = it >> 4, c8 = it & 15;
                float acc[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) acc[e] = 0.f;
#pragma unroll
                for (int s2 = 0; s2 < ATT_MAX_SPLIT; ++s2)
                    if (s2 < ns) {
                        const float w = s_wt[rl * ATT_MAX_SPLIT + s2];
                        const float4* v = reinterpret_cast<const float4*>(gP + (size_t)(s2 * rows_max + rl) * AD_PB_STRIDE + c8 * 32);
                        const float4 a = v[0], c = v[1];
                        acc[0] = fmaf(w, a.x, acc[0]); acc[1] = fmaf(w, a.y, acc[1]); acc[2] = fmaf(w, a.z, acc[2]); acc[3] = fmaf(w, a.w, acc[3]);
                        acc[4] = fmaf(w, c.x, acc[4]); acc[5] = fmaf(w, c.y, acc[5]); acc[6] = fmaf(w, c.z, acc[6]); acc[7] = fmaf(w, c.w, acc[7]);
                    }
                if (s_og[rl] >= 0)
                    *reinterpret_cast<uint4*>(p.out + (size_t)s_og[rl] * HS_HEAD_DIM + c8 * 8) =
                        make_uint4(pack_bf16(acc[0], acc[1]), pack_bf16(acc[2], acc[3]), pack_bf16(acc[4], acc[5]), pack_bf16(acc[6], acc[7]));
            }
        }
    } else if (ns > 1) {
        cluster_wait();
    }
    __syncwarp();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    if (warp == AD_MMA_WARP) tmem_dealloc(tmem, AD_TMEM_COLS);
}
