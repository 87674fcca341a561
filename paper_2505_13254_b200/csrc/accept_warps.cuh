// The row pass of the acceptance for launches with many rows: every warp on its own.  Included by accept.cu.
//
// The rows to read - the target row of every kept node, then the draft row of every kept internal node of a sequence in
// rejection mode - form a stream of rounds of 128 vectors that is cut into equal contiguous shares, one per warp of the
// device, as in the entropy pass.  Which rows those are is only known on the device (the pruned tree comes from the kernel
// ahead), so every CTA derives the list itself: a bit per kept node for "its draft row is needed", a prefix of the bit
// counts, the share bounds from the total.  A warp then meets nobody until the partials of a row that lies in several shares
// merge.  Arg-max with the lowest index on ties: a lane keeps its maximum and the first round that holds it, and the first
// such round of the warp is read once more.  Sampling sequences add sum e^((x-ref)/T) against a reference that all lanes
// share.  Sequences that finish in the row pass (greedy, deterministic proposals) are walked at the end of the CTA that
// merged their last target row.
// Bound by the rounds: 36 of 40 us on a batch of greedy and sampling rows (179 MB), read at 5.0 TB/s, 1500 clocks a round with 32 KiB of loads in flight on an SM; a row end
// takes 2 us, the last ones of all warps at the same time (stamps of every warp).  28 % of the issue slots.  Behind a ring of 32 KiB
// items with 16 warps in lockstep the call took (now): 497 greedy rows of 128256 bf16 30.5 us (27.6), 497 rows half sampling
// with their draft rows and the walk 75.8 (62.6), 1127 rows of 32000, three modes, 95.4 (55.4), 120 greedy rows 14.0 (12.6).
#pragma once

#define AW_WARPS 16
#define AW_THREADS (AW_WARPS * 32)
#define AW_MAX_SEGS 32                        // shares a row may lie in: one lane each when they merge
#define AW_ROW_END 4                          // what the end of a row segment costs, in rounds

template <bool BF16>
__global__ void __launch_bounds__(AW_THREADS, 1) accept_warp_kernel(const __grid_constant__ AcceptParams p) {
    constexpr int VE = BF16 ? 8 : 4;
    constexpr int NWORDS = HS_MAX_ROWS / 32;
    __shared__ unsigned int s_bits[NWORDS];          // kept node -> its draft row is part of the stream
    __shared__ int s_pref[NWORDS + 1];               // set bits ahead of each word
    __shared__ unsigned short s_pending[HS_MAX_BATCH];   // sequences this CTA has to walk
    __shared__ int s_npending;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) s_npending = 0;
    if (!p.have_draft) pdl_launch_dependents();      // (else behind the wait: the walk kernel relies on it)
    pdl_wait();                            // the pruned tree and the logits come from upstream
    if (p.have_draft) pdl_launch_dependents();

    // ---- the rows of the stream --------------------------------------------------------------------------------
    const int T = min(p.pr.keep_off[p.batch], p.part_rows);
    const int nwords = p.have_draft ? (T + 31) / 32 : 0;
    for (int i = tid; i < nwords; i += AW_THREADS) s_bits[i] = 0u;
    __syncthreads();
    if (p.have_draft) {
        for (int b = warp; b < p.batch; b += AW_WARPS) {
            const int md = p.mode[b], koff = p.pr.keep_off[b], nk = p.pr.n_keep[b];
            if (md != HS_ACCEPT_REJECTION) continue;
            for (int j = 1 + lane; j < nk; j += 32) {
                const int par = p.pr.new_parent[koff + j];
                const int k = koff + par;
                if (par >= 0 && par < j && k < T) atomicOr(&s_bits[k >> 5], 1u << (k & 31));
            }
        }
        __syncthreads();
        if (warp == 0) {
            int run = 0;
            for (int i0 = 0; i0 < nwords; i0 += 32) {
                const int cnt = i0 + lane < nwords ? __popc(s_bits[i0 + lane]) : 0;
                int incl = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int up = __shfl_up_sync(HS_FULL_MASK, incl, o);
                    if (lane >= o) incl += up;
                }
                if (i0 + lane < nwords) s_pref[i0 + lane] = run + incl - cnt;
                run += __shfl_sync(HS_FULL_MASK, incl, 31);
            }
            if (lane == 0) s_pref[nwords] = run;
        }
        __syncthreads();
    }
    // sequences that kept nothing (flagged upstream) and sequences in rejection mode without draft logits get their
    // result here, shared out over the warps of the grid
    for (int b = blockIdx.x * AW_WARPS + warp; b < p.batch; b += gridDim.x * AW_WARPS) {
        const int st = p.pr.status[b];
        const bool empty = p.pr.n_keep[b] <= 0 || st != 0;
        const bool nodraft = !empty && p.mode[b] == HS_ACCEPT_REJECTION && !p.have_draft;
        if (empty || nodraft) {
            const int cap = p.out.path_cap;
            for (int j = lane; j < cap; j += 32) {
                p.out.path_nodes[b * cap + j] = -1;
                p.out.path_compact[b * cap + j] = -1;
                p.out.path_tokens[b * cap + j] = -1;
            }
            if (lane == 0) {
                p.out.accept_len[b] = 0; p.out.bonus_token[b] = -1; p.out.terminal_rank[b] = -1;
                p.out.status[b] = empty ? (st != 0 ? st : HS_ERR_BAD_TREE) : HS_ERR_INVALID_ARG;
            }
        }
    }
    const int W = T + (p.have_draft ? s_pref[nwords] : 0);
    const int rr = (p.nvec + ROUND_VECS - 1) / ROUND_VECS;        // rounds per row
    const int rv = rr + AW_ROW_END;                               // places per row in the stream
    const int total = W * rv;
    const int per = max((total + p.shares - 1) / p.shares, (rr + AW_MAX_SEGS - 3) / (AW_MAX_SEGS - 2));
    const int c = blockIdx.x * AW_WARPS + warp;
    int g = c < p.shares ? min(c * per, total) : total;
    const int g1 = min(g + per, total);

    while (g < g1) {
        // ---- one segment: rounds [r0, r1) of row w of the stream --------------------------------------------------------
        const int w = g / rv, x0 = w * rv + AW_ROW_END;           // (the row's rounds stand behind its extra places)
        const int r0 = max(g - x0, 0), r1 = min(rr, g1 - x0);
        g = min(g1, x0 + rr);
        if (r0 >= r1) continue;
        int k = w;
        const bool draft = w >= T;
        if (draft) {                                              // the (w - T)-th set bit
            const int rnk = w - T;
            int lo = 0, hi = nwords;
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (s_pref[mid] <= rnk) lo = mid; else hi = mid;
            }
            k = lo * 32 + (int)__fns(s_bits[lo], 0, rnk - s_pref[lo] + 1);
        }
        const int b = sequence_of(p.pr.keep_off, p.batch, k, lane);
        const int mode = p.mode[b], nk = p.pr.n_keep[b];
        const float temp = p.temperature[b];
        const int orig = p.node_off[b] + p.pr.keep_idx[k];
        const int lrow = draft || p.target_layout == HS_ROWS_ORIGINAL ? orig : k;
        const uint4* rowv = (const uint4*)((const char*)(draft ? p.draft : p.target) + (size_t)lrow * p.row_stride * (BF16 ? 2 : 4));
        const bool sampling = mode != HS_ACCEPT_GREEDY;           // the row's normaliser is needed
        const float invT = sampling ? LOG2E / temp : 0.f, slack = sampling ? 30.f / invT : 0.f;
        float ref = -CUDART_INF_F, nref = 0.f, lm = -CUDART_INF_F;
        int lr = 0;                                               // first round with this lane's maximum
        float2 s2 = make_float2(0.f, 0.f);
        auto consume = [&](const uint4 (&d)[4], int r) {
            const float rm = round_max<BF16>(d);
            if (rm > lm) { lm = rm; lr = r; }
            if (!sampling) return;
            if (__any_sync(HS_FULL_MASK, rm > ref + slack)) {
                const float nr = fmaxf(ref, order_bits_float(__reduce_max_sync(HS_FULL_MASK, float_order_bits(rm))));
                const float f = ref == -CUDART_INF_F ? 0.f : ex2f((ref - nr) * invT);
                s2.x *= f; s2.y *= f;
                ref = nr;
                nref = -nr * invT;
            }
            const float2 l2 = make_float2(invT, invT), n2 = make_float2(nref, nref);
            const unsigned int* x = reinterpret_cast<const unsigned int*>(&d[0]);
#pragma unroll
            for (int q = 0; q < (BF16 ? 16 : 8); ++q) {
                const float2 t = fma2_ftz(BF16 ? make_float2(bf16_lo(x[q]), bf16_hi(x[q]))
                                               : make_float2(__uint_as_float(x[2 * q]), __uint_as_float(x[2 * q + 1])), l2, n2);
                s2 = add2_ftz(s2, make_float2(ex2f(t.x), ex2f(t.y)));
            }
        };
        uint4 da[4], db[4];
        load_round<BF16>(p, rowv, r0, lane, da);
        int r = r0;
#pragma unroll 1
        for (; r + 1 < r1; r += 2) {
            load_round<BF16>(p, rowv, r + 1, lane, db);
            consume(da, r);
            if (r + 2 < r1) load_round<BF16>(p, rowv, r + 2, lane, da);
            consume(db, r + 1);
        }
        if (r < r1) consume(da, r);
        // ---- end of the segment --------------------------------------------------------------------------------------------
        float M = order_bits_float(__reduce_max_sync(HS_FULL_MASK, float_order_bits(lm)));
        unsigned long long key = 0ull;
        if (!draft && M > -CUDART_INF_F) {                        // the first round that holds the maximum, once more
            const int rf = (int)__reduce_min_sync(HS_FULL_MASK, lm == M ? (unsigned int)lr : 0x7fffffffu);
            load_round<BF16>(p, rowv, rf, lane, da);
            unsigned int at = 0x7fffffffu;
#pragma unroll
            for (int j = 3; j >= 0; --j) {
                float x[8];
                unpack<BF16>(da[j], x);
#pragma unroll
                for (int e = VE - 1; e >= 0; --e)
                    if (x[e] == M) at = (unsigned int)((rf * ROUND_VECS + j * 32 + lane) * VE + e);
            }
            key = make_key(M, (int)__reduce_min_sync(HS_FULL_MASK, at));
        }
        float S = sampling ? warp_sum(s2.x + s2.y) * (M == -CUDART_INF_F ? 0.f : ex2f((ref - M) * invT)) : 0.f;
        const int c_first = x0 / per, nseg = (x0 + rr - 1) / per - c_first + 1;
        bool mine = true;                                         // this warp holds the row's final result
        if (nseg > 1) {
            // a share has at most two partial rows: slot 0 for one that began in an earlier share, slot 1 for one that goes on
            int last = 0;
            if (lane == 0) {
                p.partials[2 * c + (r0 > 0 ? 0 : 1)] =
                    make_uint4((unsigned int)key, (unsigned int)(key >> 32), __float_as_uint(M), __float_as_uint(S));
                // one release-acquire arrival at device scope: the partial is visible to whoever arrives last
                int old;
                asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(old) : "l"(&p.row_cnt[w]) : "memory");
                last = old == nseg - 1;
                if (last) p.row_cnt[w] = 0;
            }
            mine = __shfl_sync(HS_FULL_MASK, last, 0) != 0;
            if (mine) {
                unsigned long long ck = 0ull;
                float cmx = -CUDART_INF_F, cs = 0.f;
                if (lane < nseg) {
                    const uint4 q = __ldcg(&p.partials[2 * (c_first + lane) + (lane == 0 ? 1 : 0)]);
                    ck = ((unsigned long long)q.y << 32) | q.x;
                    cmx = __uint_as_float(q.z);
                    cs = __uint_as_float(q.w);
                }
                int src;
                key = warp_best_key(ck, src);
                M = warp_max(cmx);
                S = sampling ? warp_sum(cmx == -CUDART_INF_F ? 0.f : cs * ex2f((cmx - M) * invT)) : 0.f;
            }
        }
        if (mine && lane == 0) {
            if (draft) {
                p.ro.drf_ms[k] = make_float2(M, S);
            } else {
                p.ro.tgt_arg[k] = key_index(key);
                p.ro.tgt_ms[k] = make_float2(M, S);
                if (mode != HS_ACCEPT_REJECTION) {
                    // greedy sequences and deterministic proposals finish in this kernel: the CTA that completes a
                    // sequence's last target row walks its tree once its own shares are done
                    int old;
                    asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(old) : "l"(&p.seq_cnt[b]) : "memory");
                    if (old == nk - 1) {
                        p.seq_cnt[b] = 0;
                        s_pending[atomicAdd(&s_npending, 1)] = (unsigned short)b;
                    }
                }
            }
        }
        __syncwarp();
    }
    __syncthreads();                          // every warp has finished its share: the list of walks is complete
    if (tid < HS_ROW_THREADS) {
        const int npend = s_npending;
        for (int i = 0; i < npend; ++i) {
            const int b = s_pending[i];
            if (p.mode[b] == HS_ACCEPT_GREEDY) {
                const int koff = p.pr.keep_off[b], nk = p.pr.n_keep[b];
                greedy_walk(p, b, koff, nk, load_walk_node(p, koff, nk, p.node_off[b]));
            }
            else deterministic_walk(p, b);
            walk_sync();                       // the walks' shared arrays are free again
        }
        if (p.jobs) {
            // the bonus draws of deterministic-proposal sequences are shared by all CTAs
            bool any = false;
            for (int b = tid; b < p.batch; b += HS_ROW_THREADS)
                any |= p.mode[b] == HS_ACCEPT_DETERMINISTIC && p.pr.n_keep[b] > 0 && p.pr.status[b] == 0;
            if (named_bar_or(2, HS_ROW_THREADS, any)) {
                if (npend == 0) det_help(p, -1, false);
                det_leave(p, -1, gridDim.x);
            }
        }
    }
}
