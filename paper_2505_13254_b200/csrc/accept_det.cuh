// Acceptance of sequences with deterministic proposals (Sec. 2.1 with a point-mass proposal per candidate): the walk, which
// runs inside the row pass, and its bonus draw, which the CTAs of the row pass share.  Included by accept.cu.
//
// The draw sums a whole vocabulary row in double.  One CTA alone took 50 us for 128256 tokens (a chain of 63 slices, fp64
// additions that wait for one another): cut into slices of HS_ROW_THREADS * 4 vectors that every idle CTA of the launch
// takes from, a batch of 8 draws takes 13 us (accept call 108 -> 55 us).
#pragma once

// fp64 additions that depend on one another cost about 64 cycles each: sums are taken as trees, not as chains.
__device__ __forceinline__ double sum8(double a0, double a1, double a2, double a3, double a4, double a5, double a6, double a7) {
    return ((a0 + a1) + (a2 + a3)) + ((a4 + a5) + (a6 + a7));
}
__device__ __forceinline__ double sum8(const float (&m)[8]) {
    return sum8((double)m[0], (double)m[1], (double)m[2], (double)m[3], (double)m[4], (double)m[5], (double)m[6], (double)m[7]);
}

__device__ __forceinline__ int det_slices(const AcceptParams& p) {
    return min((p.nvec + HS_ROW_THREADS * 4 - 1) / (HS_ROW_THREADS * 4), DET_SLICES);
}

// masses of this thread's 4 vectors of slice ph of a target row (0 past the vocabulary and for rejected tokens)
__device__ __forceinline__ void slice_mass(const AcceptParams& p, const char* prow, float pm, float ips, float invT,
                                           const int* rej, int nrej, int ph, float (&m)[4][8]) {
    const int vsh = p.is_bf16 ? 3 : 2, ve = 1 << vsh;
    uint4 d[4];
    const int vbase = (ph * HS_ROW_THREADS + threadIdx.x) * 4;
#pragma unroll
    for (int q = 0; q < 4; ++q)
        d[q] = (vbase + q < p.nvec) ? __ldg((const uint4*)prow + vbase + q) : make_uint4(0, 0, 0, 0);
    const int inside = p.vocab - (vbase << vsh);             // tokens from the thread's first one to the end of the vocabulary
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float x[8];
        if (p.is_bf16) unpack<true>(d[q], x); else unpack<false>(d[q], x);
#pragma unroll
        for (int e = 0; e < 8; ++e)
            m[q][e] = e < ve ? exp2f((fmaxf(x[e], -1e30f) - pm) * invT) * ips : 0.f;     // (as in the accept tests below: the
                                                                     // distribution is one, masses below the normal range included)
    }
    if (inside < 4 << vsh) {                                 // (the thread that runs past the vocabulary, and those behind it)
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if ((q << vsh) + e >= inside) m[q][e] = 0.f;
    }
    for (int k = 0; k < nrej; ++k) {                         // few: the siblings rejected at this node
        const int r = rej[k] - (vbase << vsh);
        if ((unsigned int)r < 4u << vsh) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    if (e < ve && r == (q << vsh) + e) m[q][e] = 0.f;
        }
    }
}
// A warp's part of a slice: its mass (running sums in double) in every lane, the last token of positive mass as result.
__device__ __forceinline__ int slice_warp(const AcceptParams& p, const char* prow, float pm, float ips, float invT,
                                          const int* rej, int nrej, int ph, double& sum) {
    const int tid = threadIdx.x, ve = p.is_bf16 ? 8 : 4;
    float m[4][8];
    slice_mass(p, prow, pm, ips, invT, rej, nrej, ph, m);
    int last = -1;
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int e = 0; e < 8; ++e)
            if (m[q][e] > 0.f) last = ((ph * HS_ROW_THREADS + tid) * 4 + q) * ve + e;
    sum = warp_sum_d((sum8(m[0]) + sum8(m[1])) + (sum8(m[2]) + sum8(m[3])));
    return __reduce_max_sync(HS_FULL_MASK, last);
}

// HS_ROW_THREADS threads of a CTA that has nothing else to do take slices of published draws: of sequence `seq` alone, or
// (seq < 0) of any deterministic-proposal sequence of the batch.  Returns when none is left to take - or, unless `own`, when
// none has been published for a while: the CTA that publishes a draw finishes it without help as well.
#define DET_PATIENCE_NS 100000ull
__device__ __noinline__ void det_help(const AcceptParams& p, int seq, bool own) {
    __shared__ int s_job[2];
    __shared__ int s_hrej[HS_MAX_NODES];
    __shared__ double s_w[HS_ROW_THREADS / 32];
    __shared__ int s_last[HS_ROW_THREADS / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nph = det_slices(p);
    unsigned int todo = 0u;                              // warp 0: bit i = sequence lane + 32 i may still have slices to take
    if (tid < 32) {
        for (int i = 0; i * 32 < p.batch; ++i) {
            const int b = i * 32 + lane;
            if (b < p.batch && (seq < 0 ? (p.mode[b] == HS_ACCEPT_DETERMINISTIC && p.pr.n_keep[b] > 0 && p.pr.status[b] == 0) : b == seq))
                todo |= 1u << i;
        }
    }
    const unsigned long long t0 = global_timer_ns();
    for (;;) {
        if (tid < 32) {
            int job = -1, slice = 0;
            for (;;) {
                int ready = -1;                          // a published draw of this lane with slices left
                for (unsigned int w = todo; w; w &= w - 1) {
                    const int b = (__ffs(w) - 1) * 32 + lane;
                    if (ld_acquire_gpu(&p.det_cnt[b]) == 0) continue;
                    if (*(volatile int*)&p.det_cnt[DET_MAX_BATCH + b] < nph) { ready = b; break; }
                    todo &= ~(1u << (b >> 5));
                }
                const unsigned int any = __ballot_sync(HS_FULL_MASK, ready >= 0);
                if (any) {
                    // spread the CTAs over the draws: the first ready lane at or behind one that depends on the CTA
                    const unsigned int from = any & (HS_FULL_MASK << ((blockIdx.x + blockIdx.y) & 31));
                    const int src = __ffs(from ? from : any) - 1;
                    if (lane == src) {
                        slice = atomicAdd(&p.det_cnt[DET_MAX_BATCH + ready], 1);
                        job = ready;
                    }
                    job = __shfl_sync(HS_FULL_MASK, job, src);
                    slice = __shfl_sync(HS_FULL_MASK, slice, src);
                    if (slice < nph) break;
                    job = -1;
                    continue;                            // (somebody took the last one)
                }
                if (!__any_sync(HS_FULL_MASK, todo != 0u)) break;
                if (__any_sync(HS_FULL_MASK, !own && global_timer_ns() - t0 > DET_PATIENCE_NS)) break;
                __nanosleep(100);
            }
            if (lane == 0) { s_job[0] = job; s_job[1] = slice; }
        }
        walk_sync();
        const int b = s_job[0], ph = s_job[1];
        if (b < 0) break;
        const DetJob& j = p.jobs[b];
        const int nrej = __ldcg(&j.nrej);
        for (int k = tid; k < nrej; k += HS_ROW_THREADS) s_hrej[k] = __ldcg(&j.rej[k]);
        walk_sync();
        const char* row = (const char*)__ldcg((const unsigned long long*)&j.row);
        double w;
        const int last = slice_warp(p, row, __ldcg(&j.pm), __ldcg(&j.ips), __ldcg(&j.invT), s_hrej, nrej, ph, w);
        if (lane == 0) { s_w[warp] = w; s_last[warp] = last; }
        walk_sync();
        if (tid == 0) {                                  // the warps' sums in order
            int l = -1;
            for (int i = 0; i < HS_ROW_THREADS / 32; ++i) l = max(l, s_last[i]);
            p.jobs[b].sum[ph] = sum8(s_w[0], s_w[1], s_w[2], s_w[3], s_w[4], s_w[5], s_w[6], s_w[7]);
            p.jobs[b].last[ph] = l;
            asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(&p.det_cnt[2 * DET_MAX_BATCH + b]) : "memory");
        }
    }
    walk_sync();                                         // (the shared arrays are free again)
}
// A CTA that takes part in the sharing leaves; the last of `count` puts the counters of the draws back to zero.
__device__ __forceinline__ void det_leave(const AcceptParams& p, int seq, int count) {
    if (threadIdx.x == 0) {
        int* c = &p.det_cnt[3 * DET_MAX_BATCH + max(seq, 0)];
        int old;
        asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(old) : "l"(c) : "memory");
        if (old == count - 1) {
            for (int b = seq < 0 ? 0 : seq; b < (seq < 0 ? p.batch : seq + 1); ++b)
                p.det_cnt[b] = p.det_cnt[DET_MAX_BATCH + b] = p.det_cnt[2 * DET_MAX_BATCH + b] = 0;
            *c = 0;
        }
    }
}

// Acceptance of sequence b with deterministic proposals by HS_ROW_THREADS threads of a CTA: at node cur with p =
// softmax(target row / T) the kept children are tried in index order; child x with token t is accepted iff
// u_x < min(1, p_t / W), W = 1 - (mass of the tokens rejected at this node so far); a rejection removes t.  When no
// candidate is left the bonus token is drawn by inverse CDF in token order from p without the rejected tokens.
__device__ __noinline__ void deterministic_walk(const AcceptParams& p, int b) {
    __shared__ int s_tok[HS_MAX_NODES], s_orig[HS_MAX_NODES], s_rej[HS_MAX_NODES];
    __shared__ unsigned int s_kids[HS_MAX_NODES][HS_MAX_NODES / 32];     // kept children of a node as a bit mask
    __shared__ float2 s_ms[HS_MAX_NODES];                       // {max, sum} of the node's own target row
    __shared__ float s_pt[HS_MAX_NODES];                        // p(token of the node | its parent)
    __shared__ unsigned char s_event[HS_MAX_NODES];
    __shared__ double s_cross[2];                               // mass ahead of the slice with the crossing, the goal
    __shared__ int s_phx;
    __shared__ double s_scan[HS_ROW_THREADS / 32];
    __shared__ double s_phase[DET_SLICES];
    __shared__ double s_wp[DET_SLICES][HS_ROW_THREADS / 32];    // per (slice, warp) sums where nobody helps
    __shared__ int s_pick[2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthr = HS_ROW_THREADS;
    const int koff = p.pr.keep_off[b];
    const int nk = min(p.pr.n_keep[b], HS_MAX_NODES);
    const int nbase = p.node_off[b];
    const int cap = p.out.path_cap;
    for (int j = tid; j < cap; j += nthr) {
        p.out.path_nodes[b * cap + j] = -1;
        p.out.path_compact[b * cap + j] = -1;
        p.out.path_tokens[b * cap + j] = -1;
    }
    // (HS_ROW_THREADS >= HS_MAX_NODES: thread j has node j)
    const int j = tid;
    int par = -1, tok = 0;
    float u = 0.f;
    for (int i = tid; i < HS_MAX_NODES * (HS_MAX_NODES / 32); i += nthr) (&s_kids[0][0])[i] = 0u;
    if (tid == 0) { s_pick[0] = 0x7fffffff; s_pick[1] = -1; }
    const float ufin = p.uniforms ? p.uniforms[p.n_nodes_total + b] : philox_uniform(p.seed, p.offset, b, 0, 1);
    if (j < nk) {
        const int orig = p.pr.keep_idx[koff + j];
        par = p.pr.new_parent[koff + j];
        s_orig[j] = orig;
        s_ms[j] = __ldcg(&p.ro.tgt_ms[koff + j]);                // written by another CTA of this launch
        tok = p.token[nbase + orig];
        u = p.uniforms ? p.uniforms[nbase + orig] : philox_uniform(p.seed, p.offset, b, orig, 0);
        s_tok[j] = tok;
    }
    const float invT = LOG2E / p.temperature[b];
    const size_t esz = p.is_bf16 ? 2 : 4;
    walk_sync();
    const bool cand = j > 0 && j < nk && par >= 0 && par < j;
    if (cand) atomicOr(&s_kids[par][j >> 5], 1u << (j & 31));
    auto target_row = [&](int i) {
        return (const char*)p.target + (size_t)(p.target_layout == HS_ROWS_ORIGINAL ? nbase + s_orig[i] : koff + i) * p.row_stride * esz;
    };
    // Every candidate's probability under its parent's target row, all nodes at once (one round trip instead of one per
    // sibling test).  A candidate is only tested after its earlier siblings were rejected, so W = 1 - sum of their
    // probabilities, and with it the test's outcome, is known ahead of the walk.
    float pt = 0.f;
    if (cand) {
        const float2 ms = s_ms[par];
        pt = exp2f((fmaxf(load_logit(target_row(par), p.is_bf16, tok), -1e30f) - ms.x) * invT) * (1.f / ms.y);
    }
    walk_sync();                                                 // s_kids
    auto earlier = [&](int w) {                                  // this node's siblings ahead of it, by words
        return w < j >> 5 ? s_kids[par][w] : (w == j >> 5 ? s_kids[par][w] & ((1u << (j & 31)) - 1u) : 0u);
    };
    if (cand) {
#pragma unroll
        for (int w = 0; w < HS_MAX_NODES / 32; ++w)              // a token rejected at this node has left the residual
            for (unsigned int m = earlier(w); m; m &= m - 1)
                if (s_tok[w * 32 + __ffs(m) - 1] == tok) pt = 0.f;
    }
    if (j < HS_MAX_NODES) s_pt[j] = pt;
    walk_sync();
    int event = 0;                                               // 1: accepted when tested, 2: rejected and nothing is left
    if (cand) {
        double W = 1.0;
#pragma unroll
        for (int w = 0; w < HS_MAX_NODES / 32; ++w)
            for (unsigned int m = earlier(w); m; m &= m - 1) W -= (double)s_pt[w * 32 + __ffs(m) - 1];
        const float a = fminf(1.f, pt / (float)W);
        event = u < a ? 1 : (!(W - (double)pt > 0.0) ? 2 : 0);   // (2: the walk falls back to p)
    }
    if (j < HS_MAX_NODES) s_event[j] = (unsigned char)event;
    walk_sync();
    // Every warp walks the tree by itself and takes the same way: no barrier until the walk ends.
    int cur = 0, len = 0, bonus = -1;
    for (int step = 0; step < nk; ++step) {
        if (tid == 0 && len < cap) {
            p.out.path_compact[b * cap + len] = cur;
            p.out.path_nodes[b * cap + len] = s_orig[cur];
        }
        // the kept children of cur in index order: the first one with an event decides
        unsigned int rej[HS_MAX_NODES / 32];                     // children that have been rejected
        int first = -1;
#pragma unroll
        for (int w = HS_MAX_NODES / 32 - 1; w >= 0; --w) {
            rej[w] = s_kids[cur][w];
            const unsigned int ev = __ballot_sync(HS_FULL_MASK, (rej[w] >> lane & 1u) && s_event[w * 32 + lane] != 0);
            if (ev) first = w * 32 + __ffs(ev) - 1;
        }
        if (first >= 0 && s_event[first] == 1) {
            if (tid == 0 && len < cap) p.out.path_tokens[b * cap + len] = s_tok[first];
            cur = first;
            ++len;
            continue;
        }
        if (first >= 0) {
#pragma unroll
            for (int w = 0; w < HS_MAX_NODES / 32; ++w) rej[w] = 0u;
        }
        const char* prow = target_row(cur);
        const float pm = s_ms[cur].x, ips = 1.f / s_ms[cur].y;
        int nrej = 0;                                            // the rejected tokens as a list, in index order
#pragma unroll
        for (int w = 0; w < HS_MAX_NODES / 32; ++w) {
            if (warp == 0 && (rej[w] >> lane & 1u)) s_rej[nrej + __popc(rej[w] & ((1u << lane) - 1u))] = s_tok[w * 32 + lane];
            nrej += __popc(rej[w]);
        }
        // ---- the bonus token: inverse CDF over the vocabulary without the rejected tokens -------------------
        // The row is taken in slices of nthr * 4 vectors; in a slice thread t owns 4 consecutive 16-byte vectors (all
        // loads in flight together), so token order is (slice, thread, token).  The slices are summed first - by every
        // CTA of the launch that is free, where the launch shares draws; then the one that holds the crossing is
        // summed again and scanned.  (At most DET_SLICES: the launcher refuses vocabularies of more than 32 chunks.)
        walk_sync();                                         // s_rej
        const int nph = det_slices(p), ve = p.is_bf16 ? 8 : 4;
        if (p.jobs) {
            DetJob& job = p.jobs[b];
            for (int k = tid; k < nrej; k += nthr) job.rej[k] = s_rej[k];
            if (tid == 0) { job.row = prow; job.pm = pm; job.ips = ips; job.invT = invT; job.nrej = nrej; }
            walk_sync();
            if (tid == 0) st_release_gpu(&p.det_cnt[b], 1);
            det_help(p, b, true);
            if (tid == 0) {                                  // slices taken by others: they are at work on them
                const unsigned long long t0 = global_timer_ns();
                while (ld_acquire_gpu(&p.det_cnt[2 * DET_MAX_BATCH + b]) < nph)
                    if (global_timer_ns() - t0 > HS_WAIT_LIMIT_NS) { atomicExch(p.err, (int)HS_ERR_TIMEOUT); break; }
            }
            walk_sync();
            for (int ph = tid; ph < nph; ph += nthr) {
                s_phase[ph] = __ldcg(&job.sum[ph]);
                const int l = __ldcg(&job.last[ph]);
                if (l >= 0) atomicMax(&s_pick[1], l);
            }
        } else {
            int last = -1;
#pragma unroll 2
            for (int ph = 0; ph < nph; ++ph) {
                double w;
                last = max(last, slice_warp(p, prow, pm, ips, invT, s_rej, nrej, ph, w));
                if (lane == 0) s_wp[ph][warp] = w;           // (no barrier per slice: the loads of the next one go out)
            }
            if (lane == 0 && last >= 0) atomicMax(&s_pick[1], last);
            walk_sync();
            for (int ph = tid; ph < nph; ph += nthr) {
                const double* w = s_wp[ph];
                s_phase[ph] = sum8(w[0], w[1], w[2], w[3], w[4], w[5], w[6], w[7]);
            }
        }
        walk_sync();
        if (warp == 0) {
            // running totals over the (at most 64) slices; the first one that exceeds the goal holds the crossing
            static_assert(DET_SLICES == 64, "two slices per lane");
            const double v0 = lane < nph ? s_phase[lane] : 0.0, v1 = lane + 32 < nph ? s_phase[lane + 32] : 0.0;
            double i0 = v0, i1 = v1;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const double u0 = __shfl_up_sync(HS_FULL_MASK, i0, o), u1 = __shfl_up_sync(HS_FULL_MASK, i1, o);
                if (lane >= o) { i0 += u0; i1 += u1; }
            }
            i1 += __shfl_sync(HS_FULL_MASK, i0, 31);
            const double goal = (double)ufin * __shfl_sync(HS_FULL_MASK, i1, 31);
            const unsigned int x0 = __ballot_sync(HS_FULL_MASK, lane < nph && i0 > goal);
            const unsigned int x1 = __ballot_sync(HS_FULL_MASK, lane + 32 < nph && i1 > goal);
            const int phx = x0 ? __ffs(x0) - 1 : (x1 ? 32 + __ffs(x1) - 1 : -1);
            if (lane == (phx & 31)) { s_cross[0] = phx < 32 ? i0 - v0 : i1 - v1; s_cross[1] = goal; }
            if (lane == 0) s_phx = phx;
        }
        walk_sync();
        if (s_phx >= 0) {
            const int phx = s_phx;
            const double goal = s_cross[1];
            float m[4][8];
            slice_mass(p, prow, pm, ips, invT, s_rej, nrej, phx, m);
            double qs[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) qs[q] = sum8(m[q]);
            const double mine = (qs[0] + qs[1]) + (qs[2] + qs[3]);
            double incl = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const double up = __shfl_up_sync(HS_FULL_MASK, incl, o);
                if (lane >= o) incl += up;
            }
            if (lane == 31) s_scan[warp] = incl;
            walk_sync();
            double ahead[HS_ROW_THREADS / 32];
#pragma unroll
            for (int w2 = 0; w2 < HS_ROW_THREADS / 32; ++w2) ahead[w2] = w2 < warp ? s_scan[w2] : 0.0;
            double run = s_cross[0] + (sum8(ahead[0], ahead[1], ahead[2], ahead[3], ahead[4], ahead[5], ahead[6], ahead[7]) + (incl - mine));
            if (run <= goal && run + mine > goal) {              // the crossing lies in this thread's tokens
                int pick = -1, lastp = -1;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (pick < 0 && run + qs[q] > goal) {        // the vector with the crossing
                        double r2 = run;
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            const int t = (phx * nthr * 4 + tid * 4 + q) * ve + e;
                            r2 += (double)m[q][e];
                            if (m[q][e] > 0.f) lastp = t;
                            if (pick < 0 && r2 > goal) pick = t;
                        }
                        if (pick < 0) pick = lastp;              // (rounding left none: the vector's last token of positive mass)
                    }
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        if (m[q][e] > 0.f) lastp = (phx * nthr * 4 + tid * 4 + q) * ve + e;
                    run += qs[q];
                }
                if (pick < 0) pick = lastp;
                if (pick >= 0) atomicMin(&s_pick[0], pick);
            }
        }
        walk_sync();
        bonus = s_pick[0] != 0x7fffffff ? s_pick[0] : max(s_pick[1], 0);
        break;
    }
    if (tid == 0) {
        p.out.accept_len[b] = len;
        p.out.bonus_token[b] = bonus;
        p.out.terminal_rank[b] = p.pr.keep_rank[koff + cur];
        p.out.status[b] = HS_OK;
    }
}

// What a CTA of the chunk kernel does for a deterministic-proposal sequence once its chunk is merged (one call, so that the
// kernel's own registers are not shaped by it): the CTA that completed the last row walks, the others take slices of the draw.
__device__ __noinline__ void det_chunk_tail(const AcceptParams& p, int b, int nk, bool walk) {
    if (walk) deterministic_walk(p, b);
    else if (p.jobs) det_help(p, b, false);
    if (p.jobs) det_leave(p, b, nk * p.chunks);
}
