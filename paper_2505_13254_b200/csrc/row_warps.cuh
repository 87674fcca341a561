// The entropy pass for launches with many rows: every warp on its own.  Included by row_stats.cu.
//
// The matrix is a stream of rounds of 128 vectors (row after row, a row's last round may be partial) that is cut into equal
// contiguous shares, one per warp of the device (16 warps per SM).  A warp walks its share straight from global memory, four
// 16-byte vectors per lane and round with the next round in flight, and meets nobody: no barrier, no ring of slots.  Per round it
// takes the packed maximum of its 32 logits a lane (kept in shared memory), then sum e^(x-ref) and sum x e^(x-ref) against
// a reference that all lanes share and that only moves when a logit exceeds it by more than 20 (fp32 sums keep their
// relative precision for any reference near the maximum).  At the end of a row segment: a lower bound of the K-th largest
// logit from the 32 lane maxima, the few (lane, round) cells whose maximum reaches it are read again and ranked.  A row that
// lies in several shares leaves {ref, s, u, max} and K keys per share; the last warp to arrive merges.
//
// Why: the same arithmetic behind a ring of 32 KiB items and CTA-wide row ends ran at half of the issue slots with no pipe
// above 40 % busy (16 warps in lockstep, four barriers per row, 11 instructions per logit); warps that drift apart hide one
// another's row ends, and without the item bookkeeping a logit costs 7.2.  560 rows of 128256 bf16: 50.3 -> 36.8 us (3.9 TB/s).
// What bounds it, from time stamps of every warp: the rounds of 19 of 20 shares are over after 29 us, read at 5.0 TB/s (1600 clocks a round, 32 KiB of loads in
// flight on an SM); then all warps are at the row end of their last segment at once, 4.8 us each, and for 7 us next to nothing is read.  Shorter shares pay the same
// end: 83 MB 18 of 25 us, 74 MB in rows of 32000 18 of 25.5.  1088 rows: 93.8 -> 62 us, 240 rows: 37.8 -> 21.5 us, 1088 rows of 32000: 44.0 -> 24.2 us.
#pragma once

#define QW_WARPS 16
#define QW_THREADS (QW_WARPS * 32)
#define QW_ROW_END 4                    // what the end of a row segment costs, in rounds
#define QW_GROUPS 32                    // cells a lane keeps maxima for: rounds, or groups of 2^k rounds on long segments
#define QW_CAND 128                     // candidates of a segment
#define QW_MAX_SEGS 32                  // shares a row may lie in: one lane each when they merge

struct WarpSmem {
    float gm[QW_GROUPS][32];            // maxima per (group of rounds, lane)
    __align__(16) float lm[32];         // the lanes' maxima of the segment
    unsigned long long cand[QW_CAND];
    unsigned long long keys[QW_MAX_SEGS][HS_MAX_TOPK];     // merge: the sorted keys of the row's shares
    unsigned short hit[QW_GROUPS * 32];                    // cells to read again: group * 32 + lane
};
#define QW_SMEM_BYTES (QW_WARPS * sizeof(WarpSmem))

// s += e, u += e x of a lane's logits of a round, e = 2^(x log2(e) + n).  CLAMP keeps 0 * x finite for x = -inf.
template <bool BF16, bool CLAMP>
__device__ __forceinline__ void round_sums(const uint4 (&d)[4], float n, float2& s2, float2& u2) {
    const float2 l2 = make_float2(LOG2E, LOG2E), n2 = make_float2(n, n);
    const unsigned int* w = reinterpret_cast<const unsigned int*>(&d[0]);
#pragma unroll
    for (int q = 0; q < (BF16 ? 16 : 8); ++q) {
        float2 x = BF16 ? make_float2(bf16_lo(w[q]), bf16_hi(w[q]))
                        : make_float2(__uint_as_float(w[2 * q]), __uint_as_float(w[2 * q + 1]));
        if (CLAMP) { x.x = fmaxf(x.x, -1e30f); x.y = fmaxf(x.y, -1e30f); }
        const float2 t = fma2_ftz(x, l2, n2);
        const float2 e = make_float2(ex2f(t.x), ex2f(t.y));
        s2 = add2_ftz(s2, e);
        u2 = fma2_ftz(e, x, u2);
    }
}
// A lane's four vectors into its running sums; rm: the largest of them.  The reference is the same in all lanes of the warp.
template <bool BF16>
__device__ __forceinline__ void fold_round(const uint4 (&d)[4], float& ref, float& nref, float2& s2, float2& u2, float& rm) {
    rm = round_max<BF16>(d);
    if (__any_sync(HS_FULL_MASK, rm > ref + 20.f)) {
        const float nr = fmaxf(ref, order_bits_float(__reduce_max_sync(HS_FULL_MASK, float_order_bits(rm))));
        const float f = ref == -CUDART_INF_F ? 0.f : ex2f((ref - nr) * LOG2E);
        s2.x *= f; s2.y *= f; u2.x *= f; u2.y *= f;
        ref = nr;
        nref = -nr * LOG2E;
    }
    float2 s = s2, u = u2;
    round_sums<BF16, false>(d, nref, s, u);
    if (__any_sync(HS_FULL_MASK, !(u.x + u.y == u.x + u.y))) {      // a -inf among them (0 * x): again, with care
        s = s2; u = u2;
        round_sums<BF16, true>(d, nref, s, u);
    }
    s2 = s; u2 = u;
}

// K largest keys of rounds [r0, r1) of a row by repeated search (heavy ties: more candidates than the list holds).
template <bool BF16>
__device__ __noinline__ void topk_rounds_warp(const QuantParams& p, const uint4* rowv, int r0, int r1, unsigned long long* out, int lane) {
    constexpr int VE = BF16 ? 8 : 4;
    unsigned long long last = ~0ull;
    for (int i = 0; i < p.K; ++i) {
        unsigned long long best = 0ull;
        if (last != 0ull)
            for (int r = r0; r < r1; ++r) {
                uint4 d[4];
                load_round<BF16>(p, rowv, r, lane, d);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    float x[8];
                    unpack<BF16>(d[j], x);
                    const int base = (r * ROUND_VECS + j * 32 + lane) * VE;
#pragma unroll
                    for (int e = 0; e < VE; ++e)
                        if (x[e] > -CUDART_INF_F) {
                            const unsigned long long k = make_key(x[e], base + e);
                            if (k < last && k > best) best = k;
                        }
                }
            }
        int src;
        last = warp_best_key(best, src);
        if (lane == 0) out[i] = last;
    }
}

template <bool BF16>
__global__ void __launch_bounds__(QW_THREADS, 1) quantify_warp_kernel(const __grid_constant__ QuantParams p) {
    constexpr int VE = BF16 ? 8 : 4;
    extern __shared__ __align__(128) unsigned char s_dyn[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    WarpSmem& sm = reinterpret_cast<WarpSmem*>(s_dyn)[warp];
    const int K = p.K, c = blockIdx.x * QW_WARPS + warp;
    const int rr = (p.nvec + ROUND_VECS - 1) / ROUND_VECS;            // rounds per row
    const int rv = rr + p.extra;                                  // places per row in the stream: its end costs `extra` rounds
    const int total = p.rows * rv;
    int g = min(c * p.per, total);
    const int g1 = min(g + p.per, total);
    if (!p.prefetch) pdl_wait();                                  // (see quantify_cluster_kernel on the order of the two)
    pdl_launch_dependents();
    bool waited = !p.prefetch;

    while (g < g1) {
        // ---- one segment: rounds [r0, r1) of `row` --------------------------------------------------------------------
        const int row = g / rv, x0 = row * rv + p.extra;          // (the row's rounds stand behind its extra places)
        const int r0 = max(g - x0, 0), r1 = min(rr, g1 - x0);
        g = min(g1, x0 + rr);
        if (r0 >= r1) continue;
        const uint4* rowv = (const uint4*)((const char*)p.logits + (size_t)row * p.row_stride * (BF16 ? 2 : 4));
        int gsh = 0;                                              // rounds per cell = 2^gsh
        while ((r1 - r0 - 1) >> gsh >= QW_GROUPS) ++gsh;
        float ref = -CUDART_INF_F, nref = 0.f, lm = -CUDART_INF_F, cm = -CUDART_INF_F;
        float2 s2 = make_float2(0.f, 0.f), u2 = make_float2(0.f, 0.f);
        auto consume = [&](const uint4 (&d)[4], int r) {
            float rm;
            fold_round<BF16>(d, ref, nref, s2, u2, rm);
            cm = fmaxf(cm, rm);
            const int i = r - r0;
            if (gsh == 0 || ((i + 1) & ((1 << gsh) - 1)) == 0 || r + 1 == r1) {
                sm.gm[i >> gsh][lane] = cm;
                lm = fmaxf(lm, cm);
                cm = -CUDART_INF_F;
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
        // ---- Top-K of the segment ------------------------------------------------------------------------------------------
        __syncwarp();
        // (maxima of disjoint sets are distinct logits: the K-th largest of the 32 lane maxima bounds the K-th largest logit)
        sm.lm[lane] = lm;
        __syncwarp();
        int ge = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float4 f4 = reinterpret_cast<const float4*>(sm.lm)[i];
            ge += (f4.x >= lm) + (f4.y >= lm) + (f4.z >= lm) + (f4.w >= lm);
        }
        const float tau = order_bits_float(__reduce_max_sync(HS_FULL_MASK, float_order_bits(ge >= K ? lm : -CUDART_INF_F)));
        const unsigned int below = (1u << lane) - 1u;
        const int ncell = ((r1 - r0 - 1) >> gsh) + 1;
        int nhit = 0;
        for (int i0 = 0; i0 < ncell; i0 += 8) {
            float m[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) m[i] = sm.gm[(i0 + i) & (QW_GROUPS - 1)][lane];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const unsigned int b = __ballot_sync(HS_FULL_MASK, i0 + i < ncell && m[i] >= tau && m[i] > -CUDART_INF_F);
                if (b >> lane & 1u) sm.hit[nhit + __popc(b & below)] = (unsigned short)((i0 + i) * 32 + lane);
                nhit += __popc(b);
            }
        }
        __syncwarp();
        int ncand = 0;
        // a cell is four vectors per round, four lanes; sixteen cells' reads are in flight together
        for (int h0 = 0; h0 < nhit && ncand <= QW_CAND; h0 += 16)
            for (int q = 0; q < 1 << gsh; ++q) {
                uint4 d[2];
                int vec[2];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int h = h0 + i * 8 + (lane >> 2);
                    vec[i] = -1;
                    if (h < nhit) {
                        const int cell = sm.hit[h], rc = r0 + ((cell >> 5) << gsh) + q;
                        const int v = rc * ROUND_VECS + (lane & 3) * 32 + (cell & 31);
                        if (rc < r1 && v < p.nvec) vec[i] = v;
                    }
                    d[i] = vec[i] >= 0 ? __ldg(rowv + vec[i]) : make_uint4(0, 0, 0, 0);
                }
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    float x[8];
                    unpack<BF16>(d[i], x);
#pragma unroll
                    for (int e = 0; e < VE; ++e) {
                        const int idx = vec[i] * VE + e;
                        const bool take = vec[i] >= 0 && x[e] >= tau && x[e] > -CUDART_INF_F && idx < p.vocab;
                        const unsigned int b = __ballot_sync(HS_FULL_MASK, take);
                        const int at = ncand + __popc(b & below);
                        if (take && at < QW_CAND) sm.cand[at] = make_key(x[e], idx);
                        ncand += __popc(b);
                    }
                }
            }
        // sorted, best first: lane i gets the i-th key (0 = none)
        unsigned long long mine = 0ull;
        __syncwarp();
        if (ncand <= 32) {                                        // (the usual case: ranked by counting)
            const unsigned long long k = lane < ncand ? sm.cand[lane] : 0ull;
            int rank = 0;
            for (int i = 0; i < ncand; ++i) rank += sm.cand[i] > k;
            __syncwarp();
            if (lane < ncand) sm.cand[rank] = k;
            __syncwarp();
            if (lane < min(ncand, K)) mine = sm.cand[lane];
        } else if (ncand <= QW_CAND) {
            unsigned long long k[QW_CAND / 32];
#pragma unroll
            for (int i = 0; i < QW_CAND / 32; ++i) k[i] = i * 32 + lane < ncand ? sm.cand[i * 32 + lane] : 0ull;
            for (int i = 0; i < K; ++i) {
                unsigned long long b = k[0];
#pragma unroll
                for (int q = 1; q < QW_CAND / 32; ++q) b = k[q] > b ? k[q] : b;
                int src;
                const unsigned long long best = warp_best_key(b, src);
                if (lane == i) mine = best;
#pragma unroll
                for (int q = 0; q < QW_CAND / 32; ++q) if (k[q] == best) k[q] = 0ull;
            }
        } else {
            topk_rounds_warp<BF16>(p, rowv, r0, r1, sm.cand, lane);
            __syncwarp();
            if (lane < K) mine = sm.cand[lane];
        }
        float S = warp_sum(s2.x + s2.y), U = warp_sum(u2.x + u2.y);
        float M = order_bits_float(__reduce_max_sync(HS_FULL_MASK, float_order_bits(lm)));
        if (!waited) { pdl_wait(); waited = true; }               // from here on results go to global memory
        const int c_first = x0 / p.per, nseg = (x0 + rr - 1) / p.per - c_first + 1;
        bool done = nseg == 1;
        if (!done) {
            // a share has at most two partial rows: slot 0 for one that began in an earlier share, slot 1 for one that goes on
            const int ps = 2 * c + (r0 > 0 ? 0 : 1);
            if (lane < HS_MAX_TOPK) p.part_keys[(size_t)ps * HS_MAX_TOPK + lane] = mine;
            if (lane == 0) p.part_stats[ps] = make_float4(ref, S, U, M);
            __syncwarp();
            int last = 0;
            if (lane == 0) {
                // one release-acquire arrival at device scope: the partial is visible to whoever arrives last
                int old;
                asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(old) : "l"(&p.row_cnt[row]) : "memory");
                last = old == nseg - 1;
                if (last) p.row_cnt[row] = 0;                     // ready for the next launch
            }
            done = __shfl_sync(HS_FULL_MASK, last, 0) != 0;
            if (done) {
                float4 st = make_float4(-CUDART_INF_F, 0.f, 0.f, -CUDART_INF_F);
                if (lane < nseg) st = __ldcg(&p.part_stats[2 * (c_first + lane) + (lane == 0 ? 1 : 0)]);
                for (int q0 = 0; q0 < nseg; q0 += 16) {           // two shares' keys per load, eight loads in flight
                    unsigned long long k[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int q = q0 + 2 * i + (lane >> 4), ps2 = 2 * (c_first + q) + (q == 0 ? 1 : 0);
                        k[i] = q < nseg ? __ldcg(&p.part_keys[(size_t)ps2 * HS_MAX_TOPK + (lane & 15)]) : 0ull;
                    }
#pragma unroll
                    for (int i = 0; i < 8; ++i) sm.keys[q0 + 2 * i + (lane >> 4)][lane & 15] = k[i];
                }
                ref = warp_max(st.x);
                const float f = st.x == -CUDART_INF_F ? 0.f : ex2f((st.x - ref) * LOG2E);
                S = warp_sum(st.y * f);
                U = warp_sum(st.z * f);
                M = warp_max(st.w);
                __syncwarp();
                // the shares' lists are sorted: K times the best head
                int at = 0;
                unsigned long long head = lane < nseg ? sm.keys[lane][0] : 0ull;
                mine = 0ull;
                for (int i = 0; i < K; ++i) {
                    int src;
                    const unsigned long long best = warp_best_key(head, src);
                    if (lane == i) mine = best;
                    if (lane == src) { ++at; head = at < K ? sm.keys[lane][at] : 0ull; }
                }
            }
        }
        if (done) finalize_row(p, row, M, ref, S, U, mine, lane);
        __syncwarp();
    }
}
