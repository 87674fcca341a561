// Stratifier training in one launch: the whole grid sorts, then scores layer after layer.  Included by cart.cu, whose header
// describes the problem and whose layer code it uses.
//
// A cooperative launch (its CTAs wait for one another: all of them have to run at once), one CTA per SM at most, each with an equal
// share of the samples, at most eight per thread.  The sort is a least-significant-digit radix sort over the bits in which the feature
// values differ (their order bits less the smallest: passes of up to ten bits, three for up to 30 such bits, else four of eight).  A pass
// ranks and counts the digits of every share and brings the share into their order in shared memory, the counts of all shares become
// offsets (up to 32 shares: every CTA adds up the others' itself; more: 32 digits to a CTA and one barrier more), and the shares write their
// keys, equal digits together: two grid barriers, or three, of 1.2 us.  The share of the sorted order that a CTA then holds stays in its
// shared memory for all layers; a layer costs one barrier, behind which every CTA works out the same new boundaries from the
// shares' best splits.
//
// Why: nine launches (pack, four look-back passes, sums, three layers) took 70 us at any size above one CTA's and 125 us at 2^20 samples:
// their starts, the look-back chains and the reloads, not the work.  Now 41 us at 8193 samples, 43 at 20000, 54 at 200000, 76 at 2^20 and depth
// 3: there 21 us ranking (ten ballots a key), 11 us fp64 sums of the layers, 17 us in 14 barriers (one for the range, three a pass, one for
// the sums, one a layer).  Two CTAs of 512 threads per SM: 92 us (twice the entries and counts to read for every CTA).
#pragma once

#define CG_THREADS 1024
#define CG_WARPS (CG_THREADS / 32)
#define CG_ITEMS 8
#define CG_SHARE (CG_THREADS * CG_ITEMS)     // samples per CTA at most
#define CG_MAX_DIGITS 1024
#define CG_MAX_CTAS 256
#define CG_DIRECT 32                         // shares up to which every CTA adds up the others' counts itself

struct CartGrid {
    const float* x;
    const float* y;
    int n, per, depth;             // per: samples per CTA
    unsigned long long* keys;
    unsigned long long* keys2;
    unsigned int* cnt;             // [CTAs][digits] digit counts of the shares, then their offsets among the keys of the digit
    unsigned int* tot;             // [CG_MAX_DIGITS]
    uint2* range;                  // [CTAs] smallest and largest order bits of a share
    double* blk;                   // [CTAs][2] sums of y and y^2 of a share
    LayerEntry* part;              // [2][CTAs + CT_MAX_NODES] best split of a (share, node), entry share + node
    unsigned int* bar;             // [2] arrivals at grid barriers, CTAs that have left (zero between calls)
    float* thresholds;
    int* status;
    int* err;
};

struct CartGridSmem {
    unsigned long long key[CG_SHARE * 9 / 8 + 2];        // sort: the share by digit; layers: the key ahead of the share, then its keys
    unsigned short cnt[CG_WARPS * CG_MAX_DIGITS];        // sort: the warps' digit counters
    unsigned int off[CG_MAX_DIGITS];                     // sort: where the share's keys of a digit go, less their place in the share
    LayerSmem s;
    double w[CG_WARPS][2];
    unsigned int scan[CG_WARPS], ex[CG_WARPS][33];
    unsigned int lo, hi;
    int bnd2[2 * CT_MAX_NODES + 1];
    double sy2[2 * CT_MAX_NODES + 1], syy2[2 * CT_MAX_NODES + 1];
    int bad;
};
static_assert(CT_MAX_NODES <= CG_WARPS, "a warp per node");
static_assert(CG_WARPS == 32, "a warp per digit of a block of 32, a lane per run of shares");
static_assert(sizeof(CartGridSmem) <= 220 * 1024 && CG_MAX_DIGITS <= CG_THREADS, "one CTA per SM");

// A CTA leaves (one thread): the last one puts the counters back.  Every CTA leaves behind its last wait, so nobody looks at them any more.
__device__ __forceinline__ void grid_leave(const CartGrid& p) {
    if (atomicAdd(&p.bar[1], 1u) == gridDim.x - 1) { p.bar[0] = 0u; p.bar[1] = 0u; }
}

// All CTAs of the grid have come this far and see what the others stored ahead of it.  Bounded; false for all threads when the wait expired:
// the CTA has left then and has to return at once.  Above all it arrives nowhere any more: no CTA passes a later barrier, so nobody reads
// what has not been written, and CTA 0, whose last wait is for all, gives up as well and says so in the status.
__device__ __forceinline__ bool grid_sync(const CartGrid& p, unsigned int& round, bool wait = true) {
    ++round;
    __syncthreads();
    int bad = 0;
    if (threadIdx.x == 0) {
        unsigned int old;
        asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(old) : "l"(p.bar) : "memory");
        if (wait && old + 1 < round * gridDim.x) {
            const unsigned long long t0 = global_timer_ns();
            unsigned int v;
            do {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p.bar) : "memory");
                if (v < round * gridDim.x && global_timer_ns() - t0 > HS_WAIT_LIMIT_NS) bad = 1;
            } while (v < round * gridDim.x && !bad);
            if (bad) {
                atomicExch(p.err, (int)HS_ERR_TIMEOUT);
                if (blockIdx.x == 0) *p.status = HS_ERR_TIMEOUT;
                grid_leave(p);
            }
        }
    }
    return __syncthreads_or(bad) == 0;
}

// exclusive prefix of one value per thread over the CTA
__device__ __forceinline__ unsigned int scan_cta(unsigned int v, unsigned int* s_w) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const unsigned int u = __shfl_up_sync(HS_FULL_MASK, incl, o); if (lane >= o) incl += u; }
    __syncthreads();                                     // (s_w may still be read from the call before)
    if (lane == 31) s_w[warp] = incl;
    __syncthreads();
    unsigned int before = incl - v;
    const unsigned int mine = lane < warp ? s_w[lane] : 0u;
    return before + __reduce_add_sync(HS_FULL_MASK, mine);
}

__global__ void __launch_bounds__(CG_THREADS, 1) cart_grid_kernel(const __grid_constant__ CartGrid p) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    CartGridSmem& sm = *reinterpret_cast<CartGridSmem*>(s_dyn);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, c = blockIdx.x, G = gridDim.x;
    const int base = min(c * p.per, p.n), mine = min(base + p.per, p.n) - base;      // this CTA's share
    const int nit = (p.per + CG_THREADS - 1) / CG_THREADS;
    unsigned int round = 0;

    // ---- the keys, and the range of their order bits -------------------------------------------------------------------
    // (a warp has 32 nit consecutive samples, item-major)
    unsigned long long k[CG_ITEMS];
    unsigned int lo = ~0u, hi = 0u;
    if (tid == 0) { sm.lo = ~0u; sm.hi = 0u; }
#pragma unroll
    for (int i = 0; i < CG_ITEMS; ++i) {
        const int j = warp * 32 * nit + i * 32 + lane;
        k[i] = ~0ull;
        if (i < nit && j < mine) {
            k[i] = cart_key(p.x[base + j], p.y[base + j]);
            lo = min(lo, (unsigned int)(k[i] >> 32)); hi = max(hi, (unsigned int)(k[i] >> 32));
        }
    }
    __syncthreads();
    lo = __reduce_min_sync(HS_FULL_MASK, lo); hi = __reduce_max_sync(HS_FULL_MASK, hi);
    if (lane == 0) { atomicMin(&sm.lo, lo); atomicMax(&sm.hi, hi); }
    __syncthreads();
    if (tid == 0) p.range[c] = make_uint2(sm.lo, sm.hi);
    if (!grid_sync(p, round)) return;
    {
        const uint2 r = tid < G ? __ldcg(&p.range[tid]) : make_uint2(~0u, 0u);
        lo = __reduce_min_sync(HS_FULL_MASK, r.x); hi = __reduce_max_sync(HS_FULL_MASK, r.y);
        if (lane == 0) { atomicMin(&sm.lo, lo); atomicMax(&sm.hi, hi); }
        __syncthreads();
        lo = sm.lo; hi = sm.hi;
    }
    const int bits = 32 - __clz((int)(hi - lo));             // in which the feature values differ
    const int passes = bits <= 30 ? (bits + 9) / 10 : 4, width = passes ? (bits + passes - 1) / passes : 0;
    const int ND = 1 << width;

    // ---- the sort ------------------------------------------------------------------------------------------------------
    for (int pass = 0; pass < passes; ++pass) {
        const unsigned long long* in = (pass & 1) ? p.keys2 : p.keys;
        unsigned long long* out = (pass & 1) ? p.keys : p.keys2;
        unsigned short* wcnt = sm.cnt + (warp << width);     // this warp's counters
        for (int i = tid; i < CG_WARPS * ND / 2; i += CG_THREADS) reinterpret_cast<unsigned int*>(sm.cnt)[i] = 0u;
        if (pass > 0) {
#pragma unroll
            for (int i = 0; i < CG_ITEMS; ++i) {
                const int j = warp * 32 * nit + i * 32 + lane;
                k[i] = i < nit && j < mine ? __ldcg(&in[base + j]) : ~0ull;
            }
        }
        __syncthreads();
        auto digit = [&](unsigned long long key) { return (((unsigned int)(key >> 32) - lo) >> (pass * width)) & (unsigned int)(ND - 1); };
        unsigned short rank[CG_ITEMS];
#pragma unroll
        for (int i = 0; i < CG_ITEMS; ++i) {
            if (i >= nit) break;
            const bool in_share = warp * 32 * nit + i * 32 + lane < mine;
            const unsigned int d = digit(k[i]);
            unsigned int peers = __ballot_sync(HS_FULL_MASK, in_share);
#pragma unroll
            for (int b = 0; b < 10; ++b) {
                if (b >= width) break;
                const unsigned int v = __ballot_sync(HS_FULL_MASK, (d >> b) & 1u);
                peers &= ((d >> b) & 1u) ? v : ~v;
            }
            if (in_share) rank[i] = (unsigned short)(wcnt[d] + __popc(peers & ((1u << lane) - 1u)));
            __syncwarp();
            if (in_share && (peers >> lane) == 1u) wcnt[d] = (unsigned short)(rank[i] + 1);       // (the highest lane of the group)
            __syncwarp();
        }
        __syncthreads();
        // thread t: digits 2 t and 2 t + 1 (ND is at least two).  Counts of the share, places of the warps' keys in the share by digit, and the
        // share written to shared memory in that order: equal digits then leave together.
        unsigned int ca = 0, cb = 0;
        if (2 * tid < ND) {
            unsigned int* pair = reinterpret_cast<unsigned int*>(sm.cnt) + tid;
#pragma unroll
            for (int w = 0; w < CG_WARPS; ++w) {
                const unsigned int v = pair[w << (width - 1)];
                pair[w << (width - 1)] = ca | cb << 16;
                ca += v & 0xffffu; cb += v >> 16;
            }
            reinterpret_cast<uint2*>(p.cnt + (size_t)c * ND)[tid] = make_uint2(ca, cb);
        }
        const unsigned int la = scan_cta(ca + cb, sm.scan);  // (place of digit 2 t in the share)
        if (2 * tid < ND) { sm.off[2 * tid] = la; sm.off[2 * tid + 1] = la + ca; }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < CG_ITEMS; ++i) {
            if (i >= nit) break;
            if (warp * 32 * nit + i * 32 + lane < mine) {
                const unsigned int d = digit(k[i]);
                sm.key[sm.off[d] + wcnt[d] + rank[i]] = k[i];
            }
        }
        if (!grid_sync(p, round)) return;
        unsigned int oa = 0, ob = 0, ta = 0, tb = 0;         // of digits 2 t and 2 t + 1: keys of the shares ahead, keys of all shares
        if (G <= CG_DIRECT) {
            if (2 * tid < ND)
                for (int q0 = 0; q0 < G; q0 += 16) {         // sixteen loads in flight
                    uint2 v[16];
#pragma unroll
                    for (int q = 0; q < 16; ++q)
                        v[q] = q0 + q < G ? __ldcg(reinterpret_cast<const uint2*>(p.cnt + (size_t)(q0 + q) * ND) + tid) : make_uint2(0u, 0u);
#pragma unroll
                    for (int q = 0; q < 16; ++q) {
                        if (q0 + q == c) { oa = ta; ob = tb; }
                        ta += v[q].x; tb += v[q].y;
                    }
                }
        } else {
            // 32 digits per CTA, a lane per digit; the shares are cut into as many runs as there are warps
            for (int d0 = c * 32; d0 < ND; d0 += G * 32) {
                const int run = (G + CG_WARPS - 1) / CG_WARPS, s0 = min(warp * run, G), s1 = min(s0 + run, G), d = d0 + lane;
                unsigned int v[CG_MAX_CTAS / CG_WARPS], sum = 0;
#pragma unroll
                for (int q = 0; q < CG_MAX_CTAS / CG_WARPS; ++q) {
                    v[q] = s0 + q < s1 && d < ND ? __ldcg(&p.cnt[(size_t)(s0 + q) * ND + d]) : 0u;
                }
#pragma unroll
                for (int q = 0; q < CG_MAX_CTAS / CG_WARPS; ++q) sum += v[q];
                sm.ex[warp][lane] = sum;
                __syncthreads();
                unsigned int incl = sm.ex[lane][warp];       // (warp w: digit d0 + w, lane r: run r)
                sum = incl;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) { const unsigned int u = __shfl_up_sync(HS_FULL_MASK, incl, o); if (lane >= o) incl += u; }
                sm.ex[lane][warp] = incl - sum;
                if (lane == 31 && d0 + warp < ND) p.tot[d0 + warp] = incl;
                __syncthreads();
                unsigned int before = sm.ex[warp][lane];
#pragma unroll
                for (int q = 0; q < CG_MAX_CTAS / CG_WARPS; ++q) {
                    if (s0 + q < s1 && d < ND) p.cnt[(size_t)(s0 + q) * ND + d] = before;
                    before += v[q];
                }
                __syncthreads();
            }
            if (!grid_sync(p, round)) return;
            if (2 * tid < ND) {
                const uint2 t2 = __ldcg(reinterpret_cast<const uint2*>(p.tot) + tid), o2 = __ldcg(reinterpret_cast<const uint2*>(p.cnt + (size_t)c * ND) + tid);
                ta = t2.x; tb = t2.y; oa = o2.x; ob = o2.y;
            }
        }
        {
            const unsigned int first = scan_cta(ta + tb, sm.scan);
            if (2 * tid < ND) { sm.off[2 * tid] = first + oa - la; sm.off[2 * tid + 1] = first + ta + ob - (la + ca); }
        }
        __syncthreads();
#pragma unroll 4
        for (int j = tid; j < mine; j += CG_THREADS) {
            const unsigned long long key = sm.key[j];
            const unsigned int to = sm.off[digit(key)] + j;
            if (to < (unsigned int)p.n) out[to] = key;       // (always, unless two calls share the workspace at a time)
        }
        if (!grid_sync(p, round)) return;
    }
    const unsigned long long* sorted = (passes & 1) ? p.keys2 : p.keys;

    // ---- running sums ----------------------------------------------------------------------------------------------------
    LayerSmem& s = sm.s;
    if (passes == 0) {                                       // (a single feature value: any order)
#pragma unroll
        for (int i = 0; i < CG_ITEMS; ++i) {
            const int j = warp * 32 * nit + i * 32 + lane;
            if (i < nit && j < mine) sm.key[1 + pad8(j)] = k[i];
        }
        if (tid == 0) sm.key[0] = base > 0 ? cart_key(p.x[base - 1], p.y[base - 1]) : 0ull;
    } else {
        for (int j = tid; j < mine; j += CG_THREADS) sm.key[1 + pad8(j)] = __ldcg(&sorted[base + j]);
        if (tid == 0) sm.key[0] = base > 0 ? __ldcg(&sorted[base - 1]) : 0ull;        // the key ahead of the share
    }
    __syncthreads();
    const int j0 = min(tid * nit, mine), cnt = min(j0 + nit, mine) - j0;
    auto key = [&](int j) { return j0 + j < 0 ? sm.key[0] : sm.key[1 + pad8(j0 + j)]; };
    double a = 0.0, b = 0.0;
    for (int j = 0; j < cnt; ++j) { const double v = key_y(key(j)); a += v; b += v * v; }
    {
        const double ta = a, tb = b;
        scan_pair<CG_WARPS>(a, b, sm.w);
        if (tid == CG_THREADS - 1) { p.blk[2 * c] = a + ta; p.blk[2 * c + 1] = b + tb; }
    }
    if (!grid_sync(p, round)) return;
    {
        // sums ahead of every share, in one fixed order: thread t has share t
        double ba = tid < G ? __ldcg(&p.blk[2 * tid]) : 0.0, bb = tid < G ? __ldcg(&p.blk[2 * tid + 1]) : 0.0;
        const double va = ba, vb = bb;
        scan_pair<CG_WARPS>(ba, bb, sm.w);
        if (tid == c) { s.sy[0] = ba; s.syy[0] = bb; }
        if (tid == G - 1) { s.sy[1] = ba + va; s.syy[1] = bb + vb; }
        __syncthreads();
        a += s.sy[0]; b += s.syy[0];
        __syncthreads();
        if (tid == 0) { s.bnd[0] = 0; s.bnd[1] = p.n; s.sy[0] = 0.0; s.syy[0] = 0.0; sm.bad = 0; }
        __syncthreads();
    }

    // ---- the layers ------------------------------------------------------------------------------------------------------
    const int stride = G + CT_MAX_NODES;
    for (int level = 0; level < p.depth; ++level) {
        const int nodes = 1 << level;
        LayerEntry* part = p.part + (level & 1) * stride;
        layer_block(s, nodes, base + j0, cnt, a, b, key);
        // the nodes this share overlaps leave their best split in entry share + node (no two shares have an entry in common)
        if (tid < nodes && mine > 0 && s.bnd[tid] < base + mine && s.bnd[tid + 1] > base) part[c + tid] = s.top[tid];
        const bool last = level + 1 == p.depth;
        if (!grid_sync(p, round, !last || c == 0)) return;   // (the last layer's boundaries interest one CTA only)
        if (last && c != 0) break;
        // a warp per node (CT_MAX_NODES of them at most): the best of its shares' entries, then the new boundaries
        if (warp < nodes) {
            const int q0 = s.bnd[warp] / p.per, q1 = s.bnd[warp + 1] > s.bnd[warp] ? (s.bnd[warp + 1] - 1) / p.per : q0 - 1;
            unsigned long long l[CG_MAX_CTAS / 32], best = ~0ull;
            int pos[CG_MAX_CTAS / 32], at = 0x7fffffff, e = -1;
#pragma unroll
            for (int q = 0; q < CG_MAX_CTAS / 32; ++q) {
                const LayerEntry* g = &part[min(q0 + q * 32 + lane, G - 1) + warp];
                l[q] = __ldcg(&g->l); pos[q] = __ldcg(&g->pos);
            }
#pragma unroll
            for (int q = 0; q < CG_MAX_CTAS / 32; ++q)
                if (q0 + q * 32 + lane <= q1 && better(l[q], pos[q], best, at)) { best = l[q]; at = pos[q]; e = q0 + q * 32 + lane + warp; }
            const bool found = __any_sync(HS_FULL_MASK, e >= 0);
            if (found ? warp_best(e >= 0, best, at) : lane == 0) {
                const int node = warp;
                float th = CUDART_NAN_F;                      // a single feature value: the node cannot be split
                double sa = s.sy[node + 1], sb = s.syy[node + 1];
                if (!found) { sm.bad = 1; at = s.bnd[node + 1]; }
                else {
                    sa = __ldcg(&part[e].sa); sb = __ldcg(&part[e].sb);
                    th = (float)(0.5 * ((double)__ldcg(&part[e].xp) + (double)__ldcg(&part[e].x)));
                }
                if (c == 0) p.thresholds[threshold_slot(node, level, p.depth)] = th;
                sm.bnd2[2 * node] = s.bnd[node]; sm.sy2[2 * node] = s.sy[node]; sm.syy2[2 * node] = s.syy[node];
                sm.bnd2[2 * node + 1] = at; sm.sy2[2 * node + 1] = sa; sm.syy2[2 * node + 1] = sb;
                if (node == nodes - 1) { sm.bnd2[2 * nodes] = s.bnd[nodes]; sm.sy2[2 * nodes] = s.sy[nodes]; sm.syy2[2 * nodes] = s.syy[nodes]; }
            }
        }
        __syncthreads();
        if (!last && tid <= 2 * nodes) { s.bnd[tid] = sm.bnd2[tid]; s.sy[tid] = sm.sy2[tid]; s.syy[tid] = sm.syy2[tid]; }
        __syncthreads();
    }
    if (tid == 0) {
        if (c == 0) *p.status = sm.bad ? HS_ERR_SHAPE : HS_OK;
        grid_leave(p);
    }
}
