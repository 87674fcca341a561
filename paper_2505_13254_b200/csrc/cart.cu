// hs_cart_fit: training of the entropy stratifier on the device (Sec. 4.2, Eq. 2).
//
// One feature (x = Phi(P*)) and one target (y = Terminal Confidence Rank): the samples are sorted by x once, and then
// every layer of the tree scores all split positions of all its nodes in parallel from running sums of y and y^2 in
// double precision - a node is a contiguous range of the sorted samples, a split at position i costs
//     N L = nL SyyL - SyL^2 + nR SyyR - SyR^2           (Eq. 2 times the node's sample count)
// - and takes, per node, the position with the smallest L (ties: the smallest), between distinct feature values
// only.  The threshold is the midpoint of the two neighbouring feature values.  (The form without divisions orders the
// positions of a node as L does and costs ten fp64 operations instead of sixty.  For integer ranks it is exact while n Syy stays below
// 2^53 - ranks up to 59: 1.6 million samples - and rounded to fp64 like any other above.)
//
// Sort: least-significant-digit radix sort of 64-bit keys (order bits of x : bits of y), four passes over the 8-bit digits
// of x; stable, so equal feature values keep their order and need no more passes.  A bitonic network took 65 launches
// and 0.9 ms on 2^20 samples (every exchange distance beyond shared memory is a pass over all keys); a pass here reads and
// writes the keys once, which stay in L2.
//   up to CT_SMALL samples   cart_small_kernel: one CTA sorts in shared memory and fits all layers - one launch, no round
//                            trips between layers (15 us at 600 samples, 38 us at 8192; the grid kernel 41 at 8193).
//   up to 8192 per SM        cart_grid_kernel (cart_grid.cuh): the same by a resident grid, one launch.
//   more                     cart_pack_kernel (keys, digit counts of all passes), four cart_radix_kernel, cart_sums_kernel
//                            (sums per block and their scan), one cart_level_kernel per layer (what a grid can hold takes it 1.6 times as
//                            long: 125 us at 2^20 samples).
#include <math_constants.h>

#include "hs_common.cuh"
#include "hs_layout.h"
#include "hs_ptx.cuh"

#define CT_THREADS 256
#define CT_ITEMS 16
#define CT_TILE (CT_THREADS * CT_ITEMS)      // keys per CTA: 4096
#define CT_WINDOW 16                         // tiles ahead that are looked at together
#define CT_MAX_DEPTH 6
#define CT_MAX_NODES (1 << (CT_MAX_DEPTH - 1))
#define CT_SMALL_THREADS 1024
#define CT_SMALL_ITEMS 8
#define CT_SMALL (CT_SMALL_THREADS * CT_SMALL_ITEMS)

__device__ __forceinline__ float key_x(unsigned long long k) { return order_bits_float((unsigned int)(k >> 32)); }
__device__ __forceinline__ double key_y(unsigned long long k) { return (double)__uint_as_float((unsigned int)k); }
__device__ __forceinline__ unsigned long long cart_key(float x, float y) {
    return ((unsigned long long)float_order_bits(x) << 32) | __float_as_uint(y);
}
__device__ __forceinline__ unsigned int key_digit(unsigned long long k, int pass) { return (unsigned int)(k >> (32 + 8 * pass)) & 255u; }
// a double as an unsigned integer of the same order
__device__ __forceinline__ unsigned long long order_bits_d(double v) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(v);
    return (u >> 63) ? ~u : (u | (1ull << 63));
}
// The lanes of the warp whose 8-bit digit equals this lane's: eight ballots, or one match for the uppermost digit (its
// cost grows with the number of different values: 12.5 us a pass instead of 17 there, 18.4 on mantissa digits).
__device__ __forceinline__ unsigned int digit_peers(unsigned int d, int pass) {
    if (pass == 3) return __match_any_sync(HS_FULL_MASK, d);
    unsigned int m = HS_FULL_MASK;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const unsigned int v = __ballot_sync(HS_FULL_MASK, (d >> b) & 1u);
        m &= ((d >> b) & 1u) ? v : ~v;
    }
    return m;
}
// Rank of every key of a warp's NITEM x 32 keys (item-major) among the warp's keys of the same digit; cnt: the warp's 256
// digit counters, zero before.
template <int NITEM>
__device__ __forceinline__ void warp_ranks(const unsigned long long (&k)[NITEM], int pass, int* cnt, int lane, int (&rank)[NITEM]) {
#pragma unroll
    for (int i = 0; i < NITEM; ++i) {
        const unsigned int d = key_digit(k[i], pass), peers = digit_peers(d, pass);
        const int before = cnt[d];
        __syncwarp();
        if ((peers >> lane) == 1u) cnt[d] = before + __popc(peers);        // (the highest lane of the group)
        rank[i] = before + __popc(peers & ((1u << lane) - 1u));
        __syncwarp();
    }
}
// exclusive prefix over 256 values, one per thread 0..255 (all threads of the CTA call it)
__device__ __forceinline__ int scan256(int v, int* s_warp, int tid) {
    const int lane = tid & 31, warp = tid >> 5;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int u = __shfl_up_sync(HS_FULL_MASK, incl, o); if (lane >= o) incl += u; }
    if (lane == 31 && warp < 8) s_warp[warp] = incl;
    __syncthreads();
    int before = incl - v;
    for (int w = 0; w < 8; ++w) if (w < warp) before += s_warp[w];
    return before;
}

// ---- one layer: all split positions of a block of sorted keys -----------------------------------------------------
struct LayerEntry {                                  // a split of a node
    unsigned long long l;                            // N L as order bits, ~0: none
    double sa, sb;                                   // running sums of y and y^2 at its position
    float xp, x;                                     // the feature values on both sides
    int pos;                                         // 0x7fffffff: none
    int node;
};
__device__ __forceinline__ bool better(unsigned long long l, int pos, unsigned long long l2, int pos2) { return l < l2 || (l == l2 && pos < pos2); }

#define CT_ENTRIES 96           // of a block: one per warp and one per boundary in it, and one per boundary inside a thread's run
struct LayerSmem {
    int bnd[CT_MAX_NODES + 1];                       // node boundaries (positions in the sorted order)
    double sy[CT_MAX_NODES + 1], syy[CT_MAX_NODES + 1];   // running sums at the boundaries
    LayerEntry top[CT_MAX_NODES];                    // the block's best split of every node
    LayerEntry ent[CT_ENTRIES];
    int nent;
};
static_assert(CT_SMALL_THREADS / 32 + 2 * (CT_MAX_NODES - 1) <= CT_ENTRIES, "entries of a block");

// The lane of the warp with the best (l, pos) among those that are `in`: true there, false elsewhere (and everywhere if none is in).
__device__ __forceinline__ bool warp_best(bool in, unsigned long long l, int pos) {
    const unsigned int hi = __reduce_min_sync(HS_FULL_MASK, in ? (unsigned int)(l >> 32) : ~0u);
    in = in && (unsigned int)(l >> 32) == hi;
    const unsigned int lo = __reduce_min_sync(HS_FULL_MASK, in ? (unsigned int)l : ~0u);
    in = in && (unsigned int)l == lo;
    const unsigned int at = __reduce_min_sync(HS_FULL_MASK, in ? (unsigned int)pos : ~0u);
    return in && (unsigned int)pos == at;
}

// The block's best split of every node -> s.top (smallest N L, then smallest position).  A thread has `cnt` consecutive keys, key(j) =
// sorted key at position i0 + j (j = -1: the one ahead of it); (a, b): running sums of y and y^2 ahead of them.  One sweep: the thread keeps
// its best split with the sums and the feature values there (three sweeps, for N L, its position and the sums, took 2.5 times as long).
// (The right side's sums are the node's less the left's.  Against rational arithmetic, of 7500 nodes of near-equal targets that are no whole
// numbers 9 or 13 take another split, by which product is fused; 14 or 18 with the right side taken from its end, 24 so without fused products.)
template <class KeyFn>
__device__ __forceinline__ void layer_block(LayerSmem& s, int nodes, int i0, int cnt, double a, double b, KeyFn key) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) s.nent = 0;
    __syncthreads();
    LayerEntry t;
    t.l = ~0ull; t.pos = 0x7fffffff; t.node = -1; t.sa = t.sb = 0.0; t.xp = t.x = 0.f;
    double best = 0.0;
    auto push = [&]() { t.l = order_bits_d(best); s.ent[atomicAdd(&s.nent, 1)] = t; };
    if (cnt > 0) {
        int node = 0, lo, hi;
        while (node + 1 < nodes && s.bnd[node + 1] <= i0) ++node;
        double sy, syy, ty, tyy, nl, n;                               // sums ahead of the node, its sums, keys of it ahead of i, all its keys
        auto enter = [&]() {
            lo = s.bnd[node]; hi = s.bnd[node + 1];
            sy = s.sy[node]; syy = s.syy[node];
            ty = s.sy[node + 1] - sy; tyy = s.syy[node + 1] - syy;
            n = (double)(hi - lo);
        };
        enter();
        nl = (double)(i0 - lo);
        float xp = i0 > 0 ? key_x(key(-1)) : 0.f;
        for (int j = 0; j < cnt; ++j) {
            const int i = i0 + j;
            if (i >= hi) {
                while (node + 1 < nodes && s.bnd[node + 1] <= i) ++node;
                enter();
                nl = (double)(i - lo);
            }
            const unsigned long long k = key(j);
            const float x = key_x(k);
            if (i > lo && xp < x) {                                   // a threshold lies between distinct values
                const double yl = a - sy, yyl = b - syy, yr = ty - yl, yyr = tyy - yyl;
                if (node != t.node) {
                    if (t.node >= 0) push();                          // (the run lies in more than one node)
                    t.node = node; t.pos = 0x7fffffff;
                }
                const double l = (nl * yyl - yl * yl) + ((n - nl) * yyr - yr * yr);
                if (t.pos == 0x7fffffff || l < best) { best = l; t.pos = i; t.sa = a; t.sb = b; t.xp = xp; t.x = x; }
            }
            const double y = key_y(k);
            a += y; b += y * y;
            nl += 1.0;
            xp = x;
        }
    }
    // the lanes' last nodes: mostly one, else one round each
    t.l = order_bits_d(best);
    for (unsigned int rem = __ballot_sync(HS_FULL_MASK, t.node >= 0); rem;) {
        const int c = __shfl_sync(HS_FULL_MASK, t.node, __ffs(rem) - 1);
        const bool in = t.node == c;
        if (warp_best(in, t.l, t.pos)) push();
        rem &= ~__ballot_sync(HS_FULL_MASK, in);
    }
    __syncthreads();
    const int nent = s.nent;
    for (int q = warp; q < nodes; q += blockDim.x / 32) {
        unsigned long long l = ~0ull;
        int pos = 0x7fffffff, e = -1;
        for (int i = lane; i < nent; i += 32)
            if (s.ent[i].node == q && better(s.ent[i].l, s.ent[i].pos, l, pos)) { l = s.ent[i].l; pos = s.ent[i].pos; e = i; }
        if (warp_best(e >= 0, l, pos)) s.top[q] = s.ent[e];
        if (!__any_sync(HS_FULL_MASK, e >= 0) && lane == 0) { s.top[q].l = ~0ull; s.top[q].pos = 0x7fffffff; }
    }
    __syncthreads();
}

// exclusive prefix over the CTA of two doubles per thread (fixed order: lanes, then warps)
template <int NW>
__device__ __forceinline__ void scan_pair(double& a, double& b, double (*s_w)[2]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double ia = a, ib = b;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double ua = __shfl_up_sync(HS_FULL_MASK, ia, o), ub = __shfl_up_sync(HS_FULL_MASK, ib, o);
        if (lane >= o) { ia += ua; ib += ub; }
    }
    if (lane == 31) { s_w[warp][0] = ia; s_w[warp][1] = ib; }
    __syncthreads();
    if (warp == 0) {                                 // (one warp: the sums ahead of every warp)
        double wa = lane < NW ? s_w[lane][0] : 0.0, wb = lane < NW ? s_w[lane][1] : 0.0;
        const double va = wa, vb = wb;
#pragma unroll
        for (int o = 1; o < NW; o <<= 1) {
            const double ua = __shfl_up_sync(HS_FULL_MASK, wa, o), ub = __shfl_up_sync(HS_FULL_MASK, wb, o);
            if (lane >= o) { wa += ua; wb += ub; }
        }
        if (lane < NW) { s_w[lane][0] = wa - va; s_w[lane][1] = wb - vb; }
    }
    __syncthreads();
    a = s_w[warp][0] + (ia - a);
    b = s_w[warp][1] + (ib - b);
}

// position of a node's threshold in the ascending list: in-order index of the node
__device__ __forceinline__ int threshold_slot(int node, int level, int depth) { return (2 * node + 1) * (1 << (depth - 1 - level)) - 1; }

// ---- few samples: one CTA ------------------------------------------------------------------------------------------
// padded index of a key: runs of eight consecutive keys of different threads start in different banks
__device__ __forceinline__ int pad8(int i) { return i + (i >> 3); }
struct SmallSmem {
    unsigned long long key[CT_SMALL * 9 / 8 + 8];
    int cnt[CT_SMALL_THREADS / 32][256];
};

__global__ void __launch_bounds__(CT_SMALL_THREADS, 1) cart_small_kernel(const float* x, const float* y, int n, int depth,
                                                                         float* thresholds, int* status) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    constexpr int NW = CT_SMALL_THREADS / 32;
    unsigned long long* s_key = reinterpret_cast<SmallSmem*>(s_dyn)->key;
    int(*s_cnt)[256] = reinterpret_cast<SmallSmem*>(s_dyn)->cnt;
    __shared__ LayerSmem s;
    __shared__ double s_w[NW][2];
    __shared__ int s_scan[8];
    __shared__ int s_bnd2[2 * CT_MAX_NODES + 1];
    __shared__ double s_sy2[2 * CT_MAX_NODES + 1], s_syy2[2 * CT_MAX_NODES + 1];
    __shared__ int s_bad;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    pdl_launch_dependents();
    pdl_wait();
    // warp w holds keys 32 nit w .. of the input order, item-major; rounds past the samples are left out
    const int nit = (n + CT_SMALL_THREADS - 1) / CT_SMALL_THREADS;
    unsigned long long k[CT_SMALL_ITEMS];
    int rank[CT_SMALL_ITEMS];
#pragma unroll
    for (int i = 0; i < CT_SMALL_ITEMS; ++i) {
        const int j = warp * 32 * nit + i * 32 + lane;
        k[i] = (i < nit && j < n) ? cart_key(x[j], y[j]) : ~0ull;      // (padding sorts to the end)
    }
    for (int pass = 0; pass < 4; ++pass) {
        for (int i = lane; i < 256; i += 32) s_cnt[warp][i] = 0;
        __syncwarp();
#pragma unroll
        for (int i = 0; i < CT_SMALL_ITEMS; ++i) {
            if (i >= nit) break;
            unsigned long long k1[1] = {k[i]};
            int r1[1];
            warp_ranks<1>(k1, pass, s_cnt[warp], lane, r1);
            rank[i] = r1[0];
        }
        __syncthreads();
        int tot = 0;
        if (tid < 256)
            for (int w = 0; w < NW; ++w) { const int c = s_cnt[w][tid]; s_cnt[w][tid] = tot; tot += c; }
        const int first = scan256(tid < 256 ? tot : 0, s_scan, tid);
        if (tid < 256)
            for (int w = 0; w < NW; ++w) s_cnt[w][tid] += first;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < CT_SMALL_ITEMS; ++i)
            if (i < nit) s_key[pad8(s_cnt[warp][key_digit(k[i], pass)] + rank[i])] = k[i];
        __syncthreads();
        if (pass < 3) {
#pragma unroll
            for (int i = 0; i < CT_SMALL_ITEMS; ++i)
                if (i < nit) k[i] = s_key[pad8(warp * 32 * nit + i * 32 + lane)];
        }
    }
    // running sums: thread t has keys nit t .. nit t + nit - 1 of the sorted order
    const int i0 = min(tid * nit, n), cnt = min(i0 + nit, n) - i0;
    auto key = [&](int j) { return s_key[pad8(i0 + j)]; };
    double a = 0.0, b = 0.0;
    for (int j = 0; j < cnt; ++j) { const double v = key_y(key(j)); a += v; b += v * v; }
    double ta = a, tb = b;
    scan_pair<NW>(a, b, s_w);
    if (tid == CT_SMALL_THREADS - 1) { s.sy[1] = a + ta; s.syy[1] = b + tb; }
    if (tid == 0) { s.bnd[0] = 0; s.bnd[1] = n; s.sy[0] = 0.0; s.syy[0] = 0.0; s_bad = 0; }
    __syncthreads();
    for (int level = 0; level < depth; ++level) {
        const int nodes = 1 << level;
        layer_block(s, nodes, i0, cnt, a, b, key);
        if (tid < nodes) {
            const LayerEntry& t = s.top[tid];
            int at = t.pos;
            float th = CUDART_NAN_F;                  // a single feature value: the node cannot be split
            double sa = s.sy[tid + 1], sb = s.syy[tid + 1];
            if (at == 0x7fffffff) { s_bad = 1; at = s.bnd[tid + 1]; }
            else { th = (float)(0.5 * ((double)t.xp + (double)t.x)); sa = t.sa; sb = t.sb; }
            thresholds[threshold_slot(tid, level, depth)] = th;
            s_bnd2[2 * tid] = s.bnd[tid]; s_sy2[2 * tid] = s.sy[tid]; s_syy2[2 * tid] = s.syy[tid];
            s_bnd2[2 * tid + 1] = at; s_sy2[2 * tid + 1] = sa; s_syy2[2 * tid + 1] = sb;
            if (tid == nodes - 1) { s_bnd2[2 * nodes] = s.bnd[nodes]; s_sy2[2 * nodes] = s.sy[nodes]; s_syy2[2 * nodes] = s.syy[nodes]; }
        }
        __syncthreads();
        if (level + 1 < depth && tid <= 2 * nodes) { s.bnd[tid] = s_bnd2[tid]; s.sy[tid] = s_sy2[tid]; s.syy[tid] = s_syy2[tid]; }
        __syncthreads();
    }
    if (tid == 0) *status = s_bad ? HS_ERR_SHAPE : HS_OK;
}

// ---- up to eight samples per thread of a resident grid: one launch ------------------------------------------------------
#include "cart_grid.cuh"

// ---- more samples ----------------------------------------------------------------------------------------------------
struct CartParams {
    const float* x;
    const float* y;
    int n, tiles, depth;
    unsigned long long* keys;      // sorted in place over an even number of passes ...
    unsigned long long* keys2;     // ... through this copy
    unsigned int* look;            // [4][tiles][256] look-back words of the radix passes
    double* blk;                   // [tiles][2] sums of y and y^2 per tile, then ahead of it
    int* hist;                     // [4][256] digit counts (zero between calls)
    int* ticket;                   // [4] tiles started per pass (zero between calls)
    int* done;                     // [1 + depth] CTAs that have finished (zero between calls)
    int* bnd;                      // [2][CT_MAX_NODES + 1]: boundaries of the layer, and of the next
    double* bsum;                  // [2][CT_MAX_NODES + 1][2]
    unsigned long long* part_l;    // [tiles + nodes] best N L of a (tile, node), entry tile + node
    int* part_i;
    double* part_s;                // [tiles + nodes][2]
    float* thresholds;
    int* status;
    int* err;
};

__global__ void __launch_bounds__(CT_THREADS) cart_pack_kernel(const CartParams p) {
    __shared__ int s_h[4][256];
    const int tid = threadIdx.x;
    for (int q = 0; q < 4; ++q) s_h[q][tid] = 0;
    pdl_launch_dependents();
    pdl_wait();
    __syncthreads();
    for (int q = 0; q < 4; ++q) p.look[((size_t)q * p.tiles + blockIdx.x) * 256 + tid] = 0u;
    const int base = blockIdx.x * CT_TILE;
    float xv[CT_ITEMS], yv[CT_ITEMS];
#pragma unroll
    for (int i = 0; i < CT_ITEMS; ++i) {
        const int j = base + i * CT_THREADS + tid;
        xv[i] = j < p.n ? p.x[j] : 0.f;
        yv[i] = j < p.n ? p.y[j] : 0.f;
    }
#pragma unroll
    for (int i = 0; i < CT_ITEMS; ++i) {
        const int j = base + i * CT_THREADS + tid;
        const unsigned long long k = cart_key(xv[i], yv[i]);
        if (j < p.n) p.keys[j] = k;
        const unsigned int in = __ballot_sync(HS_FULL_MASK, j < p.n);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            // the uppermost digit (sign and exponent) takes few values: one atomic per group of equal digits there
            const unsigned int d = key_digit(k, q);
            if (q < 3) { if (j < p.n) atomicAdd(&s_h[q][d], 1); }
            else {
                const unsigned int m = __match_any_sync(HS_FULL_MASK, d) & in;
                if (j < p.n && __ffs(m) - 1 == (tid & 31)) atomicAdd(&s_h[q][d], __popc(m));
            }
        }
    }
    __syncthreads();
    for (int q = 0; q < 4; ++q) if (s_h[q][tid]) atomicAdd(&p.hist[q * 256 + tid], s_h[q][tid]);
}

// One pass of the radix sort.  A CTA takes tiles in the order CTAs start (a ticket), ranks its keys, publishes its digit
// counts and looks back over the tiles ahead for the counts before its own (a tile it waits for has started, so every
// wait ends; bounded all the same), reorders the tile in shared memory and writes runs of equal digits.
__global__ void __launch_bounds__(CT_THREADS) cart_radix_kernel(const CartParams p, int pass) {
    __shared__ unsigned long long s_key[CT_TILE];
    __shared__ int s_cnt[8][256];
    __shared__ int s_off[256];
    __shared__ int s_scan[8];
    __shared__ int s_tile;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned long long* in = (pass & 1) ? p.keys2 : p.keys;
    unsigned long long* out = (pass & 1) ? p.keys : p.keys2;
    for (int w = 0; w < 8; ++w) s_cnt[w][tid] = 0;
    pdl_launch_dependents();
    pdl_wait();
    if (tid == 0) s_tile = atomicAdd(&p.ticket[pass], 1);
    __syncthreads();
    const int tile = s_tile, base = tile * CT_TILE;
    const int nvalid = min(CT_TILE, p.n - base);
    unsigned long long k[CT_ITEMS];
    int rank[CT_ITEMS];
#pragma unroll
    for (int i = 0; i < CT_ITEMS; ++i) {
        const int j = warp * 32 * CT_ITEMS + i * 32 + lane;
        k[i] = j < nvalid ? in[base + j] : ~0ull;              // (past the last sample: behind everything in the last tile)
    }
    const int first = scan256(p.hist[pass * 256 + tid], s_scan, tid);      // keys with smaller digits
    warp_ranks<CT_ITEMS>(k, pass, s_cnt[warp], lane, rank);
    __syncthreads();
    int c = 0;
    for (int w = 0; w < 8; ++w) { const int v = s_cnt[w][tid]; s_cnt[w][tid] = c; c += v; }
    unsigned int* look = p.look + (size_t)pass * p.tiles * 256 + tid;
    volatile unsigned int* vlook = look;
    vlook[(size_t)tile * 256] = (tile == 0 ? 2u << 30 : 1u << 30) | (unsigned int)c;
    const int local = scan256(c, s_scan, tid);                 // (its barrier also orders s_scan's reuse)
    int before = 0;
    const unsigned long long t0 = global_timer_ns();
    // (CT_WINDOW tiles at a time: the tiles of a launch publish together, and a walk of one load per tile would be a chain of
    // as many round trips to L2 as there are tiles)
    bool found = tile == 0;
    for (int t = tile - 1; !found;) {
        unsigned int v[CT_WINDOW];
#pragma unroll
        for (int i = 0; i < CT_WINDOW; ++i) v[i] = t - i >= 0 ? vlook[(size_t)(t - i) * 256] : 2u << 30;
        bool open = true;                                      // nothing unpublished met in this window so far
#pragma unroll
        for (int i = 0; i < CT_WINDOW; ++i) {
            open = open && v[i] >> 30;
            if (open && !found) {
                before += (int)(v[i] & 0x3fffffffu);
                found = v[i] >> 31;                            // that tile knew everything ahead of it
                --t;
            }
        }
        if (!open && global_timer_ns() - t0 > HS_WAIT_LIMIT_NS) {
            atomicExch(p.err, (int)HS_ERR_TIMEOUT);
            break;
        }
    }
    if (tile > 0) vlook[(size_t)tile * 256] = (2u << 30) | (unsigned int)(before + c);
    s_off[tid] = first + before - local;
    for (int w = 0; w < 8; ++w) s_cnt[w][tid] += local;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < CT_ITEMS; ++i) s_key[s_cnt[warp][key_digit(k[i], pass)] + rank[i]] = k[i];
    __syncthreads();
#pragma unroll 4
    for (int j = tid; j < nvalid; j += CT_THREADS) {
        const unsigned long long kk = s_key[j];
        const int at = s_off[key_digit(kk, pass)] + j;
        if ((unsigned int)at < (unsigned int)p.n) out[at] = kk;    // (out of range only after a wait that expired)
    }
}

// Layer kernel: eight keys per thread (a thread's running sums are a chain of fp64 additions: with sixteen keys the chain,
// not the fp64 pipe, was the time of a launch).
#define CT_LV_THREADS 512
#define CT_LV_ITEMS (CT_TILE / CT_LV_THREADS)
#define CT_PADDED (CT_TILE + CT_TILE / 8 + 1)

// last CTA of the launch to arrive (every thread gets the answer; its earlier stores are ordered ahead)
__device__ __forceinline__ bool last_cta(int* done, int* s_last) {
    __syncthreads();
    if (threadIdx.x == 0) {
        int old;
        asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(old) : "l"(done) : "memory");
        *s_last = old == (int)gridDim.x - 1;
        if (*s_last) *done = 0;
    }
    __syncthreads();
    return *s_last != 0;
}

// sums of y and y^2 per tile; the last CTA turns them into the sums ahead of each tile
__global__ void __launch_bounds__(CT_THREADS) cart_sums_kernel(const CartParams p) {
    __shared__ double s_w[8][2];
    __shared__ int s_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    pdl_launch_dependents();
    pdl_wait();
    double a = 0.0, b = 0.0;
#pragma unroll
    for (int i = 0; i < CT_ITEMS; ++i) {
        const int j = blockIdx.x * CT_TILE + i * CT_THREADS + tid;
        if (j < p.n) { const double v = key_y(p.keys[j]); a += v; b += v * v; }
    }
    a = warp_sum_d(a); b = warp_sum_d(b);
    if (lane == 0) { s_w[warp][0] = a; s_w[warp][1] = b; }
    __syncthreads();
    if (tid == 0) {
        double ta = 0.0, tb = 0.0;
        for (int w = 0; w < 8; ++w) { ta += s_w[w][0]; tb += s_w[w][1]; }
        p.blk[2 * blockIdx.x] = ta; p.blk[2 * blockIdx.x + 1] = tb;
    }
    if (!last_cta(&p.done[0], &s_last)) return;
    const int per = (p.tiles + CT_THREADS - 1) / CT_THREADS;
    const int t0 = min(tid * per, p.tiles), t1 = min(t0 + per, p.tiles);
    a = 0.0; b = 0.0;
    for (int t = t0; t < t1; ++t) { a += __ldcg(&p.blk[2 * t]); b += __ldcg(&p.blk[2 * t + 1]); }
    const double ma = a, mb = b;
    scan_pair<8>(a, b, s_w);
    double ra = a, rb = b;
    for (int t = t0; t < t1; ++t) {
        const double va = __ldcg(&p.blk[2 * t]), vb = __ldcg(&p.blk[2 * t + 1]);
        p.blk[2 * t] = ra; p.blk[2 * t + 1] = rb;
        ra += va; rb += vb;
    }
    if (tid == CT_THREADS - 1) { p.bsum[2] = a + ma; p.bsum[3] = b + mb; }
    if (tid == 0) { p.bnd[0] = 0; p.bnd[1] = p.n; p.bsum[0] = 0.0; p.bsum[1] = 0.0; *p.status = HS_OK; }
    for (int q = tid; q < 4 * 256; q += CT_THREADS) p.hist[q] = 0;         // ready for the next call
    if (tid < 4) p.ticket[tid] = 0;
}

__global__ void __launch_bounds__(CT_LV_THREADS) cart_level_kernel(const CartParams p, int level) {
    __shared__ unsigned long long s_key[CT_PADDED];
    __shared__ LayerSmem s;
    __shared__ double s_w[CT_LV_THREADS / 32][2];
    __shared__ int s_last;
    __shared__ unsigned long long s_best[32];
    __shared__ int s_at[32], s_e[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nodes = 1 << level;
    pdl_launch_dependents();
    pdl_wait();
    const int* bnd = p.bnd + (level & 1) * (CT_MAX_NODES + 1);
    const double* bsum = p.bsum + (level & 1) * 2 * (CT_MAX_NODES + 1);
    if (tid <= nodes) { s.bnd[tid] = bnd[tid]; s.sy[tid] = bsum[2 * tid]; s.syy[tid] = bsum[2 * tid + 1]; }
    const int base = blockIdx.x * CT_TILE, nvalid = min(CT_TILE, p.n - base);
#pragma unroll
    for (int i = 0; i < CT_LV_ITEMS; ++i) {
        const int j = i * CT_LV_THREADS + tid;
        if (j < nvalid) s_key[1 + pad8(j)] = p.keys[base + j];
    }
    if (tid == 0) s_key[0] = base > 0 ? p.keys[base - 1] : 0ull;           // the key ahead of the tile
    __syncthreads();
    const int j0 = min(tid * CT_LV_ITEMS, nvalid), cnt = min(j0 + CT_LV_ITEMS, nvalid) - j0;
    auto key = [&](int j) { return j0 + j < 0 ? s_key[0] : s_key[1 + pad8(j0 + j)]; };
    double a = 0.0, b = 0.0;
    for (int j = 0; j < cnt; ++j) { const double v = key_y(key(j)); a += v; b += v * v; }
    scan_pair<CT_LV_THREADS / 32>(a, b, s_w);
    a += p.blk[2 * blockIdx.x]; b += p.blk[2 * blockIdx.x + 1];
    layer_block(s, nodes, base + j0, cnt, a, b, key);
    // the nodes this tile overlaps leave their best split in entry tile + node (no two tiles share an entry)
    if (tid < nodes && s.bnd[tid] < base + nvalid && s.bnd[tid + 1] > base) {
        const int e = blockIdx.x + tid;
        p.part_l[e] = s.top[tid].l; p.part_i[e] = s.top[tid].pos;
        p.part_s[2 * e] = s.top[tid].sa; p.part_s[2 * e + 1] = s.top[tid].sb;
    }
    if (!last_cta(&p.done[1 + level], &s_last)) return;
    // the best of a node's tiles: a power of two of warps per node, one tile per lane as long as they reach
    int* bnd2 = p.bnd + ((level + 1) & 1) * (CT_MAX_NODES + 1);
    double* bsum2 = p.bsum + ((level + 1) & 1) * 2 * (CT_MAX_NODES + 1);
    constexpr int NWL = CT_LV_THREADS / 32;
    const int wpn = max(NWL / nodes, 1);
    for (int v = warp; v < max(nodes, NWL); v += NWL) {
        const int node = v / wpn, lo = s.bnd[node], hi = s.bnd[node + 1];
        unsigned long long m = ~0ull;
        int at = 0x7fffffff, e = -1;
        if (hi > lo)
            for (int t = lo / CT_TILE + (v % wpn) * 32 + lane; t <= (hi - 1) / CT_TILE; t += 32 * wpn) {
                const unsigned long long l = __ldcg(&p.part_l[t + node]);
                const int i = __ldcg(&p.part_i[t + node]);
                if (l < m || (l == m && i < at)) { m = l; at = i; e = t + node; }
            }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long l = __shfl_xor_sync(HS_FULL_MASK, m, o);
            const int i = __shfl_xor_sync(HS_FULL_MASK, at, o), e2 = __shfl_xor_sync(HS_FULL_MASK, e, o);
            if (l < m || (l == m && i < at)) { m = l; at = i; e = e2; }
        }
        if (lane == 0) { s_best[v] = m; s_at[v] = at; s_e[v] = e; }
    }
    __syncthreads();
    if (tid < nodes) {
        const int node = tid, lo = s.bnd[node], hi = s.bnd[node + 1];
        unsigned long long m = ~0ull;
        int at = 0x7fffffff, e = -1;
        for (int w = node * wpn; w < (node + 1) * wpn; ++w)
            if (s_best[w] < m || (s_best[w] == m && s_at[w] < at)) { m = s_best[w]; at = s_at[w]; e = s_e[w]; }
        float th = CUDART_NAN_F;                              // a single feature value: the node cannot be split
        double sa = s.sy[node + 1], sb = s.syy[node + 1];
        if (at == 0x7fffffff) { *p.status = HS_ERR_SHAPE; at = hi; }
        else {
            th = (float)(0.5 * ((double)key_x(p.keys[at - 1]) + (double)key_x(p.keys[at])));
            sa = __ldcg(&p.part_s[2 * e]); sb = __ldcg(&p.part_s[2 * e + 1]);
        }
        p.thresholds[threshold_slot(node, level, p.depth)] = th;
        if (level + 1 < p.depth) {
            bnd2[2 * node] = lo; bsum2[4 * node] = s.sy[node]; bsum2[4 * node + 1] = s.syy[node];
            bnd2[2 * node + 1] = at; bsum2[4 * node + 2] = sa; bsum2[4 * node + 3] = sb;
            if (node == nodes - 1) { bnd2[2 * nodes] = hi; bsum2[4 * nodes] = s.sy[nodes]; bsum2[4 * nodes + 1] = s.syy[nodes]; }
        }
    }
}

// What the calls asked for before the radix sort (keys padded to a power of two, two running sums per sample): the same
// bytes hold the second copy of the keys, the look-back words and the per-tile arrays.
static int next_pow2(int n) { int p = 1024; while (p < n) p <<= 1; return p; }

extern "C" size_t hs_cart_workspace_bytes(int32_t n) {
    if (n < 2) return 0;
    const size_t P = next_pow2(n);
    return HS_COUNTER_BYTES + P * 8 + 2 * ((size_t)n + 1) * 8 + 2 * (((size_t)n + CT_THREADS - 1) / CT_THREADS) * 8 +
           2 * (2 << CT_MAX_DEPTH) * 4 + (1 << CT_MAX_DEPTH) * 64 * 12 + 4096;
}

// SMs that a launch into the stream may use: the device's, or those of the partition that the stream belongs to.  (A capture takes a
// cooperative launch that is too large for the partition without a word, and the graph as well.)
static int stream_sms(const hs_ctx* ctx, cudaStream_t stream) {
    if ((uintptr_t)stream <= 2 || !ctx->stream_part || !ctx->part_sms) return ctx->sm_count;      // (the default streams belong to none)
    CUgreenCtx part = nullptr;
    CUdevResource r;
    if (((CUresult(*)(CUstream, CUgreenCtx*))ctx->stream_part)((CUstream)stream, &part) != CUDA_SUCCESS || !part) return ctx->sm_count;
    if (((CUresult(*)(CUgreenCtx, CUdevResource*, CUdevResourceType))ctx->part_sms)(part, &r, CU_DEV_RESOURCE_TYPE_SM) != CUDA_SUCCESS) return ctx->sm_count;
    return min((int)r.sm.smCount, ctx->sm_count);
}

// (too_large: fewer SMs than CTAs, whatever took them; nothing was launched)
static hs_status launch_grid(hs_ctx* ctx, const float* x, const float* y, int n, int depth, float* thresholds, int* status, cudaStream_t stream, bool& too_large) {
    CartGrid p;
    p.x = x; p.y = y; p.n = n; p.depth = depth; p.thresholds = thresholds; p.status = status;
    p.per = max(CG_THREADS, (n + ctx->cart_ctas - 1) / ctx->cart_ctas);
    const int G = (n + p.per - 1) / p.per, parts = 2 * (G + CT_MAX_NODES);
    too_large = G > stream_sms(ctx, stream);
    if (too_large) return HS_OK;
    size_t o = 0;
    auto take = [&](size_t bytes) { char* q = ctx->scratch + o; o += hs_align_up(bytes, 256); return q; };
    p.keys = (unsigned long long*)take((size_t)n * 8);
    p.keys2 = (unsigned long long*)take((size_t)n * 8);
    p.cnt = (unsigned int*)take((size_t)CG_MAX_DIGITS * G * 4);
    p.tot = (unsigned int*)take(CG_MAX_DIGITS * 4);
    p.range = (uint2*)take((size_t)G * 8);
    p.blk = (double*)take((size_t)G * 16);
    p.part = (LayerEntry*)take((size_t)parts * sizeof(LayerEntry));
    if (o > ctx->scratch_bytes) return HS_ERR_WORKSPACE;
    p.bar = (unsigned int*)(ctx->counters + HS_CNT_CART);
    p.err = ctx->counters + HS_CNT_ERROR;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(G);
    cfg.blockDim = dim3(CG_THREADS);
    cfg.dynamicSmemBytes = sizeof(CartGridSmem);
    cfg.stream = stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;       // (its CTAs wait for one another)
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, cart_grid_kernel, p);
    too_large = e == cudaErrorCooperativeLaunchTooLarge;
    if (too_large) (void)cudaGetLastError();
    return e == cudaSuccess ? HS_OK : HS_ERR_CUDA;
}

extern "C" hs_status hs_cart_fit(hs_ctx* ctx, const float* x, const float* y, int32_t n, int32_t depth,
                                 float* thresholds, int32_t* status, hs_stream stream_) {
    cudaStream_t stream = (cudaStream_t)stream_;
    if (!ctx || !hs_on_device(ctx) || !x || !y || !thresholds || !status) return HS_ERR_INVALID_ARG;
    if (depth < 1 || depth > CT_MAX_DEPTH || n < (1 << depth) || n > (1 << 26)) return HS_ERR_SHAPE;
    if (hs_cart_workspace_bytes(n) - HS_COUNTER_BYTES - 4096 > ctx->scratch_bytes) return HS_ERR_WORKSPACE;
    const dim3 one(1, 1, 1);
    if (n <= CT_SMALL) {
        if (!ctx->cart_ready) {
            HS_CUDA_OK(cudaFuncSetAttribute(cart_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SmallSmem)));
            ctx->cart_ready = true;
        }
        return hs_launch(cart_small_kernel, one, dim3(CT_SMALL_THREADS), sizeof(SmallSmem), stream, ctx->pdl, one, x, y, (int)n,
                         (int)depth, thresholds, (int*)status) == cudaSuccess ? HS_OK : HS_ERR_CUDA;
    }
    if (!ctx->cart_ctas) {                           // CTAs of the grid kernel that run at once on this device
        int per_sm = 0;
        HS_CUDA_OK(cudaFuncSetAttribute(cart_grid_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(CartGridSmem)));
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, cart_grid_kernel, CG_THREADS, sizeof(CartGridSmem)) != cudaSuccess) {
            per_sm = 0;
            (void)cudaGetLastError();
        }
        cudaDriverEntryPointQueryResult found;
        if (cudaGetDriverEntryPoint("cuStreamGetGreenCtx", &ctx->stream_part, cudaEnableDefault, &found) != cudaSuccess || found != cudaDriverEntryPointSuccess)
            ctx->stream_part = nullptr;
        if (cudaGetDriverEntryPoint("cuGreenCtxGetDevResource", &ctx->part_sms, cudaEnableDefault, &found) != cudaSuccess || found != cudaDriverEntryPointSuccess)
            ctx->part_sms = nullptr;
        ctx->cart_ctas = per_sm > 0 ? min(ctx->sm_count, CG_MAX_CTAS) : -1;
    }
    if (ctx->cart_ctas > 0 && n <= ctx->cart_ctas * CG_SHARE) {
        bool too_large = false;
        const hs_status st = launch_grid(ctx, x, y, n, depth, thresholds, (int*)status, stream, too_large);
        if (!too_large) return st;
    }
    CartParams p;
    p.x = x; p.y = y; p.n = n; p.depth = depth; p.thresholds = thresholds; p.status = status;
    p.tiles = (n + CT_TILE - 1) / CT_TILE;
    size_t o = 0;
    auto take = [&](size_t bytes) { char* q = ctx->scratch + o; o += hs_align_up(bytes, 256); return q; };
    p.keys = (unsigned long long*)take((size_t)n * 8);
    p.keys2 = (unsigned long long*)take((size_t)n * 8);
    p.look = (unsigned int*)take((size_t)4 * p.tiles * 256 * 4);
    p.blk = (double*)take((size_t)p.tiles * 16);
    p.bnd = (int*)take(2 * (CT_MAX_NODES + 1) * 4);
    p.bsum = (double*)take(2 * (CT_MAX_NODES + 1) * 16);
    const size_t parts = (size_t)p.tiles + CT_MAX_NODES;
    p.part_l = (unsigned long long*)take(parts * 8);
    p.part_i = (int*)take(parts * 4);
    p.part_s = (double*)take(parts * 16);
    if (o > ctx->scratch_bytes) return HS_ERR_WORKSPACE;
    p.hist = ctx->counters + HS_CNT_CART;
    p.ticket = p.hist + 4 * 256;
    p.done = p.ticket + 4;
    p.err = ctx->counters + HS_CNT_ERROR;
    const dim3 grid(p.tiles), block(CT_THREADS);
    if (hs_launch(cart_pack_kernel, grid, block, 0, stream, ctx->pdl, one, p) != cudaSuccess) return HS_ERR_CUDA;
    for (int pass = 0; pass < 4; ++pass)
        if (hs_launch(cart_radix_kernel, grid, block, 0, stream, ctx->pdl, one, p, pass) != cudaSuccess) return HS_ERR_CUDA;
    if (hs_launch(cart_sums_kernel, grid, block, 0, stream, ctx->pdl, one, p) != cudaSuccess) return HS_ERR_CUDA;
    for (int level = 0; level < depth; ++level)
        if (hs_launch(cart_level_kernel, grid, dim3(CT_LV_THREADS), 0, stream, ctx->pdl, one, p, level) != cudaSuccess) return HS_ERR_CUDA;
    return HS_OK;
}
