// Which attention kernel takes a launch, and in how many splits of the prefix.  On its own so that the host can check which one a launch runs.
#pragma once

#define ATT_MAX_SPLIT 8

// KV splits (= cluster size) of tree_attn_umma_kernel: the number with the least time on the critical path, waves of CTAs (as many
// clusters of that size as the device runs at once) times {tiles per CTA, what lies around them, merge}, in half tiles.  A tile is
// 0.55 us; start, tree tiles and output 6.5 us, the merge of splits 2.5 us.  (The start was counted as the tree's two tiles, as if
// a further wave cost nothing else.)  us a call, splits then : now, equal lengths | lengths spread over 0.2 .. 1 of the longest:
//   one tree, 32 / 8 heads, 256 tokens 8.7 : 7.7, 320 9.0 : 8.2, of 32 / 32 heads 384 10.9 : 9.2; two trees, 32 / 32, 512 12.4 : 10.4
//   80 blocks, 2048 tokens 29.9 : 23.3 | 25.4 : 18.9;  96 blocks, 4096 51 .. 56 : 39 .. 41 | 43 : 34, 8192 71 .. 83 : 68 .. 76 | 57 .. 71 : 58 .. 75
// More blocks than SMs: their waves fill up, and with lengths that differ short blocks run beside a long one, where splits of it
// only add starts and merges.  No splits up to 128 tiles:
//   160 blocks, 2048 tokens 55 : 44 | 44 : 23, 4096 85 : 77 | 53 : 44, 8192 144 : 147 | 85 : 82 (16384 226 : 295 | 156 : 135)
//   192 blocks, 2048 56 : 48 | 44 .. 49 : 25 .. 34, 4096 86 : 82 | 58 : 42; 320 blocks, 4096 142 : 126 | 103 : 78
inline int choose_splits(int base_ctas, int sm_count, int prefix_tiles, const int* cluster_cap) {
    if (base_ctas > sm_count && prefix_tiles <= 128) return 1;
    int best = 1;
    long best_cost = 0;
    for (int s = 1; s <= ATT_MAX_SPLIT; ++s) {
        if (s > 1 && s > prefix_tiles) break;
        const long ctas = (long)base_ctas * s;
        const long cap = cluster_cap[s] > 0 ? cluster_cap[s] : sm_count;
        const long waves = (ctas + cap - 1) / cap;
        const long cost = waves * (2 * ((prefix_tiles + s - 1) / s) + 24 + (s > 1 ? 9 : 0));
        if (s == 1 || cost < best_cost) { best_cost = cost; best = s; }
    }
    return best;
}

// Splits with which tree_attn_duo_kernel takes a launch, 0: tree_attn_umma_kernel takes it.
// What is known is the number of query blocks (an upper bound: small trees leave blocks empty) and the longest prefix; how the other
// lengths lie below it the host cannot tell (the cache arrays may be larger than what is in use), so every line is drawn for equal
// lengths and for lengths spread over 0.2 .. 1 of the longest together.  The other kernel pays for whole waves of CTAs, each with 6.5 us
// around its tiles that nothing overlaps, but one CTA of it is through its tiles in half the time, which decides where the lengths
// differ.  us a call, back to back, other kernel : this one, equal lengths | spread (30 .. 40 nodes of one block, 60 of two):
//     blocks     512 tokens     1024                          2048                          4096
//     160        22.5 : 16.0    29.5 : 23.5 | 18.9 : 23.6     47 : 39 | 23 : 35             80 : 70 | 36 : 56
//     192        21.8 : 16.0    29.8 : 24.1 | 20.1 : 22.0     48 : 41 | 25 .. 34 : 37       82 : 73 | 42 : 61
//     256        24.7 : 18.9    32.6 : 27.7 | 22.3 : 22.3     51 : 47 | 36 : 39             89 : 86 | 56 : 66
//     320        34.6 : 31.7    46.3 : 48.1 | 34.3 : 27.9     73 : 79 | 46 : 40             126 : 143 | 78 : 79
//     384        35.0 : 31.9    47.8 : 48.4 | 37.8 : 38.3     76 : 85 | 54 : 58             135 : 162 | 84 : 91
//     512        48.8 : 36.2    64.4 : 55.2 | 48.3 : 40.0     101 : 94 | 75 : 70            188 : 153 | 148 : 104
//     1024       103 : 79       114 : 97 | 97 : 80            168 : 164 | 135 : 119         302 : 299 | 224 : 211
//   - a second wave of at most a sixth: up to 8 tiles; else up to 16 tiles; above three waves at any length; up to 32 tiles where the last of
//     two or three waves is at least a quarter empty and more than a sixth full.
//   At most one block per SM: only two splits let CTAs share SMs.  It pays in more than three quarters of the SMs from 256 tiles on, with one query
//   block per head from 448.  Mean of equal lengths and of three draws of spread ones (the longest is the stated one), pauses of 30 ms between
//   bursts | without pauses, under the power cap:
//     trees x nodes, heads       12288 tokens          16384                 24576                 28000                 32768
//     7 x 60, 32 / 8             111 : 110 | 107 : 107 145 : 142 | 142 : 139 210 : 201 | 210 : 203 239 : 227 | 245 : 232 281 : 264 | 287 : 271
//     9 x 60, 32 / 8             116 : 116 | 113 : 113 153 : 150 | 154 : 151 225 : 216 | 232 : 224 264 : 253 | 289 : 276 296 : 280 | 306 : 286
//     4 x 60, 64 / 8, <true>                           147 : 146 | 141 : 141 216 : 208 | 209 : 207 243 : 234 | 249 : 239
//       <false> (2.342e-3 from fp64, this one 2.337e-3)  133       | 134       199       | 208       233       | 241
//   (The other kernel's times but the last line's first two are from before its barriers were asked ahead, which took 3 to 7 % off them.  The lines stay: what goes
//   to this kernel by them would come back less exact.)
//     14 x 30, 32 / 8                                  145 : 146 | 141 : 145 213 : 210 | 223 : 216 238 : 239 | 264 : 252 276 : 278 | 296 : 286
//     18 x 30, 32 / 8                                  154 : 163 | 153 : 165 231 : 240 | 249 : 257 265 : 274 | 289 : 292 314 : 320 | 339 : 332
// Two CTAs on an SM is what runs (128 blocks of 129 tiles take 104 us alone, 256 blocks 146), also in pairs; cudaOccupancyMaxActiveClusters
// counts one, as it does for any kernel that allocates tensor memory (it does not know how many columns), so it is not asked.
inline int duo_splits(int base_ctas, int mblocks, int sm_count, int prefix_tiles) {
    if (base_ctas <= sm_count) return 4 * base_ctas > 3 * sm_count && prefix_tiles >= (mblocks > 1 ? 256 : 448) ? 2 : 0;
    if (6 * base_ctas <= 7 * sm_count) return prefix_tiles <= 8 ? 1 : 0;
    const int waves = (base_ctas + sm_count - 1) / sm_count;
    return prefix_tiles <= 16 || (prefix_tiles <= 32 && 4 * base_ctas <= 3 * waves * sm_count) || waves > 3 ? 1 : 0;
}

// Launches that tree_attn_duo_kernel takes as long for or longer, and rounds a little less (FOLLOW makes up for it): second or third waves that are at least
// a quarter empty, with several query blocks per head.  FOLLOW has its price where two waves of equal lengths follow one another: 10 trees of 60
// nodes, 32 / 8 heads, plain : FOLLOW : tree_attn_duo_kernel's better choice, equal | spread: 2048 tokens 42 : 44 : 55 | 24 : 23 : 42, 4096 71 : 77 : 76 | 43 : 44 :
// 53, 8192 132 : 147 : 144 | 82 : 82 : 85.  One query block per head was never that kernel's: plain (5 trees of 40 nodes, 32 / 32 heads,
// FOLLOW 4096 tokens 82.9 : 80.3 | 43.8 : 42.0, 8192 160 : 150 | 83 : 82).
inline bool wants_follow(int base_ctas, int mblocks, int sm_count, int prefix_tiles) {
    if (mblocks == 1 || base_ctas <= sm_count) return false;
    const int waves = (base_ctas + sm_count - 1) / sm_count;
    return prefix_tiles <= 64 ? 4 * base_ctas <= 3 * waves * sm_count : prefix_tiles <= 128 && 6 * base_ctas <= 7 * sm_count;
}

struct AttnChoice {
    bool duo;                        // tree_attn_duo_kernel
    bool follow;                     // tree_attn_umma_kernel<true>
    int splits;
};
// blocks: query blocks of all (sequence, head) pairs, mblocks: of one; cluster_cap[s]: CTAs of tree_attn_umma_kernel that run at once in clusters of s
inline AttnChoice attn_choice(int blocks, int mblocks, int sm_count, int prefix_tiles, const int* cluster_cap) {
    const int duo = duo_splits(blocks, mblocks, sm_count, prefix_tiles);
    if (duo) return {true, false, duo};
    return {false, wants_follow(blocks, mblocks, sm_count, prefix_tiles), choose_splits(blocks, sm_count, prefix_tiles, cluster_cap)};
}

// Does a launch of tree_attn_umma_kernel have CTAs that take Q as the A operand from tensor memory: those of more than ATT_Q_TILES tiles?
// With 64 columns of S the product reads Q from shared memory for longer than it multiplies (387 clocks a tile instead of 258, 623 instead of 515 with P V), but the copy
// of Q and the slower issue are paid for first, and where the tiles are not what a launch waits for nothing comes back.  us a call, from shared memory : so,
// equal lengths | mean of three draws of spread ones; tokens for each split, i.e. 27, 32, 36, 41, 64, 128 tiles in a CTA and the tree's:
//     trees x nodes, heads     1700                      2000                      2300                      2600                      4096                      8192
//     4 x 60, 64 / 8           20.1 : 20.3 | 20.2 : 20.2 22.4 : 22.3 | 22.7 : 22.0 24.4 : 23.8 | 24.5 : 23.9 27.2 : 26.1 | 26.9 : 25.4 37.1 : 35.5 | 37.8 : 34.7 66.9 : 64.1 | 63.0 : 60.3
//     7 x 60, 32 / 8           20.1 : 20.2 | 19.4 : 19.5 22.2 : 22.3 | 22.0 : 21.6 24.4 : 24.6 | 23.9 : 23.2 25.7 : 26.3 | 26.1 : 25.3 38.7 : 36.2 | 35.3 : 35.0 69.5 : 63.9 | 65.2 : 60.2
//     4 x 60, 32 / 8, 2 splits 22.0 : 23.1 | 22.5 : 21.9 24.1 : 24.8 | 24.6 : 23.5 27.4 : 27.2 | 26.8 : 25.5 30.2 : 29.3 | 29.7 : 27.6 41.8 : 39.1 | 41.3 : 37.6 76.1 : 70.0 | 72.5 : 62.7
//     2 x 60, 32 / 8, 4 splits 21.2 : 22.5 | 21.4 : 21.1 23.7 : 23.9 | 24.0 : 23.0 27.2 : 26.9 | 26.7 : 25.7 29.1 : 28.6 | 28.4 : 26.5 41.1 : 38.7 | 40.8 : 36.7 76.0 : 69.9 | 73.2 : 64.0
// Not in more than one wave (16 x 60, 32 / 8, 1700 tokens 41.5 : 44.0 | 33.3 : 33.7, 4096 77.2 : 77.4 | 50.1 : 51.9; 10 x 60 1700 37.4 : 40.8 | 23.0 : 23.0, 12000 in splits 156 :
// 162 | 114 : 118; 8 x 60, 64 / 8, 4096 72.5 : 74.8 | 60.4 : 62.9) but for FOLLOW's above 64 tiles (10 x 60, 8192 124 : 127 | 73.5 : 69.9), and not with one query
// block per head, where K and V come from DRAM (10 x 30, 32 / 8, 8192 66.5 : 68.7 | 49.3 : 50.4; 4 x 60, 32 / 32, 1700 23.1 : 24.2 | 21.0 : 21.2).
#define ATT_Q_TILES 31
inline bool q_from_tensor_memory(int blocks, int mblocks, int sm_count, int prefix_tiles, int tree_tiles, const AttnChoice& c) {
    if (c.duo || mblocks == 1 || (prefix_tiles + c.splits - 1) / c.splits + tree_tiles <= ATT_Q_TILES) return false;
    return c.follow ? prefix_tiles > 64 : blocks * c.splits <= sm_count;
}
