// Which attention kernel takes a launch, and in how many splits of the prefix.  On its own so that the host can check which one a launch runs.
#pragma once

#define ATT_MAX_SPLIT 8

// KV splits (= cluster size) of tree_attn_umma_kernel: the number with the least time on the critical path, waves of CTAs (as many
// clusters of that size as the device runs at once) times {tiles per CTA, what lies around them, merge}, in half tiles.  A tile is
// 0.5 us (0.38 in CTAs that take Q from tensor memory), start, tree tiles and output 6 us, the merge of splits 2.2 us.  us a call in 1 .. 6 splits, * the rule's (seven and
// eight splits of these do not fit at once: another wave), trees of 60 nodes, equal lengths:
//     one tree, 32 / 8 heads, 256 tokens     7.6* 9.1  8.4  8.5  8.6  8.7     384       8.6  9.4  9.1  8.2  8.7  9.2*    1024      12.7 11.9 10.3 9.8  9.7  9.6*
//                             2048           20.6 15.0 13.1 11.8 11.1 11.2*   4096      32.9 23.2 18.4 15.2 14.7 13.7*   8192      57.5 36.0 28.1 23.5 22.0 19.6*
//     one tree, 64 / 8,       512            9.7  10.1 10.3 10.3*             2048      21.3 16.1 14.2 13.7*             8192      59.3 37.1 29.6 26.0*
//     two trees, 32 / 32,     512            9.6* 11.4                        2048      20.9 17.3*
//     four trees, 32 / 8,     1024           13.9 13.8*                       4096      35.6 26.9*
//   and where splits cost a wave, equal lengths | lengths spread over 0.2 .. 1 of the longest, 1 .. 3 splits:
//     80 blocks, 4096 tokens  38.2* 46.7 39.3 | 34.6* 29.3 33.3;  96 blocks, 8192  65.7* 74.5 82.9 | 63.6* 57.5 67.0
// More blocks than SMs: their waves fill up, and with lengths that differ short blocks run beside a long one, where splits of it
// only add starts and merges.  No splits up to 128 tiles:
//     160 blocks, 2048 tokens 41.0* 51.6 60.7 | 23.4* 39.8 49.6;  8192  121.8* 113.6 116.1 | 76.0* 86.0 98.8;  16384, four there  231 202 200 202* | 125 105 117 124*
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
// differ.  us a call, back to back, other kernel : this one, equal lengths | mean of three draws of spread ones (trees of 60 nodes, 32 / 8 heads):
//     blocks     512 tokens                 1024                       2048                       4096
//     160        20.7 : 18.6 | 16.8 : 16.4  27.4 : 26.9 | 18.6 : 22.5  41.8 : 42.7 | 25.3 : 38.9  69.2 : 72.5 | 37.1 : 65.1
//     192        21.1 : 18.6 | 16.9 : 15.9  28.0 : 26.9 | 20.9 : 23.7  43.5 : 43.9 | 28.7 : 39.7  70.8 : 75.9 | 46.0 : 70.7
//     256        22.1 : 19.4 | 19.2 : 18.0  30.3 : 27.7 | 23.5 : 25.5  45.6 : 44.1 | 33.6 : 39.7  77.2 : 79.0 | 49.7 : 69.8
//     320        32.0 : 31.3 | 26.4 : 24.6  45.0 : 44.6 | 34.8 : 33.5  65.5 : 70.5 | 47.0 : 42.0  107 : 123 | 72.0 : 73.1
//     384        34.1 : 32.2 | 29.9 : 28.7  46.7 : 45.7 | 37.5 : 36.4  68.2 : 72.2 | 48.5 : 46.3  116 : 128 | 75.0 : 77.6
//     512        48.1 : 38.2 | 39.9 : 31.0  62.1 : 53.9 | 50.8 : 41.7  89.6 : 87.4 | 68.6 : 62.7  156 : 160 | 103 : 103
//     1024       87.7 : 70.7 | 78.3 : 60.0  114 : 98.9 | 93.2 : 76.8   168 : 169 | 127 : 119      295 : 309 | 200 : 204
//   - a second wave of at most a sixth: up to 8 tiles; else up to 16 tiles; above three waves at any length; up to 32 tiles where the last of
//     two or three waves is at least a quarter empty and more than a sixth full.
//   At most one block per SM: only two splits let CTAs share SMs.  In more than three quarters of the SMs that was the faster way from 256 tiles on, with one query
//   block per head from 448, and as exact as the following instance.  Since the other kernel asks its barriers ahead and takes Q from tensor memory it is the slower
//   way for several query blocks per head: the lines are from before, and would lie elsewhere today.  us a call, this kernel : <false> : <true>, equal lengths | mean of three
//   draws of spread ones, pauses of 30 ms between bursts of 20 calls (without pauses, under the power cap, the same within 5 %):
//     trees x nodes, heads    16384 tokens                      24576                             32768
//     4 x 60, 64 / 8          146 : 127 : 128 | 142 : 120 : 121 213 : 189 : 190 | 203 : 175 : 176 282 : 251 : 251 | 263 : 227 : 229
//     7 x 60, 32 / 8          147 : 127 : 128 | 136 : 118 : 118 213 : 189 : 189 | 197 : 170 : 170 281 : 251 : 252 | 257 : 223 : 224
//     9 x 60, 32 / 8          166 : 147 : 148 | 141 : 121 : 122 245 : 221 : 221 | 205 : 179 : 179 324 : 294 : 296 | 270 : 236 : 237
//     14 x 30, 32 / 8                                                                             320 : 311 : 315 | 263 : 241 : 247
//     18 x 30, 32 / 8                                                                             380 : 364 : 374 | 294 : 273 : 275
//   2-norm relative error against fp64, in 1e-3, the same order: 4 x 60 2.3423 : 2.3458 : 2.3422, 2.3416 : 2.3438 : 2.3400, 2.3436 : 2.3440 : 2.3419; 7 x 60
//   2.3422 : 2.3450 : 2.3433, 2.3420 : 2.3467 : 2.3415, 2.3424 : 2.3438 : 2.3417.
// Two CTAs on an SM is what runs (128 blocks of 129 tiles take 104 us alone, 256 blocks 146), also in pairs; cudaOccupancyMaxActiveClusters
// counts one, as it does for any kernel that allocates tensor memory (it does not know how many columns), so it is not asked.
inline int duo_splits(int base_ctas, int mblocks, int sm_count, int prefix_tiles) {
    if (base_ctas <= sm_count) return 4 * base_ctas > 3 * sm_count && prefix_tiles >= (mblocks > 1 ? 256 : 448) ? 2 : 0;
    if (6 * base_ctas <= 7 * sm_count) return prefix_tiles <= 8 ? 1 : 0;
    const int waves = (base_ctas + sm_count - 1) / sm_count;
    return prefix_tiles <= 16 || (prefix_tiles <= 32 && 4 * base_ctas <= 3 * waves * sm_count) || waves > 3 ? 1 : 0;
}

// Launches that tree_attn_duo_kernel takes as long for or longer, and rounds a little less (FOLLOW makes up for it): second or third waves that are at least
// a quarter empty, with several query blocks per head.  What FOLLOW costs, 10 trees of 60 nodes, 32 / 8 heads, plain : FOLLOW : tree_attn_duo_kernel, equal | spread:
// 2048 tokens 41.8 : 42.1 : 42.7 | 25.3 : 25.5 : 38.9, 4096 69.2 : 72.0 : 72.5 | 37.1 : 36.5 : 65.1, 8192 122 : 125 : 136 | 70.4 : 67.5 : 120 (FOLLOW's of the last two with Q from tensor memory).
// One query block per head was never that kernel's: plain (5 trees of 40 nodes, 32 / 32 heads, 4096 tokens 78.4 : 82.3 | 47.6 : 47.7, 8192 144 : 151 | 80.5 : 80.6).
inline bool wants_follow(int base_ctas, int mblocks, int sm_count, int prefix_tiles) {
    if (mblocks == 1 || base_ctas <= sm_count) return false;
    const int waves = (base_ctas + sm_count - 1) / sm_count;
    return prefix_tiles <= 64 ? 4 * base_ctas <= 3 * waves * sm_count : prefix_tiles <= 128 && 6 * base_ctas <= 7 * sm_count;
}

struct AttnChoice {
    bool duo;                        // tree_attn_duo_kernel
    bool follow;                     // tree_attn_umma_kernel with FOLLOW
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
// of Q and the slower issue are paid for first, and where the tiles are not what a launch waits for nothing comes back.  us a call, inputs rotating through more than twice
// L2, from shared memory : so, equal lengths | mean of three draws of spread ones; tokens for each split, i.e. 30, 33, 36, 41 and 64 tiles in a CTA and the tree's:
//     trees x nodes, heads     1900                      2100                      2300                      2600                      4096
//     4 x 60, 64 / 8           21.9 : 22.4 | 21.8 : 21.8 23.4 : 23.7 | 23.3 : 22.9 24.8 : 25.0 | 25.2 : 24.2 27.2 : 27.1 | 27.2 : 26.5 37.9 : 37.3 | 37.1 : 35.9
//     4 x 36, 64 / 8           20.9 : 22.1 | 20.5 : 21.4 22.4 : 23.4 | 21.7 : 22.6 23.9 : 24.7 | 22.2 : 23.6 26.0 : 26.9 | 25.5 : 26.1 37.2 : 36.9 | 34.7 : 35.2
//     7 x 60, 32 / 8           22.2 : 22.5 | 21.2 : 21.6 23.2 : 23.9 | 22.7 : 22.9 24.8 : 25.3 | 24.1 : 24.1 27.4 : 27.6 | 26.2 : 26.4 40.6 : 37.5 | 37.2 : 36.4
//     9 x 60, 32 / 8           22.2 : 23.5 | 21.9 : 22.2 23.9 : 25.2 | 22.8 : 22.8 25.9 : 26.5 | 24.5 : 24.3 29.0 : 28.9 | 26.6 : 26.8 42.0 : 40.2 | 39.7 : 37.4
//     4 x 60, 32 / 8, 2 splits 25.1 : 25.9 | 24.8 : 24.1 26.6 : 26.8 | 26.4 : 25.1 28.3 : 28.3 | 28.1 : 26.6 31.1 : 30.4 | 30.6 : 28.7 43.3 : 40.2 | 42.9 : 39.0
//     2 x 60, 32 / 8, 4 splits 24.0 : 25.2 | 23.8 : 23.4 26.0 : 26.9 | 26.0 : 25.6 27.7 : 28.3 | 27.5 : 26.8 30.1 : 30.3 | 29.2 : 27.7 42.9 : 40.6 | 42.1 : 38.2
// Not in more than one wave (16 x 60, 32 / 8, 1700 tokens 41.5 : 44.0 | 33.3 : 33.7, 4096 77.2 : 77.4 | 50.1 : 51.9; 10 x 60 1700 37.4 : 40.8 | 23.0 : 23.0, 12000 in splits 156 :
// 162 | 114 : 118; 8 x 60, 64 / 8, 4096 72.5 : 74.8 | 60.4 : 62.9; FOLLOW's 12 x 60, 32 / 8, 4096 72.8 : 74.0 | 46.8 : 47.9) but for FOLLOW's above 60 tiles with a second wave of at
// most a sixth (10 x 60, 32 / 8, 4096 71.0 : 72.2 | 38.8 : 36.9, 8192 124 : 127 | 73.5 : 69.9; at 3500 62.0 : 65.2 | 36.9 : 36.2).  With one query block per head, unsplit from 49 tiles on (10 x 30, 32 / 8,
// 2500 tokens 23.4 : 22.8 | 20.0 : 21.2), up to three quarters of the SMs (one tree of 30, 32 / 8, 16384 tokens 24.7 : 24.4, 32768 41.5 : 39.1; two trees 32768 53.7 : 49.9 | 53.7 : 49.1; 10 trees 4096 42.1 : 40.1 | 35.5 : 35.1): with
// more of them the tiles wait for DRAM (four trees, 128 CTAs, 12288 37.7 : 38.3 | 33.9 : 33.0, 24576 64.7 : 66.1 | 57.6 : 58.3; 4 x 60, 32 / 32, 1700 23.1 : 24.2 | 21.0 : 21.2).
#define ATT_Q_TILES 34
inline bool q_from_tensor_memory(int blocks, int mblocks, int sm_count, int prefix_tiles, int tree_tiles, const AttnChoice& c) {
    if (c.duo || (prefix_tiles + c.splits - 1) / c.splits + tree_tiles <= (mblocks > 1 || c.splits > 1 ? ATT_Q_TILES : 48)) return false;
    if (c.follow) return 6 * blocks <= 7 * sm_count && prefix_tiles > 60;
    return mblocks > 1 ? blocks * c.splits <= sm_count : 4 * blocks * c.splits <= 3 * sm_count;
}
