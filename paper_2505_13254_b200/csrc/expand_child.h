// The row statistics a child of an expansion level reads.  On its own so that its range can be checked on the host.
#pragma once

#include <stddef.h>

#ifdef __CUDACC__
#define HS_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define HS_HOST_DEVICE inline
#endif

// Child `t` of sequence b: token and log-confidence of the i-th best token (i = t % k) of the draft row after frontier node
// j = t / k.  Statistics row b * k + j exists only for the `nf` nodes of the frontier - at the first level that is the root alone,
// and the arrays may end right behind the last sequence's -, so nothing is read for the others.  Returns whether t is a child.
template <class Vals, class Tokens>
HS_HOST_DEVICE bool load_child(int t, int b, int k, int nf, int stride, Vals topk_val, Tokens topk_idx, Vals row_lse, int& tok, float& lc) {
    if (t >= nf * k) return false;
    const int j = t / k, i = t - j * k;
    const size_t row = (size_t)b * k + j, at = row * stride + i;
    tok = topk_idx[at];
    lc = topk_val[at] - row_lse[row];
    return true;
}
