// Rounds of a vocabulary row: 128 vectors of 16 bytes, four per lane of a warp.  Shared by the entropy pass and the acceptance.
#pragma once

#include <math_constants.h>

#include "hs_common.cuh"
#include "hs_ptx.cuh"

#define LOG2E 1.4426950408889634f
#define ROUND_VECS 128

template <bool BF16>
__device__ __forceinline__ void unpack(const uint4& v, float* x) {
    if (BF16) {
        x[0] = bf16_lo(v.x); x[1] = bf16_hi(v.x); x[2] = bf16_lo(v.y); x[3] = bf16_hi(v.y);
        x[4] = bf16_lo(v.z); x[5] = bf16_hi(v.z); x[6] = bf16_lo(v.w); x[7] = bf16_hi(v.w);
    } else {
        x[0] = __uint_as_float(v.x); x[1] = __uint_as_float(v.y);
        x[2] = __uint_as_float(v.z); x[3] = __uint_as_float(v.w);
    }
}

__device__ __forceinline__ float ex2f(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// The largest key of the warp (0 = none) and the lane that holds it; keys are distinct.
__device__ __forceinline__ unsigned long long warp_best_key(unsigned long long k, int& src) {
    const unsigned int hi = (unsigned int)(k >> 32), mh = __reduce_max_sync(HS_FULL_MASK, hi);
    const unsigned int lo = hi == mh ? (unsigned int)k : 0u, ml = __reduce_max_sync(HS_FULL_MASK, lo);
    src = __ffs(__ballot_sync(HS_FULL_MASK, hi == mh && lo == ml)) - 1;
    return ((unsigned long long)mh << 32) | ml;
}

// -inf in place of what vector v of a row holds past the vocabulary
template <bool BF16>
__device__ __forceinline__ void mask_tail(uint4& d, int v, int vocab) {
    constexpr int VE = BF16 ? 8 : 4;
    unsigned int* wd = reinterpret_cast<unsigned int*>(&d);
#pragma unroll
    for (int e = 0; e < VE; ++e)
        if (v * VE + e >= vocab) {
            if (BF16) wd[e >> 1] = (e & 1) ? ((wd[e >> 1] & 0x0000ffffu) | 0xff800000u) : ((wd[e >> 1] & 0xffff0000u) | 0x0000ff80u);
            else wd[e] = 0xff800000u;
        }
}

// One round of a segment: vectors [128 r, 128 r + 128) of the row, -inf where they lie past its end.
template <bool BF16, class P>       // P: vocab and nvec of the rows
__device__ __forceinline__ void load_round(const P& p, const uint4* rowv, int r, int lane, uint4 (&d)[4]) {
    const uint4* src = rowv + (size_t)r * ROUND_VECS + lane;
    if ((r + 1) * ROUND_VECS < p.nvec) {                       // (the row's last vector may be partial: it takes the other way)
#pragma unroll
        for (int j = 0; j < 4; ++j) d[j] = ld_stream(src + j * 32);
        return;
    }
    const unsigned int ninf = BF16 ? 0xff80ff80u : 0xff800000u;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int v = r * ROUND_VECS + j * 32 + lane;
        d[j] = v < p.nvec ? ld_stream(src + j * 32) : make_uint4(ninf, ninf, ninf, ninf);
        if (v == p.nvec - 1) mask_tail<BF16>(d[j], v, p.vocab);
    }
}
// largest of a lane's logits of a round
template <bool BF16>
__device__ __forceinline__ float round_max(const uint4 (&d)[4]) {
    if (BF16) {
        const __nv_bfloat162* w = reinterpret_cast<const __nv_bfloat162*>(&d[0]);
        __nv_bfloat162 a = __hmax2(w[0], w[1]), b = __hmax2(w[2], w[3]), c = __hmax2(w[4], w[5]), e = __hmax2(w[6], w[7]);
        a = __hmax2(a, w[8]); b = __hmax2(b, w[9]); c = __hmax2(c, w[10]); e = __hmax2(e, w[11]);
        a = __hmax2(a, w[12]); b = __hmax2(b, w[13]); c = __hmax2(c, w[14]); e = __hmax2(e, w[15]);
        a = __hmax2(__hmax2(a, b), __hmax2(c, e));
        const unsigned int u = *reinterpret_cast<const unsigned int*>(&a);
        return fmaxf(bf16_lo(u), bf16_hi(u));
    }
    const float* x = reinterpret_cast<const float*>(&d[0]);
    float a = max3(x[0], x[1], x[2]), b = max3(x[3], x[4], x[5]);
    a = max3(a, x[6], x[7]); b = max3(b, x[8], x[9]);
    a = max3(a, x[10], x[11]); b = max3(b, x[12], x[13]);
    return fmaxf(max3(a, x[14], x[15]), b);
}
