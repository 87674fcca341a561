// The token of four whose mass takes a running sum past the goal of an inverse-CDF draw.  On its own so that its roundings can be checked
// on the host.
#pragma once

#ifdef __CUDACC__
#define HS_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define HS_HOST_DEVICE inline
#endif

// t: masses (none negative), run: the sum ahead of them, at most `goal`.  `run` becomes the sum behind them, two additions of pairs deep
// (dependent fp64 additions are 64 clocks each).  Returns -1 where that does not exceed the goal; else the first token at which
// the sum taken one by one does, and where its roundings leave none the last token with mass: never one without.
HS_HOST_DEVICE int crossing_of_four(const double (&t)[4], double goal, double& run) {
    const double next = run + ((t[0] + t[1]) + (t[2] + t[3]));
    int at = -1;
    if (next > goal) {
        double r = run;
        bool found = false;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            r += t[e];
            if (!found && t[e] > 0.0) { at = e; found = r > goal; }
        }
    }
    run = next;
    return at;
}
