// fp64_steps.cuh -- what the FP64 lattice steps (lattice_fused.cu, the lattices of sweep_kernels.cu) do
// once per block instead of once per thread or site, and their sums over a warp.  The FP64 units are
// the scarce resource (a warp's operation occupies an SM's for about 15 cycles).
#pragma once

#include "gmrf_device.cuh"

namespace gmrf {

// 1/P and 1/sqrt(P) per degree and chain ([degree][Cp][2]; P takes no other values on a lattice, and two
// FP64 quotients and a root per site were a third of its FP64 operations) by one warp each, and 1/k of
// the running moments by a third (every thread's own quotient took 1.5 us of a 512-thread block).  By all
// threads (at least 96), before a block barrier.
__device__ __forceinline__ void degree_table(double *tab, double &inv_k, const double *hyp, int Cp, bool acc, const SweepCtl *ctl)
{
    const int warp = threadIdx.x >> 5;
    if (warp < 2) {
        for (int q = threadIdx.x & 31; q < 9 * Cp; q += 32) {
            const int d = q / Cp, v = q - d * Cp;
            const double P = hyp[kHypStride * v] * static_cast<double>(d) + hyp[kHypStride * v + 1];
            tab[2 * q + warp] = warp == 0 ? 1.0 / P : 1.0 / sqrt(P);
        }
    } else if (threadIdx.x == 64) {
        inv_k = acc ? 1.0 / static_cast<double>(ctl->acc_count + 1) : 0.0;
    }
}

// The sums of S and R over the lanes equal mod CV (CV a power of two, at most 16): in lanes below 16
// the S sum, in the others the R sum.  The pairs that are added are those of two shuffle trees, so the sums
// are theirs bit for bit, with half the additions after the first step.
__device__ __forceinline__ double warp_sum_pair(double S, double R, int CV)
{
    const bool high = threadIdx.x & 16;
    double keep = high ? R : S;
    keep += __shfl_xor_sync(0xffffffffu, high ? S : R, 16);
    for (int off = 8; off >= CV; off >>= 1) keep += __shfl_xor_sync(0xffffffffu, keep, off);
    return keep;
}

}  // namespace gmrf
