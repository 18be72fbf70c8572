// fp64_steps.cuh -- what the FP64 lattice steps (lattice_fused.cu, the lattices of sweep_kernels.cu) do
// once per block instead of once per thread or site, and their sums over a warp.  The FP64 units are
// the scarce resource (a warp's operation occupies an SM's for about 15 cycles).
#pragma once

#include "gmrf_device.cuh"

namespace gmrf {

// 1/sqrt(P) in 64-bit fixed point (normals_f64.cuh's square root without the last product): at most 0.51
// units in the last place, 1/sqrt(P) by two library operations 1.47; a tenth of their latency (a
// dependent FP64 operation takes 36 ns).
__device__ __forceinline__ double rsqrt_fixed(double P)
{
    const uint64_t b = static_cast<uint64_t>(__double_as_longlong(P));
    const int E = static_cast<int>(b >> 52);
    if (E < 1 || E >= 0x7FF) return 1.0 / sqrt(P);  // zero, subnormal, negative, infinite or NaN
    // P = A / 2^64 * 2^ex, A / 2^64 in [1/4, 1), ex even
    uint64_t A = (b << 11) | 0x8000000000000000ull;
    int ex = E - 1022;
    const int odd = ex & 1;
    const float af = __uint_as_float((static_cast<uint32_t>(126 - odd) << 23) + (static_cast<uint32_t>(A >> 40) & 0x7FFFFFu));
    A >>= odd;
    ex += odd;
    const uint32_t y0 = __float2uint_rz(rsqrt_approx(af) * 0x1p30f);
    const uint64_t s0 = mul_32_64(y0, A);
    const int64_t r = static_cast<int64_t>((1ull << 60) - mul_32_64(y0, s0));  // 1 - A y0^2, 60 fraction bits
    const int64_t rh = r >> 12;
    const int64_t c = (r >> 1) + ((3 * (rh * rh)) >> 39);
    const int64_t y = static_cast<int64_t>(y0) << 31;
    return double_of(static_cast<uint64_t>(y + __mul64hi(y, c << 4)), 3 - (ex >> 1), false);
}

// The coefficients of a lattice site's draw x = ca s + (cb (y - beta0) + crs z) per degree and chain
// ([degree][Cp][3]; P = tau d + 1/sigma^2 takes no other values): ca = tau rho / P, cb = 1/(sigma^2 P), crs =
// 1/sqrt(P).  One operation is left between the neighbours' sum and the draw, and the quotient and the
// root of every site (a third of its FP64 operations) are gone (64^2: 10.1 -> 9.9 us per sweep, 48^3 with two chains
// 38 -> 36, against a table of 1/P and 1/sqrt(P) alone).  A warp each makes the first two and the
// third, another 1/k of the running moments (every thread's own quotient took 1.5 us of a 512-thread
// block).  By all threads (at least 96), before a block barrier.
__device__ __forceinline__ void degree_table(double *tab, double &inv_k, const double *hyp, int Cp, double rho, bool acc,
                                             const SweepCtl *ctl)
{
    const int warp = threadIdx.x >> 5;
    if (warp < 2) {
        for (int q = threadIdx.x & 31; q < 9 * Cp; q += 32) {
            const int d = q / Cp, v = q - d * Cp;
            const double tau = hyp[kHypStride * v], isig = hyp[kHypStride * v + 1];
            const double P = tau * static_cast<double>(d) + isig;
            if (warp == 0) {
                const double rP = 1.0 / P;
                tab[3 * q] = tau * rho * rP;
                tab[3 * q + 1] = isig * rP;
            } else {
                tab[3 * q + 2] = rsqrt_fixed(P);
            }
        }
    } else if (threadIdx.x == 64) {
        inv_k = acc ? 1.0 / static_cast<double>(ctl->acc_count + 1) : 0.0;
    }
}

// The draw from entry q of that table.
__device__ __forceinline__ double table_draw(const double *q, double s, double res, double z)
{
    return fma(q[0], s, fma(q[1], res, q[2] * z));
}

// A sum of neighbours (or warps) by pairs: half the latency of one after the other.
template <int N>
__device__ __forceinline__ double pair_sum(const double *t, int stride)
{
    if constexpr (N == 1) return t[0];
    else return pair_sum<(N + 1) / 2>(t, stride) + pair_sum<N / 2>(t + (N + 1) / 2 * stride, stride);
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
