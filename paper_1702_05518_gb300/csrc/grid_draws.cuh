// grid_draws.cuh -- what the grid-sweep kernels (colour_grid.cu: whole sweeps of a per-colour
// sampler in one cooperative launch) share: the end of a sweep, where every block sums all blocks'
// partials and draws tau, beta0 and sigma^2 of every chain, and the end of the launch.
#pragma once

#include "gmrf_device.cuh"
#include "gmrf_internal.h"
#include "grid_barrier.cuh"
#include "hyper_task.cuh"

namespace gmrf {

constexpr int kGridChains = 8;   // the most chains (padded) of a grid sweep
constexpr int kGridGpre = 128;   // sweeps whose precomputed variates are staged in shared memory

// One per block, in shared memory.
struct GridShared {
    float hs[kGridChains][3];                 // tau, 1/sigma^2, beta0 of the current sweep per chain
    double dcur[kGridChains][2];              // tau and sigma^2 (FP64) as last drawn, per chain
    double gsh[kGridGpre][kGridChains][3];    // the batch's precomputed variates
    int abort;
};

// By all threads of the block, before a block barrier.
__device__ __forceinline__ void grid_draws_init(GridShared &sh, const HyperArgs &h, int count, long long sweep0)
{
    const int Cp = h.Cp, tid = threadIdx.x, nt = blockDim.x;
    const long long bbase = h.ctl->batch_base, bcount = h.ctl->batch_count;
    for (int q = tid; q < Cp * 3; q += nt) {
        const int v = q / 3, k = q - 3 * v;
        sh.hs[v][k] = static_cast<const float *>(h.hyp)[v * kHypStride + k];
    }
    if (tid < Cp) {
        sh.dcur[tid][0] = h.tau[tid];
        sh.dcur[tid][1] = h.sig2[tid];
    }
    if (tid == 0) sh.abort = 0;
    for (int q = tid; q < min(count, kGridGpre) * Cp * 3; q += nt) {
        const int it = q / (Cp * 3), rem = q - it * Cp * 3, v = rem / 3, k = rem - 3 * v;
        const long long kb = sweep0 + it - bbase;
        sh.gsh[it][v][k] = (h.gpre && kb >= 0 && kb < bcount) ? h.gpre[(kb * h.nfields * Cp + v) * 4 + k] : 0.0;
    }
}

// The draws at the end of sweep sw (the it-th of the launch), by warp 2v + which of every block for
// chain v: which 0 tau, 1 beta0 and then sigma^2, from the partials pm ([chain][S, R, A][block]) and
// the batch's precomputed variates, by hyper_draw; with `rec` (one block) also stored and traced.
__device__ __forceinline__ void grid_draw(GridShared &sh, const HyperArgs &h, const double *pm, int nblk,
                                          const FieldDev &f, long long sw, int it, bool rec)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp >= 2 * h.Cp) return;
    const int chain = warp >> 1, which = warp & 1;
    const bool need_sum = which ? (h.draw || h.draw_beta) : h.draw;
    const bool need_a = which && h.draw_beta;
    double S = 0.0, A = 0.0;
    if (need_sum) {
        const double *pc = pm + chain * 3 * nblk;
        hyper_sums_by_field(pc + which * nblk, pc + 2 * nblk, need_a, nblk, S, A);
    }
    if (lane == 0) {
        const long long kb = sw - h.ctl->batch_base;
        const bool pre = h.gpre && kb >= 0 && kb < h.ctl->batch_count;
        double gpv = 0.0, zb = 0.0;
        if (pre) {
            if (it < kGridGpre) {
                gpv = sh.gsh[it][chain][which];
                zb = sh.gsh[it][chain][2];
            } else {
                const double *gp = h.gpre + (kb * h.nfields * h.Cp + chain) * 4;
                gpv = gp[which];
                zb = gp[2];
            }
        }
        // (the tau draw reads neither sigma^2 nor beta0, which the other warp replaces)
        const double cur = sh.dcur[chain][which], s2old = which ? sh.dcur[chain][1] : 0.0;
        const double b = which ? static_cast<double>(sh.hs[chain][2]) : 0.0;
        double val, bval;
        hyper_draw<float>(h, which, chain, chain, sw, S, A, cur, s2old, b, gpv, zb, pre, 0, f.stream, f.n, f.rank, val,
                          bval, rec);
        if (which == 0) {
            if (h.draw) sh.hs[chain][0] = static_cast<float>(val);
        } else {
            if (h.draw_beta) sh.hs[chain][2] = static_cast<float>(bval);
            if (h.draw) sh.hs[chain][1] = static_cast<float>(1.0 / val);
        }
        sh.dcur[chain][which] = val;
    }
}

// The block's sums of V chains per thread (chain vector cv = thread mod CV, CV a power of two):
// a shuffle tree over the lanes of a chain vector, then the warps in order; FP32, stored in FP64 as
// partial `blk` of pm.  `red`: [warps][kGridChains][3] in shared memory.  Ends before a block barrier.
template <int V, int NT>
__device__ __forceinline__ void grid_partials(const float (&aS)[V], const float (&aR)[V], const float (&aA)[V], int CV,
                                              int Cp, float (&red)[NT / 32][kGridChains][3], double *pm, int nblk)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int v = 0; v < V; ++v) {
        float sS = aS[v], sR = aR[v], sA = aA[v];
        for (int o = 16; o >= CV; o >>= 1) {
            sS += __shfl_xor_sync(0xffffffffu, sS, o);
            sR += __shfl_xor_sync(0xffffffffu, sR, o);
            sA += __shfl_xor_sync(0xffffffffu, sA, o);
        }
        if (lane < CV) {
            red[warp][lane * V + v][0] = sS;
            red[warp][lane * V + v][1] = sR;
            red[warp][lane * V + v][2] = sA;
        }
    }
    __syncthreads();
    if (threadIdx.x < Cp * 3) {
        const int chain = threadIdx.x / 3, k = threadIdx.x - 3 * chain;
        float s = 0.0f;
#pragma unroll
        for (int w = 0; w < NT / 32; ++w) s += red[w][chain][k];
        pm[(chain * 3 + k) * nblk + blockIdx.x] = static_cast<double>(s);
    }
}

// The end of a launch: the last block to finish advances the counters and clears the barrier.
__device__ __forceinline__ void grid_finish(SweepCtl *ctl, long long sweep_end, long long acc_count)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&ctl->ticket, 1ull) == gridDim.x - 1) {
            ctl->sweep = sweep_end;
            ctl->fnext = sweep_end;
            ctl->acc_count = acc_count;
            ctl->ticket = 0;
            ctl->gbar = 0;
            ctl->gabort = 0;
        }
    }
}

}  // namespace gmrf
