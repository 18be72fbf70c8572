// colour_grid.cu -- grid sweeps: a batch of whole sweeps of a per-colour sampler (Algorithm 1 with
// the conjugate draws of Sec. 3.1) in one cooperative launch, for a single FP32 field whose colour
// steps are too short for a launch each.  Every block owns a share of every colour class; a colour
// step ends at a grid barrier (grid_barrier.cuh), and after the last one every block sums all blocks'
// partials and draws the parameters (grid_draws.cuh), so a sweep is K barriers and no launch.
//
// What a step waits for is latency, so everything that does not depend on the other blocks happens
// while the barrier completes: a thread loads the graph row, observation, running moments and
// degree of its next position and draws its normals between the block's arrival and its wait.
// After the wait only the neighbours' values are left to gather.  The gathers are ordinary loads:
// the barrier's acquire orders them after the other blocks' stores, and within a step a value is
// read by several positions of a block from L1.
#include <cuda_runtime.h>

#include "gmrf_device.cuh"
#include "gmrf_internal.h"
#include "grid_draws.cuh"

namespace gmrf {
namespace {

constexpr int kGridThreads = 512;  // 16 drawing warps (two per chain); 128 registers
constexpr int kGridMaxColours = 64;

// CSR graphs: V chains per thread (two, or the one there is), W: weighted edges.  A block's share of a
// class is a contiguous range of positions (breadth-first order, so neighbours tend to lie in the
// same share).  The first R neighbours of a row are loaded ahead and kept; longer rows (one vertex in
// 60 of a Delaunay graph) load the rest after the wait, two dependent round trips.  Bound by the
// latency of a step (arrival, wait, gathers): 100,003 weighted sites, 6 colours, 4 chains on 152
// blocks take 20.5 us per sweep, where a launch per colour and one for the draws took 59; four
// chains per thread with 8 neighbours ahead (registers allow no more) took 26.
template <int V, bool W>
__global__ void __launch_bounds__(kGridThreads, 1) csr_grid_kernel(const GridSweepArgs ra)
{
    constexpr int R = 12;
    const StepArgs &a = ra.s;
    const HyperArgs &h = ra.h;
    __shared__ GridShared sh;
    __shared__ float red[kGridThreads / 32][kGridChains][3];
    __shared__ int coffs[kGridMaxColours + 1];
    const int tid = threadIdx.x;
    const FieldDev f = a.fields[0];
    const int K = f.ncolors, Cp = a.Cp, CV = Cp / V, cvs = __ffs(CV) - 1;
    const int c0 = (tid & (CV - 1)) * V;  // first chain of this thread
    const int nblk = gridDim.x;
    const long long sweep0 = a.ctl->sweep;
    long long acc_count = a.ctl->acc_count;
    const float rho = static_cast<float>(a.rho);
    const int32_t *rp = a.rp + f.rp0, *ci = a.ci + f.nnz0;
    const float *wr = W ? static_cast<const float *>(a.w) + f.nnz0 : nullptr;
    const float *DEG = static_cast<const float *>(a.deg) + f.csr0;
    const int32_t *perm = a.perm + f.csr0;
    const float *Y = static_cast<const float *>(a.y) + f.slot0;
    float *X = static_cast<float *>(a.x) + f.slot0 * Cp + c0;
    float *MEAN = static_cast<float *>(a.mean) + f.slot0 * Cp + c0;
    float *M2 = static_cast<float *>(a.m2) + f.slot0 * Cp + c0;
    for (int c = tid; c <= K; c += kGridThreads) coffs[c] = a.coff[f.coff0 + c];
    grid_draws_init(sh, h, ra.count, sweep0);
    __syncthreads();

    // This block's positions of class c: [lo, lo + cnt).
    auto share = [&](int c, int &lo, int &cnt) {
        const int len = coffs[c + 1] - coffs[c], per = (len + nblk - 1) / nblk;
        const int o = min(static_cast<int>(blockIdx.x) * per, len);
        lo = coffs[c] + o;
        cnt = min(per, len - o);
    };
    // One position's data that no other block writes.
    int p = -1, rb = 0, nn = 0, id[R];
    float w[R], yv = 0, d = 0, z[V], mu[V], mm[V];
    auto fetch = [&](int pos, long long sw, bool acc) {
        p = pos;
        rb = rp[pos];
        nn = rp[pos + 1] - rb;
#pragma unroll
        for (int q = 0; q < R; ++q) {
            id[q] = q < nn ? ci[rb + q] : 0;
            if (W) w[q] = q < nn ? wr[rb + q] : 0.0f;
        }
        yv = Y[pos];
        d = DEG[pos];
        const uint32_t site = static_cast<uint32_t>(perm[pos]);
        if (acc) {
            Vec<float, V>::ld(MEAN + static_cast<int64_t>(pos) * Cp, mu);
            Vec<float, V>::ld(M2 + static_cast<int64_t>(pos) * Cp, mm);
        }
        site_normals<float, V>(a.key, site, static_cast<uint32_t>(sw), f.stream, static_cast<uint32_t>(c0), a.lanes, z);
    };
    float aS[V], aR[V], aA[V];
    auto update = [&](int lo_class, bool acc, float inv_k) {
        float nb[R][V], s[V];
#pragma unroll
        for (int q = 0; q < R; ++q) {
#pragma unroll
            for (int v = 0; v < V; ++v) nb[q][v] = 0.0f;
            if (q < nn) Vec<float, V>::ld(X + static_cast<int64_t>(id[q]) * Cp, nb[q]);
        }
#pragma unroll
        for (int v = 0; v < V; ++v) s[v] = 0.0f;
#pragma unroll
        for (int q = 0; q < R; ++q)
#pragma unroll
            for (int v = 0; v < V; ++v) s[v] += W ? w[q] * nb[q][v] : nb[q][v];
        for (int k = rb + R; k < rb + nn; ++k) {
            float xv[V];
            Vec<float, V>::ld(X + static_cast<int64_t>(ci[k]) * Cp, xv);
            const float wv = W ? wr[k] : 1.0f;
#pragma unroll
            for (int v = 0; v < V; ++v) s[v] += wv * xv[v];
        }
        float xn[V], e[V];
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const float tau = sh.hs[c0 + v][0], isig = sh.hs[c0 + v][1], beta = sh.hs[c0 + v][2];
            const float P = tau * d + isig;
            const float m = (tau * rho * s[v] + (yv - beta) * isig) * rcp_approx(P);
            xn[v] = m + z[v] * rsqrt_approx(P);
            const float r = (yv - beta) - xn[v];
            aR[v] += r * r;
            aA[v] += r;
            e[v] = 0.0f;
        }
        Vec<float, V>::st(X + static_cast<int64_t>(p) * Cp, xn);
#pragma unroll
        for (int q = 0; q < R; ++q)
            if (q < nn && id[q] < lo_class) {  // a neighbour of lower colour: final
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    const float df = xn[v] - nb[q][v];
                    e[v] += W ? w[q] * df * df : df * df;
                }
            }
        for (int k = rb + R; k < rb + nn; ++k) {
            const int jn = ci[k];
            if (jn >= lo_class) continue;
            float xv[V];
            Vec<float, V>::ld(X + static_cast<int64_t>(jn) * Cp, xv);
            const float wv = W ? wr[k] : 1.0f;
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const float df = xn[v] - xv[v];
                e[v] += wv * df * df;
            }
        }
#pragma unroll
        for (int v = 0; v < V; ++v) aS[v] += (1.0f - rho) * d * xn[v] * xn[v] + rho * e[v];
        if (acc) {
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const float delta = xn[v] - mu[v];
                mu[v] += delta * inv_k;
                mm[v] += delta * (xn[v] - mu[v]);
            }
            Vec<float, V>::st(MEAN + static_cast<int64_t>(p) * Cp, mu);
            Vec<float, V>::st(M2 + static_cast<int64_t>(p) * Cp, mm);
        }
    };

    int lo, cnt;
    share(0, lo, cnt);
    bool acc = sweep_accumulated(sweep0, a.burn_in, a.thin);
    if ((tid >> cvs) < cnt) fetch(lo + (tid >> cvs), sweep0, acc);
    unsigned long long arrivals = ra.extra_arrivals;
    for (int it = 0; it < ra.count; ++it) {
        const long long sw = sweep0 + it;
        const bool acc_next = sweep_accumulated(sw + 1, a.burn_in, a.thin);
        const float inv_k = acc ? 1.0f / static_cast<float>(acc_count + 1) : 0.0f;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            aS[v] = 0.0f;
            aR[v] = 0.0f;
            aA[v] = 0.0f;
        }
        for (int c = 0; c < K; ++c) {
            for (int q = tid; (q >> cvs) < cnt; q += kGridThreads) {
                if (q != tid) fetch(lo + (q >> cvs), sw, acc);  // beyond one position per thread
                update(coffs[c], acc, inv_k);
            }
            if (c + 1 == K) grid_partials<V, kGridThreads>(aS, aR, aA, CV, Cp, red, ra.pm, nblk);
            __syncthreads();  // the block's stores of this step
            if (tid == 0) grid_arrive(a.ctl);
            arrivals += nblk;
            const bool last = c + 1 == K && it + 1 == ra.count;
            if (!last) {
                const bool wrap = c + 1 == K;
                share(wrap ? 0 : c + 1, lo, cnt);
                if ((tid >> cvs) < cnt) fetch(lo + (tid >> cvs), wrap ? sw + 1 : sw, wrap ? acc_next : acc);
            }
            if (tid == 0 && grid_wait(a.ctl, arrivals, ra.wait_ns)) sh.abort = 1;
            __syncthreads();
            if (sh.abort) break;
        }
        if (sh.abort) break;
        if (acc) ++acc_count;
        acc = acc_next;
        grid_draw(sh, h, ra.pm, nblk, f, sw, it, blockIdx.x == 0);
        __syncthreads();
    }
    grid_finish(a.ctl, sweep0 + ra.count, acc_count);
}

template <typename Kernel>
cudaError_t launch_coop(Kernel kernel, int blocks, const GridSweepArgs &ra, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(kGridThreads);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, ra);
}

// The kernel of a configuration, passed to `use` (null if there is none).
template <typename Use>
cudaError_t with_csr_kernel(int Cp, bool weighted, Use &&use)
{
    if (Cp > 1) return weighted ? use(csr_grid_kernel<2, true>) : use(csr_grid_kernel<2, false>);
    return weighted ? use(csr_grid_kernel<1, true>) : use(csr_grid_kernel<1, false>);
}

}  // namespace

cudaError_t plan_csr_grid(int Cp, bool weighted, int ncolors, int largest_class, int *blocks)
{
    *blocks = 0;
    if (Cp > kGridChains || ncolors > kGridMaxColours || largest_class < 1) return cudaSuccess;
    int dev = 0, sms = 0, coop = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (e == cudaSuccess)
        e = with_csr_kernel(Cp, weighted, [&](auto *k) {
            return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kGridThreads, 0);
        });
    if (e != cudaSuccess || !coop || per_sm < 1) return e;
    const int64_t items = static_cast<int64_t>(largest_class) * (Cp < 2 ? 1 : Cp / 2);
    const int most = sms < 32 * kSumRows ? sms : 32 * kSumRows;  // partials one warp sums (hyper_sums_by_field)
    if (items > static_cast<int64_t>(most) * kGridThreads * kGridItems) return cudaSuccess;
    const int64_t want = (items + kGridMinItems - 1) / kGridMinItems;
    *blocks = static_cast<int>(want < most ? want : most);
    return cudaSuccess;
}

cudaError_t launch_csr_grid(int blocks, const GridSweepArgs &ra, cudaStream_t stream)
{
    return with_csr_kernel(ra.s.Cp, ra.s.w != nullptr, [&](auto *k) { return launch_coop(k, blocks, ra, stream); });
}

}  // namespace gmrf
