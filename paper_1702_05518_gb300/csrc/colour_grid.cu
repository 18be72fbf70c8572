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
#include "packed_f32.cuh"

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
        double *const pm = ra.pm + (it & 1) * 3 * Cp * nblk;  // (a graph of one colour has one barrier per sweep)
        for (int c = 0; c < K; ++c) {
            for (int q = tid; (q >> cvs) < cnt; q += kGridThreads) {
                if (q != tid) fetch(lo + (q >> cvs), sw, acc);  // beyond one position per thread
                update(coffs[c], acc, inv_k);
            }
            if (c + 1 == K) grid_partials<V, kGridThreads>(aS, aR, aA, CV, Cp, red, pm, nblk);
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
        grid_draw(sh, h, pm, nblk, f, sw, it, blockIdx.x == 0);
        __syncthreads();
    }
    grid_finish(a.ctl, sweep0 + ra.count, acc_count);
}

// Units of GS sites in a row of W sites of a 3-D lattice: for one or two chains the GS = 4 / chains
// sites of a Philox block, which are consecutive natural sites, so a block across a row end is a
// unit of both rows; for more chains a site has blocks of its own and a unit is a pair.
__host__ __device__ constexpr int unit_sites(int Cp) { return Cp == 1 ? 4 : 2; }
__host__ __device__ inline int units_per_row(int Cp, int W)
{
    const int gs = unit_sites(Cp);
    return (W + gs - 1) / gs + ((Cp < 4 && W % gs != 0) ? 1 : 0);
}

// 3-D 6-neighbour lattices, parity colouring.  A thread owns M units (row, unit of the row) and
// updates in each colour step the sites of that colour among them, V chains of each: one Philox
// block serves sites of both colours, and a unit's normals and observations stay in registers for the
// sweep.  With four sites to a unit the two of a colour lie two columns apart and share an in-row
// neighbour and everything that depends on the row.  A block's units are consecutive, so all
// neighbours but those a plane apart mostly lie in the block's own range and come from L1.  The loads
// of two units are issued together.  Bound by the latency of a sweep (two barriers, the partials' sums
// and the draws, about 8 us however small the lattice) and, beyond, by instruction issue.  Per
// sweep, against a launch per colour and one for the draws: 91 x 109 x 91 with one chain 14.5 us (26
// before, 29 with the draws' sums by one warp), 60 x 60 x 61 with two chains 11 (26), with four 12.5
// (19.5), 40 x 40 x 41 with eight 13 (34).
template <int CP, int M>
__global__ void __launch_bounds__(kGridThreads, 1) lattice3d_grid_kernel(const GridSweepArgs ra)
{
    constexpr int V = CP < 4 ? CP : 4, CV = CP / V, GS = unit_sites(CP), NK = GS / 2;
    constexpr int UB = (CP == 1 && M > 1) ? 2 : 1;  // units whose loads are in flight together
    const StepArgs &a = ra.s;
    const HyperArgs &h = ra.h;
    __shared__ GridShared sh;
    __shared__ float red[kGridThreads / 32][kGridChains][3];
    __shared__ float coef[7][3][CP];  // per degree and chain: tau rho / P, (1/sigma^2) / P, 1/sqrt(P)
    const int tid = threadIdx.x;
    const FieldDev f = a.fields[0];
    const int L = f.dims[0], H = f.dims[1], W = f.dims[2], cols = f.cols, plane = H * cols;
    const int c0 = (tid & (CV - 1)) * V;
    const int nblk = gridDim.x;
    const long long sweep0 = a.ctl->sweep;
    long long acc_count = a.ctl->acc_count;
    const float rho = static_cast<float>(a.rho), om = 1.0f - rho;
    const int64_t sub = static_cast<int64_t>(f.rows) * cols;
    float *XF = static_cast<float *>(a.x) + f.slot0 * CP + c0;
    float *MF = static_cast<float *>(a.mean) + f.slot0 * CP + c0;
    float *QF = static_cast<float *>(a.m2) + f.slot0 * CP + c0;
    const float *YF = static_cast<const float *>(a.y) + f.slot0;
    grid_draws_init(sh, h, ra.count, sweep0);

    // This block's items (a unit's chain vector each): item m of the thread is item0 + m NT.  A
    // unit's place, found once per launch: the column j0 of its first site (it may lie before the
    // row; beyond it for no unit), the slot ro of its row's first column, and flags: bit 0 the
    // colour of column j0, bits 1..4 which of the rows i - 1, i + 1, l - 1, l + 1 exist.
    const int upr = units_per_row(CP, W);
    const int items = f.rows * upr * CV;
    const int per = ((items + nblk - 1) / nblk + CV - 1) / CV * CV;
    int j0[M], ro[M];
    uint32_t fl[M];
    float z[M][GS][V], y[M][GS];
#pragma unroll
    for (int m = 0; m < M; ++m) {
        const int64_t q = static_cast<int64_t>(blockIdx.x) * per + tid + m * kGridThreads;
        const bool on = tid + m * kGridThreads < per && q < items;
        const int unit = on ? static_cast<int>(q / CV) : 0;
        const int r = fast_div(unit, ra.u_m, ra.u_s), l = fast_div(r, f.h_m, f.h_s), i = r - l * H;
        j0[m] = CP < 4 ? ((r * W) / GS + unit - r * upr) * GS - r * W : (unit - r * upr) * GS;
        if (!on) j0[m] = W;
        ro[m] = r * cols;
        fl[m] = static_cast<uint32_t>((l + i + j0[m]) & 1) | (i > 0 ? 2u : 0u) | (i + 1 < H ? 4u : 0u) |
                (l > 0 ? 8u : 0u) | (l + 1 < L ? 16u : 0u);
#pragma unroll
        for (int k = 0; k < GS; ++k) {
            const int j = j0[m] + k;
            y[m][k] = 0.0f;
            if (static_cast<unsigned>(j) < static_cast<unsigned>(W)) y[m][k] = YF[((l + i + j) & 1) * sub + ro[m] + (j >> 1)];
        }
    }
    auto normals = [&](long long sw) {
#pragma unroll
        for (int m = 0; m < M; ++m) {
            if (j0[m] >= W) continue;
            const int s0 = fast_div(ro[m], f.cols_m, f.cols_s) * W + j0[m];  // natural index of the unit's first site
#pragma unroll
            for (int b = 0; b < (CP < 4 ? 1 : GS); ++b) {
                const uint32_t blk = CP < 4 ? static_cast<uint32_t>(s0 / GS) : static_cast<uint32_t>(s0 + b);
                const uint4 w = philox4x32_10_rk(make_uint4(blk, static_cast<uint32_t>(sw), f.stream,
                                                            (kTagX << 24) | static_cast<uint32_t>(c0 >> 2)), a.rk);
                f2 z01, z23;
                box_muller_block_f32x2(w, z01, z23);
                float q[4];
                upk(z01, q[0], q[1]);
                upk(z23, q[2], q[3]);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if constexpr (CP < 4) z[m][k / V][k % V] = q[k];
                    else z[m][b][k] = q[k];
                }
            }
        }
    };
    normals(sweep0);
    __syncthreads();

    float aS[V], aR[V], aA[V];
    bool acc = false;
    float inv_k = 0.0f;
    // The sites of a unit that a colour step updates, columns j and (GS 4) j + 2: in-row neighbours
    // j - 1, j + 1 (, j + 3) and the neighbours in the four rows around.
    struct Pair {
        float in[NK + 1][V], off[4][NK][V], mu[NK][V], mm[NK][V];
        int rb;
        uint32_t in_ok, on;
    };
    auto load = [&](Pair &t, int m, int c) {
        const int j = j0[m] + static_cast<int>((fl[m] ^ c) & 1u);
        t.rb = ro[m] + (j >> 1);
        t.in_ok = 0u;
        t.on = 0u;
        const int64_t so = c * sub + t.rb, oo = (1 - c) * sub + t.rb;
        const float *xo = XF + oo * CP;
        const float *xi = xo + ((j & 1) - 1) * CP;
#pragma unroll
        for (int k = 0; k <= NK; ++k) {
            const bool ok = static_cast<unsigned>(j - 1 + 2 * k) < static_cast<unsigned>(W);
            t.in_ok |= ok ? 1u << k : 0u;
#pragma unroll
            for (int v = 0; v < V; ++v) t.in[k][v] = 0.0f;
            if (ok) Vec<float, V>::ld(xi + k * CP, t.in[k]);
        }
#pragma unroll
        for (int k = 0; k < NK; ++k) {
            const bool on = static_cast<unsigned>(j + 2 * k) < static_cast<unsigned>(W);
            t.on |= on ? 1u << k : 0u;
            const int step[4] = {-cols * CP, cols * CP, -plane * CP, plane * CP};
#pragma unroll
            for (int d = 0; d < 4; ++d) {
#pragma unroll
                for (int v = 0; v < V; ++v) t.off[d][k][v] = 0.0f;
                if (on && ((fl[m] >> (1 + d)) & 1u)) Vec<float, V>::ld(xo + step[d] + k * CP, t.off[d][k]);
            }
            if (acc && on) {
                Vec<float, V>::ld(MF + (so + k) * CP, t.mu[k]);
                Vec<float, V>::ld(QF + (so + k) * CP, t.mm[k]);
            }
        }
    };
    auto update = [&](Pair &t, int m, int c) {
        const bool odd = ((fl[m] ^ c) & 1u) != 0;
        const int64_t so = c * sub + t.rb;
#pragma unroll
        for (int k = 0; k < NK; ++k) {
            if (!((t.on >> k) & 1u)) continue;
            const uint32_t in2 = (t.in_ok >> k) & 3u;
            const int dg = __popc((fl[m] & 30u) | (in2 << 8));
            const float yv = odd ? y[m][2 * k + 1] : y[m][2 * k];
            float xn[V];
#pragma unroll
            for (int v = 0; v < V; ++v) {
                float s = t.in[k][v] + t.in[k + 1][v];
#pragma unroll
                for (int d = 0; d < 4; ++d) s += t.off[d][k][v];
                const float yb = yv - sh.hs[c0 + v][2];
                const float zv = odd ? z[m][2 * k + 1][v] : z[m][2 * k][v];
                xn[v] = fmaf(zv, coef[dg][2][c0 + v], fmaf(coef[dg][0][c0 + v], s, yb * coef[dg][1][c0 + v]));
                const float r = yb - xn[v];
                aR[v] = fmaf(r, r, aR[v]);
                aA[v] += r;
            }
            Vec<float, V>::st(XF + (so + k) * CP, xn);
            if (c == 1) {
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    float e = 0.0f;
#pragma unroll
                    for (int q = 0; q < 2; ++q)
                        if ((in2 >> q) & 1u) {
                            const float df = xn[v] - t.in[k + q][v];
                            e = fmaf(df, df, e);
                        }
#pragma unroll
                    for (int d = 0; d < 4; ++d)
                        if ((fl[m] >> (1 + d)) & 1u) {
                            const float df = xn[v] - t.off[d][k][v];
                            e = fmaf(df, df, e);
                        }
                    aS[v] = fmaf(rho, e, aS[v]);
                }
            }
            if (om != 0.0f) {
#pragma unroll
                for (int v = 0; v < V; ++v) aS[v] = fmaf(om * static_cast<float>(dg) * xn[v], xn[v], aS[v]);
            }
            if (acc) {
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    const float delta = xn[v] - t.mu[k][v];
                    t.mu[k][v] = fmaf(delta, inv_k, t.mu[k][v]);
                    t.mm[k][v] = fmaf(delta, xn[v] - t.mu[k][v], t.mm[k][v]);
                }
                Vec<float, V>::st(MF + (so + k) * CP, t.mu[k]);
                Vec<float, V>::st(QF + (so + k) * CP, t.mm[k]);
            }
        }
    };

    unsigned long long arrivals = ra.extra_arrivals;
    for (int it = 0; it < ra.count; ++it) {
        const long long sw = sweep0 + it;
        acc = sweep_accumulated(sw, a.burn_in, a.thin);
        inv_k = acc ? 1.0f / static_cast<float>(acc_count + 1) : 0.0f;
        if (tid < 7 * CP) {
            const int dg = tid / CP, v = tid - dg * CP;
            const float P = fmaf(sh.hs[v][0], static_cast<float>(dg), sh.hs[v][1]);
            const float rP = rcp_approx(P);
            coef[dg][0][v] = sh.hs[v][0] * rho * rP;
            coef[dg][1][v] = sh.hs[v][1] * rP;
            coef[dg][2][v] = rsqrt_approx(P);
        }
#pragma unroll
        for (int v = 0; v < V; ++v) {
            aS[v] = 0.0f;
            aR[v] = 0.0f;
            aA[v] = 0.0f;
        }
        __syncthreads();
        double *const pm = ra.pm + (it & 1) * 3 * CP * nblk;
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
#pragma unroll
            for (int m0 = 0; m0 < M; m0 += UB) {
                Pair t[UB];
#pragma unroll
                for (int u = 0; u < UB; ++u) load(t[u], m0 + u, c);
#pragma unroll
                for (int u = 0; u < UB; ++u) update(t[u], m0 + u, c);
            }
            if (c == 1) grid_partials<V, kGridThreads>(aS, aR, aA, CV, CP, red, pm, nblk);
            __syncthreads();  // the block's stores of this step
            if (tid == 0) grid_arrive(a.ctl);
            arrivals += nblk;
            if (c == 1 && it + 1 < ra.count) normals(sw + 1);
            if (tid == 0 && grid_wait(a.ctl, arrivals, ra.wait_ns)) sh.abort = 1;
            __syncthreads();
            if (sh.abort) break;
        }
        if (sh.abort) break;
        if (acc) ++acc_count;
        grid_draw(sh, h, pm, nblk, f, sw, it, blockIdx.x == 0);
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

// Units per thread of the 3-D kernel: 1, 2 or 4, up to what its registers hold.
template <typename Use>
cudaError_t with_lattice3d_kernel(int Cp, int M, Use &&use)
{
    switch (Cp) {
    case 1: return M == 1 ? use(lattice3d_grid_kernel<1, 1>) : M == 2 ? use(lattice3d_grid_kernel<1, 2>) : use(lattice3d_grid_kernel<1, 4>);
    case 2: return M == 1 ? use(lattice3d_grid_kernel<2, 1>) : M == 2 ? use(lattice3d_grid_kernel<2, 2>) : use(lattice3d_grid_kernel<2, 4>);
    case 4: return M == 1 ? use(lattice3d_grid_kernel<4, 1>) : use(lattice3d_grid_kernel<4, 2>);
    default: return M == 1 ? use(lattice3d_grid_kernel<8, 1>) : use(lattice3d_grid_kernel<8, 2>);
    }
}
int64_t lattice3d_items(int Cp, int64_t rows, int W) { return rows * units_per_row(Cp, W) * (Cp == 8 ? 2 : 1); }
int lattice3d_units(int Cp, int64_t rows, int W, int blocks)  // per thread: 1, 2 or 4; 0 too many
{
    const int64_t per = (lattice3d_items(Cp, rows, W) + blocks - 1) / blocks + 1;  // (rounded to pairs of items)
    for (int m : {1, 2, 4})
        if (per <= static_cast<int64_t>(m) * kGridThreads) return (m == 4 && Cp >= 4) ? 0 : m;
    return 0;
}

// The SMs of the device if `per_sm` blocks (at least one) can be resident on each for a cooperative
// launch, at most the partials that one warp sums (hyper_sums_by_field); else 0.
template <typename With>
cudaError_t grid_capacity(With &&with, int *most)
{
    *most = 0;
    int dev = 0, sms = 0, coop = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (e == cudaSuccess)
        e = with([&](auto *k) { return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kGridThreads, 0); });
    if (e == cudaSuccess && coop && per_sm >= 1) *most = sms < 32 * kSumRows ? sms : 32 * kSumRows;
    return e;
}
int grid_size(int64_t items, int most)
{
    const int64_t want = (items + kGridMinItems - 1) / kGridMinItems;
    return static_cast<int>(want < most ? want : most);
}

}  // namespace

cudaError_t plan_csr_grid(int Cp, bool weighted, int ncolors, int largest_class, int *blocks)
{
    *blocks = 0;
    if (Cp > kGridChains || ncolors > kGridMaxColours || largest_class < 1) return cudaSuccess;
    int most = 0;
    const cudaError_t e = grid_capacity([&](auto &&use) { return with_csr_kernel(Cp, weighted, use); }, &most);
    if (e != cudaSuccess || !most) return e;
    const int64_t items = static_cast<int64_t>(largest_class) * (Cp < 2 ? 1 : Cp / 2);
    if (items <= static_cast<int64_t>(most) * kGridThreads * kGridItems) *blocks = grid_size(items, most);
    return cudaSuccess;
}

cudaError_t launch_csr_grid(int blocks, const GridSweepArgs &ra, cudaStream_t stream)
{
    return with_csr_kernel(ra.s.Cp, ra.s.w != nullptr, [&](auto *k) { return launch_coop(k, blocks, ra, stream); });
}

cudaError_t plan_lattice3d_grid(int Cp, int64_t rows, int W, int *blocks)
{
    *blocks = 0;
    if (Cp > kGridChains || rows < 1) return cudaSuccess;
    int most = 0;
    const cudaError_t e = grid_capacity([&](auto &&use) { return with_lattice3d_kernel(Cp, 4, use); }, &most);
    if (e != cudaSuccess || !most) return e;
    const int b = grid_size(lattice3d_items(Cp, rows, W), most);
    if (lattice3d_units(Cp, rows, W, b)) *blocks = b;
    return cudaSuccess;
}

cudaError_t launch_lattice3d_grid(int blocks, int64_t rows, int W, const GridSweepArgs &ra, cudaStream_t stream)
{
    GridSweepArgs g = ra;
    fast_div_magic(static_cast<uint32_t>(units_per_row(ra.s.Cp, W)), g.u_m, g.u_s);
    return with_lattice3d_kernel(ra.s.Cp, lattice3d_units(ra.s.Cp, rows, W, blocks),
                                 [&](auto *k) { return launch_coop(k, blocks, g, stream); });
}

}  // namespace gmrf
