// sweep_kernels.cu -- the per-colour fused update of the chromatic Gibbs sampler (Algorithm 1,
// steps 2-3), the fused reductions behind the conjugate hyperparameter draws (Sec. 3.1), the
// hyperparameter draw itself, and the pack/unpack kernels of the colour-split layout.
//
// One launch of colour_step_kernel covers colour class c of every field: each block takes one
// tile (a range of sub-array rows of a lattice field, or of permuted positions of a CSR field)
// and, for every site i of the tile and every chain,
//     s_i = sum_j w_ij x_j                         (neighbours all have other colours)
//     P_i = tau d_i + 1/sigma^2,  m_i = (tau rho s_i + y_i/sigma^2) / P_i
//     x_i = m_i + z_i / sqrt(P_i),                 z_i Philox/Box-Muller normal of (site, sweep)
// (with the intercept of Sec. 3.1, y_i - beta0 in place of y_i) and accumulates, per chain, the
// sums the conjugate draws need:
//     (1 - rho) d_i x_i^2 + rho sum_{j lower colour} w_ij (x_i - x_j)^2,
//     (y_i - beta0 - x_i)^2  and  y_i - beta0 - x_i,
// so that after the last colour every undirected edge has been counted once, at its endpoint
// of higher colour, with both endpoints final: summed over sites this is x'(D - rho W)x.
// Thread, warp and block partial sums are in the state precision (a tile holds at most a few
// thousand terms); the sums over tiles are FP64; every sum is taken in a fixed order, so
// results are reproducible run to run.  When the sweep is accumulated, the Welford
// running mean and M2 of the site are updated in the same pass.
#include <cuda_runtime.h>

#include <type_traits>

#include "fp64_steps.cuh"
#include "gmrf_device.cuh"
#include "gmrf_internal.h"
#include "gamma_pre.cuh"
#include "hyper_task.cuh"
#include "pg.cuh"

namespace gmrf {
namespace {

template <typename T> struct Arith;
template <> struct Arith<float> {
    // 1/P and 1/sqrt(P) within 1 ulp (P is a normal float): well inside the FP32 parity budget.
    __device__ __forceinline__ static float rcp(float x) { return rcp_approx(x); }
    __device__ __forceinline__ static float rsq(float x) { return rsqrt_approx(x); }
};
template <> struct Arith<double> {
    __device__ __forceinline__ static double rcp(double x) { return 1.0 / x; }
    __device__ __forceinline__ static double rsq(double x) { return 1.0 / sqrt(x); }
};

// Observation models of the colour kernels (compile-time): Gaussian noise without or with the
// intercept beta0 (Sec. 3.1), or binomial counts with the logistic link and Polya-Gamma
// augmentation (Sec. 3.2; y holds the successes, the trials come separately).
enum : int { kModelGauss = 0, kModelGaussIntercept = 1, kModelBinomial = 2 };

template <typename T, int V>
struct SiteCtx {
    T tau[V], isig[V], beta[V];  // per chain of this thread
    T accS[V], accR[V], accA[V]; // thread partial sums
    T inv_k;             // 1 / (accumulated count) when accumulating
    bool acc;
    const T *tab;        // FP64 lattices: the draws' coefficients by degree and chain (fp64_steps.cuh)
    bool icar;           // rho = 1
};
// Whether a kernel uses that table.
template <typename T, int KIND, int MODEL> constexpr bool kDegreeTable = sizeof(T) == 8 && KIND != kCsr && MODEL != kModelBinomial;

// Draw (or, in reduce-only mode, read) the V chain values of one site given its neighbour sum s
// and the neighbour values nb[k] of the neighbours flagged in `lower_mask` (those of lower
// colour), and fold the site's terms into the partial sums.  zdrawn: its normals if already drawn.
//
// Binomial model: psi | beta0, x_i ~ PG(m_i, beta0 + x_i) was drawn from the site's value at the
// start of the sweep (the Polya-Gamma stage); x_i gets precision tau d_i + psi and mean
// (tau rho s_i + kappa_i - psi beta0) / P,
// kappa_i = y_i - m_i / 2; the partial sums then collect psi and kappa_i - psi x_i (for beta0)
// in place of the Gaussian residual sums.
template <typename T, int V, int NB, int MODEL, bool TAB = false>
__device__ __forceinline__ void finish_site(const StepArgs &a, SiteCtx<T, V> &cx, T *xp, T *meanp, T *m2p,
                                            T yv, int mtr, T d, uint32_t site, uint32_t sweep, uint32_t stream,
                                            uint32_t chain0, const T (&s)[V], const T (&nb)[NB][V],
                                            uint32_t lower_mask, const T (&wnb)[NB], const T *zdrawn = nullptr,
                                            int dg = 0)
{
    const T rho = static_cast<T>(a.rho);
    T xn[V];
    // Running moments first, so their loads do not wait behind the store of x (possible alias);
    // with four chains per thread the registers are better spent elsewhere.
    T mu[V], mm[V];
    constexpr bool kEarly = V <= 2;
    if (kEarly && cx.acc) {
        Vec<T, V>::ld(meanp, mu);
        Vec<T, V>::ld(m2p, mm);
    }
    T psi[V];
    const T kappa = yv - static_cast<T>(0.5) * static_cast<T>(mtr);
    if (MODEL == kModelBinomial && a.update) {
        T z[V];
        // psi of this site and chain, drawn by the Polya-Gamma stage from the start-of-sweep state
        Vec<T, V>::ld(static_cast<const T *>(a.psi) + (xp - static_cast<T *>(a.x)), psi);
        if (zdrawn) {
#pragma unroll
            for (int v = 0; v < V; ++v) z[v] = zdrawn[v];
        } else {
            site_normals<T, V>(a.key, site, sweep, stream, chain0, a.lanes, z);
        }
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const T P = cx.tau[v] * d + psi[v];
            const T m = (cx.tau[v] * rho * s[v] + kappa - psi[v] * cx.beta[v]) * Arith<T>::rcp(P);
            xn[v] = m + z[v] * Arith<T>::rsq(P);
        }
        Vec<T, V>::st(xp, xn);
    } else if (a.update) {
        T z[V];
        if (zdrawn) {
#pragma unroll
            for (int v = 0; v < V; ++v) z[v] = zdrawn[v];
        } else {
            site_normals<T, V>(a.key, site, sweep, stream, chain0, a.lanes, z);
        }
#pragma unroll
        for (int v = 0; v < V; ++v) {
            if constexpr (TAB) {
                xn[v] = table_draw(cx.tab + (dg * a.Cp + static_cast<int>(chain0) + v) * 3, pair_sum<NB>(&nb[0][v], V),
                                   yv - cx.beta[v], z[v]);
            } else {
                const T P = cx.tau[v] * d + cx.isig[v];
                const T m = (cx.tau[v] * rho * s[v] + (yv - cx.beta[v]) * cx.isig[v]) * Arith<T>::rcp(P);
                xn[v] = m + z[v] * Arith<T>::rsq(P);
            }
        }
        Vec<T, V>::st(xp, xn);
    } else {
        Vec<T, V>::ld(xp, xn);
#pragma unroll
        for (int v = 0; v < V; ++v) psi[v] = 0;  // reduce-only passes are not used with this model
    }
#pragma unroll
    for (int v = 0; v < V; ++v) {
        T e = 0;
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            if ((lower_mask >> k) & 1u) {
                const T df = xn[v] - nb[k][v];
                e += wnb[k] * df * df;
            }
        }
        // (FP64 lattices, rho = 1: the first term is 0 and four of a site's operations)
        if (TAB && cx.icar) cx.accS[v] += e;
        else cx.accS[v] += (static_cast<T>(1) - rho) * (TAB ? static_cast<T>(dg) : d) * xn[v] * xn[v] + rho * e;
        if (MODEL == kModelBinomial) {
            cx.accR[v] += psi[v];
            cx.accA[v] += kappa - psi[v] * xn[v];
        } else {
            const T r = (yv - cx.beta[v]) - xn[v];
            cx.accR[v] += r * r;
            cx.accA[v] += r;
        }
    }
    if (cx.acc) {
        if (!kEarly) {
            Vec<T, V>::ld(meanp, mu);
            Vec<T, V>::ld(m2p, mm);
        }
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const T delta = xn[v] - mu[v];
            mu[v] += delta * cx.inv_k;
            mm[v] += delta * (xn[v] - mu[v]);
        }
        Vec<T, V>::st(meanp, mu);
        Vec<T, V>::st(m2p, mm);
    }
}

// Lattices with parity colourings: 2-D 4-neighbour and 3-D 6-neighbour.  Site of colour c in
// sub-array row r = l*H + i, column h sits at j = 2h + p, p = (c + l + i) & 1; its in-row
// neighbours are columns h - 1 + p and h + p of the other colour's row r, the others column h
// of rows r -+ 1 (i -+ 1) and r -+ H (l -+ 1).  Neighbour k has a fixed position in nb[k];
// missing ones (outside the lattice) are masked.
template <typename T, int V, bool THREE_D, int MODEL>
__device__ void lattice_parity_tile(const StepArgs &a, const FieldDev &f, const Tile &t, SiteCtx<T, V> &cx,
                                    int CV, int cv_shift, uint32_t sweep)
{
    constexpr int NB = THREE_D ? 6 : 4;
    const int L = THREE_D ? f.dims[0] : 1;
    const int H = THREE_D ? f.dims[1] : f.dims[0];
    const int W = THREE_D ? f.dims[2] : f.dims[1];
    const int c = t.colour;
    const int cols = f.cols;
    T *X = static_cast<T *>(a.x);
    const T *Y = static_cast<const T *>(a.y);
    T *MEAN = static_cast<T *>(a.mean);
    T *M2 = static_cast<T *>(a.m2);
    const int Cp = a.Cp;
    const int cvo = (threadIdx.x & (CV - 1)) * V;  // chain offset of this thread (fixed)
    const int64_t self_base = f.slot0 + static_cast<int64_t>(c) * f.rows * cols;
    const int64_t oth_base = f.slot0 + static_cast<int64_t>(1 - c) * f.rows * cols;
    const T *XO = X + oth_base * Cp + cvo;
    T *XS = X + self_base * Cp + cvo;
    T *MS = MEAN + self_base * Cp + cvo;
    T *QS = M2 + self_base * Cp + cvo;
    const T *YS = Y + self_base;
    const uint32_t lower_all = (c == 1) ? 0xffu : 0u;  // all neighbours have the other colour
    const int plane = H * cols;
    const int nelem = t.count * cols * CV;
    for (int e = threadIdx.x; e < nelem; e += kBlock) {
        const int cv = e & (CV - 1);
        const int sr = e >> cv_shift;
        const int rr = fast_div(sr, f.cols_m, f.cols_s);
        const int h = sr - rr * cols;
        const int r = t.start + rr;
        const int l = THREE_D ? fast_div(r, f.h_m, f.h_s) : 0;
        const int i = THREE_D ? r - l * H : r;
        const int p = (c + l + i) & 1;
        const int j = 2 * h + p;
        if (j >= W)
            continue;
        uint32_t valid = (j > 0 ? 1u : 0u) | (j + 1 < W ? 2u : 0u) | (i > 0 ? 4u : 0u) | (i + 1 < H ? 8u : 0u);
        if (THREE_D) valid |= (l > 0 ? 16u : 0u) | (l + 1 < L ? 32u : 0u);
        const int rb = r * cols + h;
        int ns[NB];
        ns[0] = rb - 1 + p;
        ns[1] = rb + p;
        ns[2] = rb - cols;
        ns[3] = rb + cols;
        if (THREE_D) {
            ns[4] = rb - plane;
            ns[5] = rb + plane;
        }
        T nb[NB][V], wnb[NB], s[V];
#pragma unroll
        for (int v = 0; v < V; ++v) s[v] = 0;
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            wnb[k] = 1;
            if ((valid >> k) & 1u) {
                Vec<T, V>::ld(XO + ns[k] * Cp, nb[k]);
            } else {
#pragma unroll
                for (int v = 0; v < V; ++v) nb[k][v] = 0;
            }
#pragma unroll
            for (int v = 0; v < V; ++v) s[v] += nb[k][v];
        }
        const uint32_t site = static_cast<uint32_t>(r * W + j);
        const int mtr = MODEL == kModelBinomial ? a.trials[self_base + rb] : 0;
        finish_site<T, V, NB, MODEL, kDegreeTable<T, kLat3D6, MODEL>>(a, cx, XS + rb * Cp, MS + rb * Cp, QS + rb * Cp, YS[rb], mtr, static_cast<T>(__popc(valid)),
                              site, sweep, f.stream, static_cast<uint32_t>(cv * V), s, nb, lower_all & valid, wnb, nullptr,
                              __popc(valid));
    }
}

// 2-D 8-neighbour lattice with the 2x2 colouring c = 2 (i & 1) + (j & 1): the site of colour
// c = 2a + b at sub-array (u, v) is (2u + a, 2v + b); neighbour (i + di, j + dj) lives in
// colour 2((a + di) & 1) + ((b + dj) & 1) at sub-array (u + ((a + di) >> 1), v + ((b + dj) >> 1)).
template <typename T, int V, int MODEL>
__device__ void lattice8_tile(const StepArgs &a, const FieldDev &f, const Tile &t, SiteCtx<T, V> &cx, int CV,
                              int cv_shift, uint32_t sweep)
{
    constexpr int NB = 8;
    const int H = f.dims[0], W = f.dims[1];
    const int c = t.colour;
    const int ca = c >> 1, cb = c & 1;
    const int cols = f.cols;
    T *X = static_cast<T *>(a.x);
    const T *Y = static_cast<const T *>(a.y);
    T *MEAN = static_cast<T *>(a.mean);
    T *M2 = static_cast<T *>(a.m2);
    const int Cp = a.Cp;
    const int cvo = (threadIdx.x & (CV - 1)) * V;  // chain offset of this thread (fixed)
    const int sub = f.rows * cols;
    const T *XF = X + f.slot0 * Cp + cvo;
    T *XS = X + (f.slot0 + static_cast<int64_t>(c) * sub) * Cp + cvo;
    T *MS = MEAN + (f.slot0 + static_cast<int64_t>(c) * sub) * Cp + cvo;
    T *QS = M2 + (f.slot0 + static_cast<int64_t>(c) * sub) * Cp + cvo;
    const T *YS = Y + f.slot0 + static_cast<int64_t>(c) * sub;
    // Per direction (block-uniform): offset of the neighbour's slot relative to (u, v) in its
    // colour's sub-array, and whether that colour is lower than c.
    int doff[NB];
    uint32_t lower = 0;
#pragma unroll
    for (int k = 0, q = 0; q < 9; ++q) {
        const int di = q / 3 - 1, dj = q % 3 - 1;
        if (di == 0 && dj == 0) continue;
        const int cc = 2 * ((ca + di) & 1) + ((cb + dj) & 1);
        doff[k] = cc * sub + ((ca + di) >> 1) * cols + ((cb + dj) >> 1);
        if (cc < c) lower |= 1u << k;
        ++k;
    }
    const int nelem = t.count * cols * CV;
    for (int e = threadIdx.x; e < nelem; e += kBlock) {
        const int cv = e & (CV - 1);
        const int sr = e >> cv_shift;
        const int rr = fast_div(sr, f.cols_m, f.cols_s);
        const int vv = sr - rr * cols;
        const int u = t.start + rr;
        const int i = 2 * u + ca, j = 2 * vv + cb;
        if (i >= H || j >= W)
            continue;
        const int base = u * cols + vv;
        uint32_t valid = 0;
#pragma unroll
        for (int k = 0, q = 0; q < 9; ++q) {
            const int di = q / 3 - 1, dj = q % 3 - 1;
            if (di == 0 && dj == 0) continue;
            const bool ok = (i + di >= 0) && (i + di < H) && (j + dj >= 0) && (j + dj < W);
            valid |= ok ? (1u << k) : 0u;
            ++k;
        }
        T nb[NB][V], wnb[NB], s[V];
#pragma unroll
        for (int v = 0; v < V; ++v) s[v] = 0;
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            wnb[k] = 1;
            if ((valid >> k) & 1u) {
                Vec<T, V>::ld(XF + (doff[k] + base) * Cp, nb[k]);
            } else {
#pragma unroll
                for (int v = 0; v < V; ++v) nb[k][v] = 0;
            }
#pragma unroll
            for (int v = 0; v < V; ++v) s[v] += nb[k][v];
        }
        const uint32_t site = static_cast<uint32_t>(i * W + j);
        const int mtr = MODEL == kModelBinomial ? a.trials[f.slot0 + static_cast<int64_t>(c) * sub + base] : 0;
        finish_site<T, V, NB, MODEL, kDegreeTable<T, kLat2D8, MODEL>>(a, cx, XS + base * Cp, MS + base * Cp, QS + base * Cp, YS[base], mtr,
                              static_cast<T>(__popc(valid)), site, sweep, f.stream, static_cast<uint32_t>(cv * V),
                              s, nb, lower & valid, wnb, nullptr, __popc(valid));
    }
}

// The neighbours of a row that stay in registers: their loads are all issued before any is used, and the
// lower-colour terms of the prior sum need no second pass over them.
template <int V> constexpr int kCsrRow = V == 4 ? 6 : 8;

// One position of a CSR field: what no kernel of a sweep writes (row, weights, degree, observation,
// site), and its normals when drawn.  A block loads its threads' first positions before it waits for the
// previous colour step (csr_ahead), so that after the wait only the neighbours' values are left to gather.
template <typename T, int V>
struct CsrSite {
    int pos, rb, re, jn[kCsrRow<V>], mtr;
    T wnb[kCsrRow<V>], yv, d, z[V];
    uint32_t site, sweep;  // sweep: of the normals
    bool drawn;
};

template <typename T, int V, int MODEL>
__device__ __forceinline__ void csr_load(const StepArgs &a, const FieldDev &f, int pos, CsrSite<T, V> &c)
{
    const int32_t *rp = a.rp + f.rp0, *ci = a.ci + f.nnz0;
    const T *wr = a.w ? static_cast<const T *>(a.w) + f.nnz0 : nullptr;
    c.pos = pos;
    c.rb = rp[pos];
    c.re = rp[pos + 1];
#pragma unroll
    for (int q = 0; q < kCsrRow<V>; ++q) {
        const int k = c.rb + q;
        c.jn[q] = k < c.re ? ci[k] : -1;
        c.wnb[q] = k < c.re ? (wr ? wr[k] : static_cast<T>(1)) : static_cast<T>(0);
    }
    c.yv = static_cast<const T *>(a.y)[f.slot0 + pos];
    c.d = static_cast<const T *>(a.deg)[f.csr0 + pos];
    c.site = static_cast<uint32_t>(a.perm[f.csr0 + pos]);
    c.mtr = MODEL == kModelBinomial ? a.trials[f.slot0 + pos] : 0;
    c.drawn = false;
}

// The thread's first position, before the dependency wait (pos < 0: none).  From colour 1 on the
// normals too: the previous launch is a colour step of the same sweep, which let this one start after
// its own wait, so everything before it, the draws that advanced the sweep number included, is complete
// (csr_tile checks the number all the same: a stage launched alone may follow another kernel).
template <typename T, int V, int MODEL>
__device__ __forceinline__ void csr_ahead(const StepArgs &a, const FieldDev &f, const Tile &t, CsrSite<T, V> &c)
{
    const int CV = a.Cp / V, e = threadIdx.x;
    c.pos = -1;
    if (e >= t.count * CV) return;
    csr_load<T, V, MODEL>(a, f, t.start + e / CV, c);
    if (a.update && t.colour > 0) {
        c.sweep = static_cast<uint32_t>(*reinterpret_cast<volatile const long long *>(&a.ctl->sweep));
        site_normals<T, V>(a.key, c.site, c.sweep, f.stream, static_cast<uint32_t>((e % CV) * V), a.lanes, c.z);
        c.drawn = true;
    }
}

// CSR field: permuted positions [start, start + count) of one colour class; neighbours are read
// through the permuted row; a neighbour has lower colour iff its position is below the class's
// first position.
template <typename T, int V, int MODEL>
__device__ void csr_tile(const StepArgs &a, const FieldDev &f, const Tile &t, SiteCtx<T, V> &cx, int CV,
                         int cv_shift, uint32_t sweep, CsrSite<T, V> &c)
{
    T *X = static_cast<T *>(a.x);
    T *MEAN = static_cast<T *>(a.mean);
    T *M2 = static_cast<T *>(a.m2);
    const T *Wt = static_cast<const T *>(a.w);
    const int64_t Cp = a.Cp;
    const int32_t *ci = a.ci + f.nnz0;
    const T *wr = Wt ? Wt + f.nnz0 : nullptr;
    const int32_t lo = a.coff[f.coff0 + t.colour];
    const T rho = static_cast<T>(a.rho);
    const int nelem = t.count * CV;
    constexpr int R = kCsrRow<V>;
    for (int e = threadIdx.x; e < nelem; e += kBlock) {
        const int cv = e & (CV - 1);
        if (e != static_cast<int>(threadIdx.x)) csr_load<T, V, MODEL>(a, f, t.start + (e >> cv_shift), c);
        const int pos = c.pos, rb = c.rb, re = c.re;
        T nb[R][V], s[V];
        uint32_t lower = 0;
#pragma unroll
        for (int v = 0; v < V; ++v) s[v] = 0;
#pragma unroll
        for (int q = 0; q < R; ++q) {
            if (c.jn[q] >= 0) {
                Vec<T, V>::ld(X + (f.slot0 + c.jn[q]) * Cp + cv * V, nb[q]);
                lower |= (c.jn[q] < lo ? 1u : 0u) << q;
            } else {
#pragma unroll
                for (int v = 0; v < V; ++v) nb[q][v] = 0;
            }
#pragma unroll
            for (int v = 0; v < V; ++v) s[v] += c.wnb[q] * nb[q][v];
        }
        for (int k = rb + R; k < re; ++k) {  // rows longer than R
            T xv[V];
            Vec<T, V>::ld(X + (f.slot0 + ci[k]) * Cp + cv * V, xv);
            const T wv = wr ? wr[k] : static_cast<T>(1);
#pragma unroll
            for (int v = 0; v < V; ++v) s[v] += wv * xv[v];
        }
        const int64_t self = f.slot0 + pos;
        finish_site<T, V, R, MODEL>(a, cx, X + self * Cp + cv * V, MEAN + self * Cp + cv * V, M2 + self * Cp + cv * V, c.yv,
                                    c.mtr, c.d, c.site, sweep, f.stream, static_cast<uint32_t>(cv * V), s, nb, lower, c.wnb,
                                    c.drawn && c.sweep == sweep ? c.z : nullptr);
        if (re - rb > R) {
            // the lower-colour edges beyond the first R
            T xn[V], e2[V];
            Vec<T, V>::ld(X + self * Cp + cv * V, xn);
#pragma unroll
            for (int v = 0; v < V; ++v) e2[v] = 0;
            for (int k = rb + R; k < re; ++k) {
                const int jn = ci[k];
                if (jn >= lo) continue;
                T xv[V];
                Vec<T, V>::ld(X + (f.slot0 + jn) * Cp + cv * V, xv);
                const T wv = wr ? wr[k] : static_cast<T>(1);
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    const T df = xn[v] - xv[v];
                    e2[v] += wv * df * df;
                }
            }
#pragma unroll
            for (int v = 0; v < V; ++v) cx.accS[v] += rho * e2[v];
        }
    }
}

// MODEL: the observation model; without the intercept beta0 = 0 and the third sum is not
// needed, which the compiler then removes, registers included.
// FP64: two blocks per SM (128 registers), or a class of more tiles than SMs runs in two waves (48^3, two chains,
// 231 tiles: 44 us per sweep against 38).
template <typename T, int V, int KIND, int MODEL>
__global__ void __launch_bounds__(kBlock, sizeof(T) == 4 ? (KIND == kCsr ? 2 : 3) : 2) colour_step_kernel(const StepArgs a)
{
    // Tiles and fields are never written by a sweep: read before the dependency wait.
    const Tile t = a.tiles[blockIdx.x];
    const FieldDev f = a.fields[t.field];
    CsrSite<T, V> ahead;
    if constexpr (KIND == kCsr) csr_ahead<T, V, MODEL>(a, f, t, ahead);
    pdl_wait_then_release();
    const int CV = a.Cp / V;
    const int cv = threadIdx.x % CV;  // fixed per thread: kBlock is a multiple of CV
    const long long sweep_ll = a.ctl->sweep;
    const uint32_t sweep = static_cast<uint32_t>(sweep_ll);

    SiteCtx<T, V> cx;
    const T *hyp = static_cast<const T *>(a.hyp);
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const int64_t hc = (static_cast<int64_t>(t.field) * a.Cp + cv * V + v) * kHypStride;
        cx.tau[v] = hyp[hc];
        cx.isig[v] = hyp[hc + 1];
        cx.beta[v] = MODEL != kModelGauss ? hyp[hc + 2] : static_cast<T>(0);
        cx.accS[v] = 0;
        cx.accR[v] = 0;
        cx.accA[v] = 0;
    }
    cx.acc = false;
    cx.inv_k = 0;
    constexpr bool kTab = kDegreeTable<T, KIND, MODEL>;
    if (a.update && a.acc_enabled && sweep_accumulated(sweep_ll, a.burn_in, a.thin)) {
        cx.acc = true;
        if (!kTab) cx.inv_k = static_cast<T>(1) / static_cast<T>(a.ctl->acc_count + 1);
    }

    __shared__ T tab[kTab ? 9 * kMaxChains * 3 : 1], s_inv_k;
    cx.tab = tab;
    cx.icar = a.rho == 1.0;
    if constexpr (kTab) {
        degree_table(tab, s_inv_k, hyp + static_cast<int64_t>(t.field) * a.Cp * kHypStride, a.Cp, a.rho, cx.acc, a.ctl);
        __syncthreads();
        cx.inv_k = s_inv_k;
    }

    const int cv_shift = __ffs(CV) - 1;
    if constexpr (KIND == kLat2D4) lattice_parity_tile<T, V, false, MODEL>(a, f, t, cx, CV, cv_shift, sweep);
    else if constexpr (KIND == kLat3D6) lattice_parity_tile<T, V, true, MODEL>(a, f, t, cx, CV, cv_shift, sweep);
    else if constexpr (KIND == kLat2D8) lattice8_tile<T, V, MODEL>(a, f, t, cx, CV, cv_shift, sweep);
    else csr_tile<T, V, MODEL>(a, f, t, cx, CV, cv_shift, sweep, ahead);

    // Deterministic block reduction of the 3 V partial sums of each chain in the state precision:
    // a shuffle tree over the lanes that share a chain vector (lanes equal mod CV), then the
    // warps' sums in order; the tile's sum is stored in FP64 and summed over tiles in FP64.
    __shared__ T red[kBlock / 32][kMaxChains][3];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int v = 0; v < V; ++v) {
        T sS = cx.accS[v];
        T sR = cx.accR[v];
        T sA = MODEL != kModelGauss ? cx.accA[v] : static_cast<T>(0);
        if constexpr (kTab) {
            if (CV <= 16) {
                sS = warp_sum_pair(sS, sR, CV);
                sR = __shfl_xor_sync(0xffffffffu, sS, 16);
            }
            for (int off = 16; off >= CV && MODEL != kModelGauss; off >>= 1) sA += __shfl_xor_sync(0xffffffffu, sA, off);
        } else {
            for (int off = 16; off >= CV; off >>= 1) {
                sS += __shfl_xor_sync(0xffffffffu, sS, off);
                sR += __shfl_xor_sync(0xffffffffu, sR, off);
                if (MODEL != kModelGauss) sA += __shfl_xor_sync(0xffffffffu, sA, off);
            }
        }
        if (lane < CV) {
            red[warp][lane * V + v][0] = sS;
            red[warp][lane * V + v][1] = sR;
            red[warp][lane * V + v][2] = sA;
        }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < a.Cp * 3; q += kBlock) {
        const int chain = q / 3, k = q - 3 * chain;
        T acc = 0;
        if constexpr (kTab) acc = pair_sum<kBlock / 32>(&red[0][chain][k], kMaxChains * 3);
        else
            for (int w = 0; w < kBlock / 32; ++w) acc += red[w][chain][k];
        double *dst = reinterpret_cast<double *>(a.partials + static_cast<int64_t>(t.part) * a.Cp + chain);
        dst[k] = static_cast<double>(acc);
    }
}

// The hyperparameter stage for fields of fewer than 256 tiles: one warp per task of hyper_task
// (eight per block).  With a single block its thread 0 advances the counters after a barrier; with
// several, the last block to finish does (ticket counter; no block waits for another).
constexpr int kHyperWarps = 8;

__device__ __forceinline__ void hyper_end(const HyperArgs &a, long long sweep)
{
    bool last = gridDim.x == 1;
    __syncthreads();
    if (!last && threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(&a.ctl->ticket, 1ull) == gridDim.x - 1;
    }
    if (threadIdx.x == 0 && last) {
        hyper_advance(a, sweep);
        a.ctl->ticket = 0;
    }
}

template <typename T>
__global__ void __launch_bounds__(kHyperWarps * 32) hyper_kernel(const HyperArgs a)
{
    // Let the next sweep kernel be scheduled now: it does its own early work (observations,
    // predicted normals) while this draw waits for and runs after the current sweep.
    pdl_release();
    pdl_wait();
    const int task = blockIdx.x * kHyperWarps + (threadIdx.x >> 5);
    const long long sweep = a.ctl->sweep;
    if (task < a.nfields * a.Cp * 2) hyper_task<T>(a, task, sweep);
    hyper_end(a, sweep);
}

// The same for fields of 256 tiles or more: one block per task, its warps taking a row of the
// partials each (the order of hyper_sums).  A launch is bound by latency: one warp per task waits
// for an L2 round trip and eight dependent FP64 additions per 256 partials; with a block per task
// every partial of up to 256 is loaded at once: 1222 partials of 4
// chains 19.1 -> 9.6 us, 1240 of one chain 15.1 -> 9.2 us, 608 of 8 chains 13.4 -> 7.1 us (alone,
// cold).
template <typename T>
__global__ void __launch_bounds__(kSumRows * 32) hyper_wide_kernel(const HyperArgs a)
{
    __shared__ double rs[kSumRows][32], ra[kSumRows][32];
    pdl_release();
    pdl_wait();
    const long long sweep = a.ctl->sweep;
    const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
    const HyperCtx c = hyper_ctx<T>(a, blockIdx.x, sweep, threadIdx.x == 0);
    double S = 0.0, A = 0.0;
    if (c.need_sum) {
        const int nparts = a.fields[c.fi].nparts;
        const Part3 *P = a.partials + static_cast<int64_t>(a.fields[c.fi].part0) * a.Cp + c.chain;
        constexpr int U = 4;  // loads in flight per thread
        for (int k0 = threadIdx.x; k0 < nparts; k0 += U * kSumRows * 32) {
            double vs[U], va[U];
#pragma unroll
            for (int j = 0; j < U; ++j) {
                const int k = k0 + j * kSumRows * 32;
                vs[j] = 0.0;
                va[j] = 0.0;
                if (k < nparts)
                    part_values<false>(P + static_cast<int64_t>(k) * a.Cp, c.which, c.need_a, vs[j], va[j]);
            }
#pragma unroll
            for (int j = 0; j < U; ++j) {
                S += vs[j];
                if (c.need_a) A += va[j];
            }
        }
        rs[row][lane] = S;
        ra[row][lane] = A;
        __syncthreads();
        if (row == 0) {
            S = 0.0;
            A = 0.0;
#pragma unroll
            for (int j = 0; j < kSumRows; ++j) {
                S += rs[j][lane];
                if (c.need_a) A += ra[j][lane];
            }
            S = lane_tree(S);
            if (c.need_a) A = lane_tree(A);
        }
    }
    if (threadIdx.x == 0) hyper_finish<T>(a, c, sweep, S, A);
    hyper_end(a, sweep);
}

// The Polya-Gamma stage of the binomial model: psi of (slot, chain) is the sum of m_i draws of
// PG(1, c); psi = 0 for sites without trials and for padding slots.  A block takes kPgSlots (slot,
// chain) pairs and spreads their draws over its threads in one sequence, so that a warp's lanes are
// full whatever the m_i (with a warp per pair half the lanes had no draw, and the proposal's mixture
// weight, a dozen special functions, was computed by one lane of each warp; here by one thread per
// pair).  A pair's draws are added in a fixed order that does not depend on the block: draw k into
// lane k mod 32 in turn, then a shuffle tree over the lanes.  Bound by the instructions of the
// rejection loops and their divergence (16 of 32 lanes active, 49 % issue): 14,926 sites with 226,000
// draws 34 -> 22 us.
constexpr int kPgSlots = 32, kPgThreads = 256, kPgPass = 1024;  // kPgPass: draws between barriers

// Natural site of a slot of field f (rel: relative to the field), -1 for the padding of a lattice layout.
__device__ __forceinline__ int64_t site_of_slot(const PgArgs &a, const FieldDev &f, int64_t rel)
{
    if (f.kind == kCsr) return a.perm[f.csr0 + rel];
    const int64_t sub = static_cast<int64_t>(f.rows) * f.cols;
    const int64_t c = rel / sub, r = (rel - c * sub) / f.cols, h = rel - c * sub - r * f.cols;
    if (f.kind == kLat2D8) {
        const int64_t i = 2 * r + (c >> 1), j = 2 * h + (c & 1);
        return (i < f.dims[0] && j < f.dims[1]) ? i * f.dims[1] + j : -1;
    }
    if (f.kind == kLat2D4) {
        const int64_t j = 2 * h + ((c + r) & 1);
        return j < f.dims[1] ? r * f.dims[1] + j : -1;
    }
    const int64_t l = r / f.dims[1], i = r - l * f.dims[1], j = 2 * h + ((c + l + i) & 1);
    return j < f.dims[2] ? r * f.dims[2] + j : -1;
}

template <typename T>
__global__ void __launch_bounds__(kPgThreads) pg_stage_kernel(const PgArgs a)
{
    __shared__ T s_z[kPgSlots], s_w[kPgSlots], s_val[kPgPass], s_acc[kPgSlots][32];
    __shared__ int s_end[kPgSlots];  // draws of the block's pairs up to and with this one
    __shared__ uint32_t s_site[kPgSlots], s_chain[kPgSlots], s_stream[kPgSlots];
    pdl_wait_then_release();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t sweep = static_cast<uint32_t>(a.ctl->sweep);
    const T *X = static_cast<const T *>(a.x);
    const T *hyp = static_cast<const T *>(a.hyp);
    T *PSI = static_cast<T *>(a.psi);
    const int64_t tasks = a.slots * a.C;
    int fb = 0;
    for (int64_t first = static_cast<int64_t>(blockIdx.x) * kPgSlots; first < tasks;
         first += static_cast<int64_t>(gridDim.x) * kPgSlots) {
        for (int q = tid; q < kPgSlots * 32; q += kPgThreads) s_acc[q >> 5][q & 31] = 0;
        if (warp == 0) {
            static_assert(kPgSlots == 32, "a pair per lane of the first warp");
            const int64_t task = first + lane;
            int m = 0;
            if (task < tasks) {
                const int64_t slot = task / a.C;
                const int chain = static_cast<int>(task - slot * a.C);
                int fi = 0;  // field of the slot (fields are few; their slot ranges are in order)
                while (fi + 1 < a.nfields && a.fields[fi + 1].slot0 <= slot) ++fi;
                const FieldDev &f = a.fields[fi];
                const int64_t site = site_of_slot(a, f, slot - f.slot0);
                m = site >= 0 ? a.trials[slot] : 0;
                if (m > 0) {
                    const T eta = hyp[(static_cast<int64_t>(fi) * a.Cp + chain) * kHypStride + 2] + X[slot * a.Cp + chain];
                    // the sampler's arithmetic follows the state precision (pg.cuh)
                    const T z = static_cast<T>(0.5) * fabs(eta);
                    s_z[lane] = z;
                    s_w[lane] = pg_exp_weight<T>(z);
                    s_site[lane] = static_cast<uint32_t>(site);
                    s_chain[lane] = static_cast<uint32_t>(chain);
                    s_stream[lane] = f.stream;
                }
            }
            int end = m;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, end, o);
                if (lane >= o) end += v;
            }
            s_end[lane] = end;
        }
        __syncthreads();
        const int total = s_end[kPgSlots - 1];
        auto pair_of = [&](int q) {  // the first pair that ends beyond draw q
            int p = 0;
#pragma unroll
            for (int o = kPgSlots / 2; o >= 1; o >>= 1)
                if (s_end[p + o - 1] <= q) p += o;
            return p;
        };
        for (int q0 = 0; q0 < total; q0 += kPgPass) {
            const int q1 = min(total, q0 + kPgPass);
            for (int q = q0 + tid; q < q1; q += kPgThreads) {
                const int p = pair_of(q), start = p > 0 ? s_end[p - 1] : 0;
                PgStream st;
                pg_stream_init(st, a.key, s_site[p], sweep, s_stream[p], s_chain[p], static_cast<uint32_t>(q - start));
                const T z = s_z[p];
                T j = pg_jstar<T>(z, s_w[p], st);
                if (j < static_cast<T>(0)) {
                    ++fb;
                    j = z > static_cast<T>(0) ? tanh(z) / z : static_cast<T>(1);
                }
                s_val[q - q0] = static_cast<T>(0.25) * j;
            }
            __syncthreads();
            // the pass's draws into the pairs' lanes, by the thread of a lane's first draw in the pass
            for (int q = q0 + tid; q < q1; q += kPgThreads) {
                const int p = pair_of(q), start = p > 0 ? s_end[p - 1] : 0;
                if (q - max(start, q0) >= 32) continue;
                const int end = min(s_end[p], q1);
                T acc = s_acc[p][(q - start) & 31];
                for (int k = q; k < end; k += 32) acc += s_val[k - q0];
                s_acc[p][(q - start) & 31] = acc;
            }
            __syncthreads();
        }
        for (int p = warp; p < kPgSlots; p += kPgThreads / 32) {
            T sum = s_acc[p][lane];
            for (int off = 16; off >= 1; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
            if (lane == 0 && first + p < tasks) {
                const int64_t slot = (first + p) / a.C;
                PSI[slot * a.Cp + (first + p - slot * a.C)] = sum;
            }
        }
        __syncthreads();
    }
    if (fb) atomicAdd(reinterpret_cast<unsigned long long *>(&a.ctl->fallbacks), static_cast<unsigned long long>(fb));
}

// Natural order -> colour-split layout: y and the chains' initial states (x0 = y by default;
// chains >= C of the padded layout start at y too).
template <typename T>
__global__ void pack_kernel(const FieldDev *fields, int32_t fidx, int32_t C, int32_t Cp, const double *y_nat,
                            const double *x0_nat, const int32_t *perm_inv, T *x, T *y)
{
    const FieldDev f = fields[fidx];
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < f.n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t slot = f.slot0 + (f.kind == kCsr ? perm_inv[f.csr0 + i] : lattice_slot_of_site(f, i));
        const double yv = y_nat[i];
        y[slot] = static_cast<T>(yv);
        for (int c = 0; c < Cp; ++c)
            x[slot * Cp + c] = static_cast<T>((x0_nat && c < C) ? x0_nat[static_cast<int64_t>(c) * f.n + i] : yv);
    }
}

// Natural order -> colour-split layout of a per-site integer array (binomial trials).
__global__ void pack_int_kernel(const FieldDev *fields, int32_t fidx, const int32_t *v_nat, const int32_t *perm_inv,
                                int32_t *v)
{
    const FieldDev f = fields[fidx];
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < f.n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t slot = f.slot0 + (f.kind == kCsr ? perm_inv[f.csr0 + i] : lattice_slot_of_site(f, i));
        v[slot] = v_nat[i];
    }
}

// Colour-split layout -> natural order for one chain: out[i] = src (or m2 * inv_km1).
template <typename T>
__global__ void unpack_kernel(const FieldDev *fields, int32_t fidx, int32_t Cp, int32_t chain, const T *src,
                              const T *m2, double inv_km1, const int32_t *perm_inv, double *out)
{
    const FieldDev f = fields[fidx];
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < f.n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t slot = f.slot0 + (f.kind == kCsr ? perm_inv[f.csr0 + i] : lattice_slot_of_site(f, i));
        if (m2) out[i] = static_cast<double>(m2[slot * Cp + chain]) * inv_km1;
        else out[i] = static_cast<double>(src[slot * Cp + chain]);
    }
}

// a / d for the divisor d that a launch shares (r = 1 / d): a quotient estimate and one residual
// correction (Markstein, IBM J. Res. Dev. 1990), three FP64 operations where a division takes an
// order of magnitude more of the FP64 pipe; quotients that are not finite take the division.
struct Divisor {
    double d, r;
};
__device__ __forceinline__ double divide(double a, const Divisor &v)
{
    const double q = a * v.r;
    return isfinite(q) ? fma(fma(-q, v.d, a), v.r, q) : a / v.d;
}

// Running moments pooled over the C chains of one field, natural order, FP64: mean = the chains'
// means averaged; var = the sum over chains of M2_c + k (mean_c - mean)^2, over C k - 1 (the
// variance of all C k draws); 0 and NaN where k accumulated draws per chain are too few.  CP: the layout's chains when
// 1, 2, 4 or 8 (a site's values are loaded as vectors and kept in registers), else 0.
//
// Bound by the FP64 pipe (measured: about one lane per clock and SM): four FP64 operations per
// chain and site (the mean's sum, the difference, its square, M2's sum) and three per quotient.
// With divisions, a second load and conversion of the means, and k inside the sum, a 256^3 field
// of 8 chains took 2490 us and one chain of 2047 x 1931 sites 183 us, now 1800 and 87 us (moving
// the conversions to integer operations changed nothing).
template <typename T, int CP>
__global__ void __launch_bounds__(256) pool_kernel(const FieldDev *fields, int32_t fidx, int32_t Cp_, int32_t C,
                                                   const SweepCtl *ctl, const T *mean, const T *m2, const int32_t *perm_inv,
                                                   double *out_mean, double *out_var)
{
    const FieldDev f = fields[fidx];
    const int Cp = CP ? CP : Cp_;
    constexpr int V = CP == 0 ? 1 : (sizeof(T) == 8 ? (CP < 2 ? CP : 2) : (CP < 4 ? CP : 4));
    constexpr int NR = CP ? CP : 1;
    const int64_t k = ctl->acc_count;
    const double kd = static_cast<double>(k);
    const Divisor by_c{static_cast<double>(C), 1.0 / static_cast<double>(C)};
    const double dof = static_cast<double>(C * k - 1);
    const Divisor by_dof{dof, 1.0 / dof};
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < f.n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t slot = f.slot0 + (f.kind == kCsr ? perm_inv[f.csr0 + i] : lattice_slot_of_site(f, i));
        const T *mp = mean + slot * Cp, *qp = m2 + slot * Cp;
        T mr[NR], qr[NR];
        if constexpr (CP > 0) {
#pragma unroll
            for (int c = 0; c < CP; c += V) Vec<T, V>::ld(mp + c, reinterpret_cast<T(&)[V]>(mr[c]));
            if (out_var) {
#pragma unroll
                for (int c = 0; c < CP; c += V) Vec<T, V>::ld(qp + c, reinterpret_cast<T(&)[V]>(qr[c]));
            }
        }
        double mu = 0.0, ss = 0.0, dd = 0.0;
        if constexpr (CP > 0) {
            double md[NR];
#pragma unroll
            for (int c = 0; c < CP; ++c) {
                md[c] = static_cast<double>(mr[c]);
                if (c < C) mu += md[c];
            }
            if (CP > 1) mu = divide(mu, by_c);
            if (out_var) {
#pragma unroll
                for (int c = 0; c < CP; ++c)
                    if (c < C) {
                        const double d = md[c] - mu;
                        if (CP > 1) dd = fma(d, d, dd);
                        ss += static_cast<double>(qr[c]);
                    }
            }
        } else {
            for (int c = 0; c < C; ++c) mu += static_cast<double>(mp[c]);
            mu = divide(mu, by_c);
            if (out_var)
                for (int c = 0; c < C; ++c) {
                    const double d = static_cast<double>(mp[c]) - mu;
                    dd = fma(d, d, dd);
                    ss += static_cast<double>(qp[c]);
                }
        }
        if (out_mean) out_mean[i] = k < 1 ? 0.0 : mu;
        if (out_var) out_var[i] = C * k < 2 ? __longlong_as_double(0x7ff8000000000000ll) : divide(fma(kd, dd, ss), by_dof);
    }
}

__global__ void philox_words_kernel(uint2 key, uint32_t c1, uint32_t c2, uint32_t c3, int64_t count, uint4 *out)
{
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < count;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        out[i] = philox4x32_10(make_uint4(static_cast<uint32_t>(i), c1, c2, c3), key);
}

template <typename T>
__global__ void site_normals_kernel(uint2 key, uint32_t sweep, uint32_t stream, uint32_t chain, int lanes,
                                    int64_t count, T *out)
{
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < count;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        T z[1];
        site_normals<T, 1>(key, static_cast<uint32_t>(i), sweep, stream, chain, lanes, z);
        out[i] = z[0];
    }
}

// One thread per (sweep of the batch, field, chain, variate): the unit-rate Marsaglia-Tsang
// variates of tau and 1/sigma^2 and the intercept's standard normal, with the counters of that
// sweep's draws.  They are independent of the state, so a whole batch runs in parallel and the
// per-sweep draw reduces to a division by the rate (and a shift for the intercept).
__global__ void gamma_pre_kernel(const GammaPreArgs a)
{
    pdl_wait_then_release();
    const long long base = a.ctl->sweep;
    const int total = gamma_pre_tasks(a);
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < total; q += gridDim.x * blockDim.x) gamma_pre_task(a, q, base);
    if (blockIdx.x == 0 && threadIdx.x == 0) gamma_pre_record(a, base);
}

__global__ void ctl_reset_kernel(SweepCtl *ctl, long long start_sweep)
{
    SweepCtl c{};
    c.sweep = start_sweep;
    c.fnext = start_sweep;
    *ctl = c;
}

int grid_for(int64_t n, int block)
{
    int64_t g = (n + block - 1) / block;
    if (g < 1) g = 1;
    if (g > 152 * 32) g = 152 * 32;
    return static_cast<int>(g);
}

}  // namespace

template <int KIND, int MODEL>
cudaError_t launch_model(int precision, int V, const StepArgs &a, cudaStream_t stream)
{
    const dim3 grid(a.ntiles), block(kBlock);
    if (precision == 0) {
        if (V == 4) return launch_sweep_kernel(colour_step_kernel<float, 4, KIND, MODEL>, grid, block, 0, stream, a);
        if (V == 2) return launch_sweep_kernel(colour_step_kernel<float, 2, KIND, MODEL>, grid, block, 0, stream, a);
        return launch_sweep_kernel(colour_step_kernel<float, 1, KIND, MODEL>, grid, block, 0, stream, a);
    }
    if (V == 2) return launch_sweep_kernel(colour_step_kernel<double, 2, KIND, MODEL>, grid, block, 0, stream, a);
    return launch_sweep_kernel(colour_step_kernel<double, 1, KIND, MODEL>, grid, block, 0, stream, a);
}

template <int KIND>
cudaError_t launch_kind(int precision, int V, const StepArgs &a, cudaStream_t stream)
{
    if (a.binomial) return launch_model<KIND, kModelBinomial>(precision, V, a, stream);
    if (a.intercept) return launch_model<KIND, kModelGaussIntercept>(precision, V, a, stream);
    return launch_model<KIND, kModelGauss>(precision, V, a, stream);
}

cudaError_t launch_colour_step(int precision, int V, int kind, const StepArgs &a, cudaStream_t stream)
{
    if (a.ntiles <= 0) return cudaSuccess;
    switch (kind) {
    case kLat2D4: return launch_kind<kLat2D4>(precision, V, a, stream);
    case kLat2D8: return launch_kind<kLat2D8>(precision, V, a, stream);
    case kLat3D6: return launch_kind<kLat3D6>(precision, V, a, stream);
    default: return launch_kind<kCsr>(precision, V, a, stream);
    }
}

cudaError_t launch_hyper(int precision, const HyperArgs &a, cudaStream_t stream)
{
    if (a.max_parts >= 32 * kSumRows) {
        const int tasks = a.nfields * a.Cp * 2;
        if (precision == 0) return launch_sweep_kernel(hyper_wide_kernel<float>, tasks, kSumRows * 32, 0, stream, a);
        return launch_sweep_kernel(hyper_wide_kernel<double>, tasks, kSumRows * 32, 0, stream, a);
    }
    const int grid = (a.nfields * a.Cp * 2 + kHyperWarps - 1) / kHyperWarps;
    if (precision == 0) return launch_sweep_kernel(hyper_kernel<float>, grid, kHyperWarps * 32, 0, stream, a);
    return launch_sweep_kernel(hyper_kernel<double>, grid, kHyperWarps * 32, 0, stream, a);
}

cudaError_t launch_pack(int precision, const FieldDev *fields_dev, const FieldDev &f, int32_t fidx, int32_t C,
                        int32_t Cp, const double *y_nat, const double *x0_nat, const int32_t *perm_inv, void *x,
                        void *y, cudaStream_t stream)
{
    const int grid = grid_for(f.n, 256);
    if (precision == 0)
        pack_kernel<float><<<grid, 256, 0, stream>>>(fields_dev, fidx, C, Cp, y_nat, x0_nat, perm_inv,
                                                     static_cast<float *>(x), static_cast<float *>(y));
    else
        pack_kernel<double><<<grid, 256, 0, stream>>>(fields_dev, fidx, C, Cp, y_nat, x0_nat, perm_inv,
                                                      static_cast<double *>(x), static_cast<double *>(y));
    return cudaGetLastError();
}

cudaError_t launch_pg_stage(int precision, const PgArgs &a, cudaStream_t stream)
{
    const int64_t tasks = a.slots * a.C;
    int64_t blocks = (tasks + kPgSlots - 1) / kPgSlots;
    if (blocks > 152 * 64) blocks = 152 * 64;
    if (blocks < 1) blocks = 1;
    if (precision == 0) return launch_sweep_kernel(pg_stage_kernel<float>, static_cast<int>(blocks), kPgThreads, 0, stream, a);
    return launch_sweep_kernel(pg_stage_kernel<double>, static_cast<int>(blocks), kPgThreads, 0, stream, a);
}

namespace {

// The checks of data uploaded for gmrf_sampler_set_data, on the device: bit 0 of *flag when a y
// is not finite, bit 1 a trials count outside 0..4095, bit 2 a success count outside
// [0, trials], bit 3 an x0 not finite (x0 may be null; trials null unless binomial).
__global__ void check_data_kernel(const double *y, const int32_t *trials, const double *x0, int64_t n, int64_t nx0,
                                  unsigned int *flag)
{
    unsigned int bad = 0;
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n; i += stride) {
        const double v = y[i];
        if (!isfinite(v)) bad |= 1u;
        if (trials) {
            const int32_t m = trials[i];
            if (m < 0 || m > 4095) bad |= 2u;
            if (!(v >= 0.0 && v <= static_cast<double>(m))) bad |= 4u;
        }
    }
    if (x0)
        for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < nx0; i += stride)
            if (!isfinite(x0[i])) bad |= 8u;
    bad = __reduce_or_sync(0xffffffffu, bad);
    if (bad && (threadIdx.x & 31) == 0) atomicOr(flag, bad);
}

}  // namespace

cudaError_t launch_check_data(const double *y, const int32_t *trials, const double *x0, int64_t n, int64_t nx0,
                              unsigned int *flag, cudaStream_t stream)
{
    check_data_kernel<<<grid_for(n > nx0 ? n : nx0, 256), 256, 0, stream>>>(y, trials, x0, n, nx0, flag);
    return cudaGetLastError();
}

cudaError_t launch_pack_int(const FieldDev *fields_dev, const FieldDev &f, int32_t fidx, const int32_t *v_nat,
                            const int32_t *perm_inv, int32_t *v, cudaStream_t stream)
{
    pack_int_kernel<<<grid_for(f.n, 256), 256, 0, stream>>>(fields_dev, fidx, v_nat, perm_inv, v);
    return cudaGetLastError();
}

cudaError_t launch_unpack(int precision, const FieldDev *fields_dev, const FieldDev &f, int32_t fidx, int32_t Cp,
                          int32_t chain, const void *src, const void *m2, double inv_km1, const int32_t *perm_inv,
                          double *out, cudaStream_t stream)
{
    const int grid = grid_for(f.n, 256);
    if (precision == 0)
        unpack_kernel<float><<<grid, 256, 0, stream>>>(fields_dev, fidx, Cp, chain, static_cast<const float *>(src),
                                                       static_cast<const float *>(m2), inv_km1, perm_inv, out);
    else
        unpack_kernel<double><<<grid, 256, 0, stream>>>(fields_dev, fidx, Cp, chain, static_cast<const double *>(src),
                                                        static_cast<const double *>(m2), inv_km1, perm_inv, out);
    return cudaGetLastError();
}

cudaError_t launch_pool(int precision, const FieldDev *fields_dev, const FieldDev &f, int32_t fidx, int32_t Cp,
                        int32_t C, const SweepCtl *ctl, const void *mean, const void *m2, const int32_t *perm_inv,
                        double *out_mean, double *out_var, cudaStream_t stream)
{
    const int grid = grid_for(f.n, 256);
    auto go = [&](auto *kernel, auto *me, auto *q) {
        kernel<<<grid, 256, 0, stream>>>(fields_dev, fidx, Cp, C, ctl, me, q, perm_inv, out_mean, out_var);
    };
    auto pick = [&](auto *me, auto *q) {
        using T = std::remove_cv_t<std::remove_pointer_t<decltype(me)>>;
        switch (Cp) {
        case 1: return go(pool_kernel<T, 1>, me, q);
        case 2: return go(pool_kernel<T, 2>, me, q);
        case 4: return go(pool_kernel<T, 4>, me, q);
        case 8: return go(pool_kernel<T, 8>, me, q);
        default: return go(pool_kernel<T, 0>, me, q);
        }
    };
    if (precision == 0) pick(static_cast<const float *>(mean), static_cast<const float *>(m2));
    else pick(static_cast<const double *>(mean), static_cast<const double *>(m2));
    return cudaGetLastError();
}

cudaError_t launch_gamma_pre(const GammaPreArgs &a, cudaStream_t stream)
{
    const int total = a.count * a.nfields * a.Cp * 4;
    if (total <= 0) return cudaSuccess;
    return launch_sweep_kernel(gamma_pre_kernel, (total + 127) / 128, 128, 0, stream, a);
}

cudaError_t launch_ctl_reset(SweepCtl *ctl, long long start_sweep, cudaStream_t stream)
{
    ctl_reset_kernel<<<1, 1, 0, stream>>>(ctl, start_sweep);
    return cudaGetLastError();
}

cudaError_t launch_philox_words(uint64_t seed, uint32_t c1, uint32_t c2, uint32_t c3, int64_t count, uint32_t *out,
                                cudaStream_t stream)
{
    if (count <= 0) return cudaSuccess;
    philox_words_kernel<<<grid_for(count, 256), 256, 0, stream>>>(philox_key(seed), c1, c2, c3, count,
                                                                   reinterpret_cast<uint4 *>(out));
    return cudaGetLastError();
}

cudaError_t launch_site_normals(uint64_t seed, uint32_t sweep, uint32_t stream_id, uint32_t chain, int lanes,
                                int precision, int64_t count, void *out, cudaStream_t stream)
{
    if (count <= 0) return cudaSuccess;
    if (precision == 0)
        site_normals_kernel<float><<<grid_for(count, 256), 256, 0, stream>>>(philox_key(seed), sweep, stream_id, chain,
                                                                            lanes, count, static_cast<float *>(out));
    else
        site_normals_kernel<double><<<grid_for(count, 256), 256, 0, stream>>>(philox_key(seed), sweep, stream_id, chain,
                                                                             lanes, count, static_cast<double *>(out));
    return cudaGetLastError();
}

}  // namespace gmrf
