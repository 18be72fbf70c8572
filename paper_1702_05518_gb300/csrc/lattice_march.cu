// lattice_march.cu -- sweeps of FP32 2-D lattice fields (both neighbourhoods) by marching warps: all
// colour steps of Algorithm 1 in one pass over the rows, with the state in registers.
//
// A warp owns a strip of columns (NC consecutive columns per lane) and a chunk of its rows.  It walks
// the rows once: when row i's first colours are drawn, the last colours of the row before have all
// their neighbours final, so they follow at once, and a value is read, drawn and written within a
// few rows' time.
//   4-neighbour lattice, colours (i + j) mod 2: step i draws colour 0 of row i (from the old colour 1
//     of rows i - 1, i, i + 1), then colour 1 of row i - 1 (from the new colour 0 of rows i - 2 .. i).
//   8-neighbour lattice, colours 2 (i mod 2) + (j mod 2): step e (even) draws colours 0 and 1 of row e
//     (from the old odd rows e -+ 1), then colours 2 and 3 of row e - 1 (from the new rows e - 2, e).
// Vertical neighbours are the lane's own registers and horizontal ones a warp shuffle away: no shared
// memory and no block barrier in a sweep.  The sites beyond the strip and chunk that its own sites
// depend on are drawn again (identically: the draws are functions of their counters): one lane on
// either side (two for the 8-neighbour lattice with two chains: it needs four columns, the other two), and a
// row above and below (an even row below).  The new state goes to the other of two buffers, so no warp reads a
// neighbour's new values, and each owned site's terms of the two sums of the conjugate draws and its
// running moments are folded in as it is drawn.
//
// A lane has four columns with one chain and two with two, one Philox block's normals for its sites of a
// row; where a row starts within a block (a row length that is no multiple), the normals move over by
// that offset through a shuffle.
//
// Two forms of the same arithmetic in the same order, block for block: one launch per sweep (samplers
// of several fields, or without the resident path), and a batch of sweeps of a single field in one
// cooperative launch (a grid barrier per sweep, every block drawing the parameters; the normals of a
// chunk's first rows are drawn into shared memory while the barrier completes).
//
// Bound by instruction issue and its latencies (126 registers: four warps per scheduler, 47 % issue): about
// 124 instructions per site-update, 33 of them the normals and a fifth for sites drawn again (the
// tiled kernel of lattice_fused.cu, whose threads walk shared-memory tiles colour by colour, takes 300
// to 340).  Per sweep, against that kernel and a launch for the draws: 4-neighbour 2047 x 1931 one
// chain 24 us (46 without accumulation, 58 with, and 8), 8-neighbour 2048 x 2048 one chain 26 (49,
// quad kernel), 1900 x 1900 two chains 37 (66); the 112 lattices of a batch of 5.1 million sites 44 (84,
// 103 with accumulation).  Four chains in registers spill (8-neighbour 512 x 512, three chains: 25 us per
// sweep against 14 for the tiles kept resident), so more than two take the tiled kernel.
#include <cuda_runtime.h>

#include <type_traits>

#include "gmrf_device.cuh"
#include "gmrf_internal.h"
#include "grid_draws.cuh"
#include "packed_f32.cuh"

namespace gmrf {
namespace {

constexpr int kMarchThreads = 512;
constexpr int kMarchWarps = kMarchThreads / 32;
constexpr int kAheadBytes = 160 * 1024;  // shared memory of a block for normals drawn ahead

constexpr int march_cols(int V) { return V >= 2 ? 2 : 4; }                          // columns per lane
constexpr int march_halo(int kind, int V) { return (kind == kLat2D8 && V >= 2) ? 2 : 1; }  // lanes per side
constexpr int march_own(int kind, int V) { return (32 - 2 * march_halo(kind, V)) * march_cols(V); }

// One chunk of a sweep by one warp, V chains (all of the sampler's).  PLAIN: the intrinsic prior and no
// intercept (no degree terms, no third sum).
template <int KIND, int V, bool PLAIN>
struct March {
    static constexpr bool E8 = KIND == kLat2D8;
    static constexpr int NC = march_cols(V), NP = NC / 2, HL = march_halo(KIND, V);

    const MarchArgs &a;
    const FieldDev &f;
    static constexpr int Cp = V;
    int Hl, Wl, cols, rows, cs;      // cs: slots of a colour
    bool inner;                      // every column of the strip and its halo is on the lattice
    int c0;                          // first column of the lane (a multiple of NC, may be off the lattice)
    int ra, rb;                      // rows of the chunk (the 8-neighbour lattice: both even, or rb = H)
    bool mine;                       // the lane's columns are the strip's own
    const float *X, *Y;
    float *XW, *MEAN, *M2;
    float tau[V], isig[V], beta[V], tr[V];
    float rho, om, inv_k;
    bool acc;
    uint32_t sweep;
    float aS[V], aR[V], aA[V], aC[V];  // the sums; aC: the compensation of aA (with the intercept)
    int nrow;                          // rows around (0 .. 2) that rP and rs are for
    float rP[NC][V], rs[NC][V];        // 1/P and 1/sqrt(P) per column
    const float *zs;                   // normals drawn ahead: [row - first][NC V][thread], or null
    int zfirst, zcount;

    __device__ __forceinline__ March(const MarchArgs &a_, const FieldDev &f_) : a(a_), f(f_) {}

    __device__ __forceinline__ void place(const MarchTile &t, int warp)
    {
        const int lane = threadIdx.x & 31;
        Hl = f.dims[0];
        Wl = f.dims[1];
        cols = f.cols;
        rows = f.rows;
        cs = rows * cols;
        const int strips = (Wl + march_own(KIND, V) - 1) / march_own(KIND, V);
        const int chunk = t.block * kMarchWarps + warp;
        const int strip = chunk % strips, rc = chunk / strips;
        ra = min(rc * t.rows, Hl);
        rb = min(ra + t.rows, Hl);
        c0 = strip * march_own(KIND, V) + (lane - HL) * NC;
        mine = lane >= HL && lane < 32 - HL;
        inner = strip > 0 && strip * march_own(KIND, V) + (32 - HL) * NC < Wl;
        Y = static_cast<const float *>(a.f.y) + f.slot0;
        MEAN = static_cast<float *>(a.f.mean) + f.slot0 * Cp;
        M2 = static_cast<float *>(a.f.m2) + f.slot0 * Cp;
        rho = static_cast<float>(a.f.rho);
        om = 1.0f - rho;
        zs = nullptr;
        zfirst = zcount = 0;
    }
    __device__ __forceinline__ bool active() const { return ra < rb; }
    // Rows whose normals the chunk needs: [first_row, last_row].
    __device__ __forceinline__ int first_row() const { return E8 ? ra : ra - 1; }
    __device__ __forceinline__ int last_row() const { return rb; }
    // Column c0 + k exists (IN: every column of the strip and its halo does); the lane's q-th pair of
    // columns (one site of each of two colours) has one that does (c0 is even).
    template <bool IN = false>
    __device__ __forceinline__ bool col(int k) const { return IN || static_cast<unsigned>(c0 + k) < static_cast<unsigned>(Wl); }
    template <bool IN>
    __device__ __forceinline__ bool pair(int q) const { return col<IN>(2 * q); }

    __device__ __forceinline__ void start(long long sw, bool acc_, float inv_k_)
    {
        X = static_cast<const float *>((sw & 1) ? a.f.x_alt : a.f.x) + f.slot0 * Cp;
        XW = static_cast<float *>((sw & 1) ? a.f.x : a.f.x_alt) + f.slot0 * Cp;
        sweep = static_cast<uint32_t>(sw);
        acc = acc_;
        inv_k = inv_k_;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            tr[v] = tau[v] * rho;
            aS[v] = 0.0f;
            aR[v] = 0.0f;
            aA[v] = 0.0f;
            aC[v] = 0.0f;
        }
        nrow = -1;
    }

    // Slots: a row's place in every colour's sub-array is `off` (the lane's first site of the colour: the
    // site at column c0 + p lies at c0 / 2 for p = 0 and 1), the sub-arrays are `cs` apart.
    __device__ __forceinline__ int row_off(int i) const { return (E8 ? i >> 1 : i) * cols + (c0 >> 1); }
    __device__ __forceinline__ bool in_rows(int i) const { return static_cast<unsigned>(i) < static_cast<unsigned>(Hl); }
    // Values of the lane's sites of colour c in a row (zero off the lattice; padding slots are zero).
    template <bool IN>
    __device__ __forceinline__ void load(int c, int off, bool row, float (&v)[NP][V]) const
    {
#pragma unroll
        for (int q = 0; q < NP; ++q) {
#pragma unroll
            for (int k = 0; k < V; ++k) v[q][k] = 0.0f;
            if (row && pair<IN>(q)) Vec<float, V>::ld(X + static_cast<int64_t>(c * cs + off + q) * Cp, v[q]);
        }
    }
    template <bool IN>
    __device__ __forceinline__ void load_y(int c, int off, bool row, float (&v)[NP]) const
    {
#pragma unroll
        for (int q = 0; q < NP; ++q) v[q] = (row && pair<IN>(q)) ? Y[c * cs + off + q] : 0.0f;
    }

    // The normals of row i's NC sites.
    __device__ __forceinline__ void draw(uint32_t sw, int i, float (&z)[NC][V]) const
    {
        constexpr int G = V == 1 ? 4 : 2;  // sites of a Philox block
        constexpr int NB = NC / G;
        const int flat = i * Wl + c0;
        const int s = (i * Wl) & (G - 1);  // c0 is a multiple of G: the same for every lane
        // One chain: the lane's block is the one that its first sites lie in (s <= 1) or the next
        // (s >= 2), so that the columns that the outermost lanes need never lie beyond them (columns 0
        // to 2 of the last lane and 2, 3 of the first).
        const int ahead = G == 4 && s >= 2 ? 1 : 0;
        float n[NC][V];
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const uint32_t blk = static_cast<uint32_t>((flat >> (G == 4 ? 2 : 1)) + b + ahead);
            const uint4 w = philox4x32_10_rk(make_uint4(blk, sw, f.stream, kTagX << 24), a.rk);
            f2 z01, z23;
            box_muller_block_f32x2(w, z01, z23);
            float q[4];
            upk(z01, q[0], q[1]);
            upk(z23, q[2], q[3]);
#pragma unroll
            for (int k = 0; k < 4; ++k) n[b * G + k / V][k % V] = q[k];
        }
        // Site k's normal is number k + s of the blocks from the one that the lane's first site lies in.
        if (s == 0) {
#pragma unroll
            for (int k = 0; k < NC; ++k)
#pragma unroll
                for (int v = 0; v < V; ++v) z[k][v] = n[k][v];
        } else if (G == 2 || s == 1) {  // the last from the next lane's first
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const float t = __shfl_down_sync(0xffffffffu, n[0][v], 1);
#pragma unroll
                for (int k = 0; k < NC; ++k) z[k][v] = k + 1 < NC ? n[k + 1 < NC ? k + 1 : k][v] : t;
            }
        } else if constexpr (G == 4) {  // the first 4 - s from the last of the lane before
            const float t3 = __shfl_up_sync(0xffffffffu, n[3][0], 1);
            if (s == 2) {
                z[0][0] = __shfl_up_sync(0xffffffffu, n[2][0], 1);
                z[1][0] = t3;
                z[2][0] = n[0][0];
                z[3][0] = n[1][0];
            } else {
                z[0][0] = t3;
                z[1][0] = n[0][0];
                z[2][0] = n[1][0];
                z[3][0] = n[2][0];
            }
        }
    }
    __device__ __forceinline__ void normals(int i, float (&z)[NC][V]) const
    {
        if (static_cast<unsigned>(i - zfirst) < static_cast<unsigned>(zcount)) {
            const float *p = zs + static_cast<int64_t>(i - zfirst) * (NC * V) * kMarchThreads + threadIdx.x;
#pragma unroll
            for (int k = 0; k < NC * V; ++k) z[k / V][k % V] = p[k * kMarchThreads];
        } else {
            draw(sweep, i, z);
        }
    }

    // 1/P and 1/sqrt(P) of the lane's columns in row i, kept until a row with another number of rows
    // around (a warp's rows agree; they change at the first and last row only).
    template <bool IN>
    __device__ __forceinline__ void coefficients(int i)
    {
        const int nr = (i > 0 ? 1 : 0) + (i + 1 < Hl ? 1 : 0);
        if (nr == nrow) return;
        nrow = nr;
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            const int nc = (col<IN>(k - 1) ? 1 : 0) + (col<IN>(k + 1) ? 1 : 0);
            const float d = static_cast<float>(E8 ? (nc + 1) * (nr + 1) - 1 : nc + nr);
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const float P = fmaf(tau[v], d, isig[v]);
                rP[k][v] = rcp_approx(P);
                rs[k][v] = rsqrt_approx(P);
            }
        }
    }
    template <bool IN>
    __device__ __forceinline__ float degree(int k) const
    {
        const int nc = (col<IN>(k - 1) ? 1 : 0) + (col<IN>(k + 1) ? 1 : 0);
        return static_cast<float>(E8 ? (nc + 1) * (nrow + 1) - 1 : nc + nrow);
    }

    // The new value of column k from its neighbours' sum; the sums of the draws except the edges.
    template <bool IN>
    __device__ __forceinline__ void site(int k, const float (&s)[V], float y, const float (&z)[V], bool own, float (&xn)[V])
    {
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const float yb = PLAIN ? y : y - beta[v];
            const float m = fmaf(tr[v], s[v], yb * isig[v]) * rP[k][v];
            xn[v] = col<IN>(k) ? fmaf(z[v], rs[k][v], m) : 0.0f;
            if (own) {
                const float r = yb - xn[v];
                aR[v] = fmaf(r, r, aR[v]);
                if constexpr (!PLAIN) {  // Kahan's compensated sum: the residuals cancel
                    const float q = r - aC[v], t = aA[v] + q;
                    aC[v] = (t - aA[v]) - q;
                    aA[v] = t;
                    aS[v] = fmaf(om * degree<IN>(k) * xn[v], xn[v], aS[v]);
                }
            }
        }
    }
    __device__ __forceinline__ void edge(float (&e)[V], const float (&x)[V], const float (&n)[V], bool there) const
    {
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const float df = there ? x[v] - n[v] : 0.0f;
            e[v] = fmaf(df, df, e[v]);
        }
    }
    __device__ __forceinline__ void add_edges(const float (&e)[V])
    {
#pragma unroll
        for (int v = 0; v < V; ++v) aS[v] = PLAIN ? aS[v] + e[v] : fmaf(rho, e[v], aS[v]);
    }
    // Own sites of one colour written back, and their running moments.
    template <bool IN>
    __device__ __forceinline__ void load_moments(int c, int off, bool own, float (&mu)[NP][V], float (&mm)[NP][V]) const
    {
        if (!acc) return;
#pragma unroll
        for (int q = 0; q < NP; ++q)
            if (own && pair<IN>(q)) {
                const int64_t so = static_cast<int64_t>(c * cs + off + q) * Cp;
                Vec<float, V>::ld(MEAN + so, mu[q]);
                Vec<float, V>::ld(M2 + so, mm[q]);
            }
    }
    template <bool IN>
    __device__ __forceinline__ void store(int c, int off, int p, bool own, const float (&xn)[NP][V], float (&mu)[NP][V],
                                          float (&mm)[NP][V])
    {
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            if (!(own && col<IN>(p + 2 * q))) continue;
            const int64_t so = static_cast<int64_t>(c * cs + off + q) * Cp;
            Vec<float, V>::st(XW + so, xn[q]);
            if (acc) {
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    const float delta = xn[q][v] - mu[q][v];
                    mu[q][v] = fmaf(delta, inv_k, mu[q][v]);
                    mm[q][v] = fmaf(delta, xn[q][v] - mu[q][v], mm[q][v]);
                }
                Vec<float, V>::st(MEAN + so, mu[q]);
                Vec<float, V>::st(M2 + so, mm[q]);
            }
        }
    }

    // ---- 4-neighbour lattice ------------------------------------------------------------------
    // Colour C of row i, whose sites are columns P, P + 2 of the lane: o the other colour in rows
    // i - 1, i, i + 1 (U and D in the same columns, M in the columns between).
    template <bool IN, int C, int P>
    __device__ __forceinline__ void half_row(int i, const float (&U)[NP][V], const float (&M)[NP][V], const float (&D)[NP][V],
                                             const float (&y)[NP], const float (&z)[NP][V], bool own, float (&xn)[NP][V])
    {
        float side[V];
#pragma unroll
        for (int v = 0; v < V; ++v)
            side[v] = P == 0 ? __shfl_up_sync(0xffffffffu, M[NP - 1][v], 1) : __shfl_down_sync(0xffffffffu, M[0][v], 1);
        coefficients<IN>(i);
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            const int k = P + 2 * q;
            float Lf[V], Rt[V], s[V];
#pragma unroll
            for (int v = 0; v < V; ++v) {
                Lf[v] = P == 0 ? (q == 0 ? side[v] : M[q > 0 ? q - 1 : 0][v]) : M[q][v];
                Rt[v] = P == 0 ? M[q][v] : (q == NP - 1 ? side[v] : M[q < NP - 1 ? q + 1 : q][v]);
            }
#pragma unroll
            for (int v = 0; v < V; ++v) s[v] = ((U[q][v] + Lf[v]) + Rt[v]) + D[q][v];
            const bool o = own && col<IN>(k);
            site<IN>(k, s, y[q], z[q], o, xn[q]);
            if (C == 1 && o) {
                float e[V];
#pragma unroll
                for (int v = 0; v < V; ++v) e[v] = 0.0f;
                edge(e, xn[q], U[q], i > 0);
                edge(e, xn[q], Lf, col<IN>(k - 1));
                edge(e, xn[q], Rt, col<IN>(k + 1));
                edge(e, xn[q], D[q], i + 1 < Hl);
                add_edges(e);
            }
        }
    }
    // The window carried from step to step.
    struct Win4 {
        float o1[2][NP][V];            // old colour 1 of rows i - 1, i
        float n0[2][NP][V];            // new colour 0 of rows i - 2, i - 1
        float y1[NP], z1[NP][V];       // observations and normals of colour 1 in row i - 1
    };
    // Step i; P = i mod 2: colour 0 of row i and colour 1 of row i - 1 both are columns P, P + 2.
    template <bool IN, int P>
    __device__ __forceinline__ void step4(int i, int off, Win4 &w)
    {
        const bool own0 = mine && i >= ra && i < rb, own1 = mine && i > ra;  // (i <= rb: row i - 1 < rb)
        float nx[NP][V], y0[NP], yn[NP], mu0[NP][V], mm0[NP][V], mu1[NP][V], mm1[NP][V], z[NC][V];
        load<IN>(1, off + cols, in_rows(i + 1), nx);
        load_y<IN>(0, off, in_rows(i), y0);
        load_y<IN>(1, off, in_rows(i), yn);
        load_moments<IN>(0, off, own0, mu0, mm0);
        load_moments<IN>(1, off - cols, own1, mu1, mm1);
        normals(i, z);
        float z0[NP][V], x0[NP][V];
#pragma unroll
        for (int q = 0; q < NP; ++q)
#pragma unroll
            for (int v = 0; v < V; ++v) {
                z0[q][v] = z[P + 2 * q][v];
                x0[q][v] = 0.0f;
            }
        if (in_rows(i)) {
            half_row<IN, 0, P>(i, w.o1[0], w.o1[1], nx, y0, z0, own0, x0);
            store<IN>(0, off, P, own0, x0, mu0, mm0);
        }
        if (i > ra) {
            float x1[NP][V];
            half_row<IN, 1, P>(i - 1, w.n0[0], w.n0[1], x0, w.y1, w.z1, own1, x1);
            store<IN>(1, off - cols, P, own1, x1, mu1, mm1);
        }
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            w.y1[q] = yn[q];
#pragma unroll
            for (int v = 0; v < V; ++v) {
                w.o1[0][q][v] = w.o1[1][q][v];
                w.o1[1][q][v] = nx[q][v];
                w.n0[0][q][v] = w.n0[1][q][v];
                w.n0[1][q][v] = x0[q][v];
                w.z1[q][v] = z[(1 - P) + 2 * q][v];
            }
        }
    }
    template <bool IN>
    __device__ __forceinline__ void march4()
    {
        Win4 w;
        int off = row_off(ra - 1);
        load<IN>(1, off - cols, in_rows(ra - 2), w.o1[0]);
        load<IN>(1, off, in_rows(ra - 1), w.o1[1]);
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            w.y1[q] = 0.0f;
#pragma unroll
            for (int v = 0; v < V; ++v) {
                w.n0[0][q][v] = 0.0f;
                w.n0[1][q][v] = 0.0f;
                w.z1[q][v] = 0.0f;
            }
        }
#pragma unroll 1
        for (int i = ra - 1; i <= rb; ++i, off += cols) {
            if (i & 1) step4<IN, 1>(i, off, w);
            else step4<IN, 0>(i, off, w);
        }
    }

    // ---- 8-neighbour lattice ------------------------------------------------------------------
    // Rows as columns -1 .. NC of the lane (index k + 1), the outer two from the lanes beside.
    using Row = float[NC + 2][V];
    __device__ __forceinline__ void sides(Row &r) const
    {
#pragma unroll
        for (int v = 0; v < V; ++v) {
            r[0][v] = __shfl_up_sync(0xffffffffu, r[NC][v], 1);
            r[NC + 1][v] = __shfl_down_sync(0xffffffffu, r[1][v], 1);
        }
    }
    // One colour of a row: the columns B, B + 2 of `row` (in-row neighbours in `row` itself).  LOW:
    // which neighbours are of lower colour: 0 none, 1 the in-row ones, 2 the rows above and below,
    // 3 all.
    template <bool IN, int B, int LOW>
    __device__ __forceinline__ void half_row8(int i, const Row &U, Row &row, const Row &D, const float (&y)[NP],
                                              const float (&z)[NC][V], bool own, float (&xn)[NP][V])
    {
        const bool up = i > 0, down = i + 1 < Hl;
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            const int k = B + 2 * q;  // column; index k + 1 in a row
            float s[V];
#pragma unroll
            for (int v = 0; v < V; ++v)
                s[v] = ((((((U[k][v] + U[k + 1][v]) + U[k + 2][v]) + row[k][v]) + row[k + 2][v]) + D[k][v]) + D[k + 1][v]) +
                       D[k + 2][v];
            const bool o = own && col<IN>(k);
            site<IN>(k, s, y[q], z[k], o, xn[q]);
            if (LOW && o) {
                float e[V];
#pragma unroll
                for (int v = 0; v < V; ++v) e[v] = 0.0f;
                if (LOW & 2) {
                    edge(e, xn[q], U[k], up && col<IN>(k - 1));
                    edge(e, xn[q], U[k + 1], up);
                    edge(e, xn[q], U[k + 2], up && col<IN>(k + 1));
                }
                if (LOW & 1) {
                    edge(e, xn[q], row[k], col<IN>(k - 1));
                    edge(e, xn[q], row[k + 2], col<IN>(k + 1));
                }
                if (LOW & 2) {
                    edge(e, xn[q], D[k], down && col<IN>(k - 1));
                    edge(e, xn[q], D[k + 1], down);
                    edge(e, xn[q], D[k + 2], down && col<IN>(k + 1));
                }
                add_edges(e);
            }
        }
#pragma unroll
        for (int q = 0; q < NP; ++q)
#pragma unroll
            for (int v = 0; v < V; ++v) row[B + 2 * q + 1][v] = xn[q][v];
    }
    template <bool IN>
    __device__ __forceinline__ void march8()
    {
        Row odd, even, nodd, neven;  // old odd row e - 1, new even row e - 2; and those two rows on
        float t[NP][V], u[NP][V];
        int off = row_off(ra);  // of rows e and e + 1
        auto load_odd = [&](int i, int o, Row &r) {
            load<IN>(2, o, in_rows(i), t);
            load<IN>(3, o, in_rows(i), u);
#pragma unroll
            for (int q = 0; q < NP; ++q)
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    r[2 * q + 1][v] = t[q][v];
                    r[2 * q + 2][v] = u[q][v];
                }
        };
        load_odd(ra - 1, off - cols, odd);
        sides(odd);
#pragma unroll
        for (int k = 0; k < NC + 2; ++k)
#pragma unroll
            for (int v = 0; v < V; ++v) even[k][v] = 0.0f;
#pragma unroll 1
        for (int e = ra; e <= rb; e += 2, off += cols) {
            const bool own_e = mine && e < rb, do_o = e > ra, own_o = mine && do_o;
            float y0[NP], y1[NP], y2[NP], y3[NP], z[NC][V], xn[NP][V], mu[2][NP][V], mm[2][NP][V];
            load_odd(e + 1, off, nodd);
            load<IN>(1, off, in_rows(e), t);
            load_y<IN>(0, off, in_rows(e), y0);
            load_y<IN>(1, off, in_rows(e), y1);
            load_moments<IN>(0, off, own_e, mu[0], mm[0]);
            load_moments<IN>(1, off, own_e, mu[1], mm[1]);
            if (e < Hl) {
                normals(e, z);
                coefficients<IN>(e);
            }
            sides(nodd);
#pragma unroll
            for (int q = 0; q < NP; ++q)
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    neven[2 * q + 1][v] = 0.0f;
                    neven[2 * q + 2][v] = t[q][v];  // old colour 1
                }
#pragma unroll
            for (int v = 0; v < V; ++v) neven[0][v] = __shfl_up_sync(0xffffffffu, neven[NC][v], 1);
            if (e < Hl) {
                half_row8<IN, 0, 0>(e, odd, neven, nodd, y0, z, own_e, xn);
                store<IN>(0, off, 0, own_e, xn, mu[0], mm[0]);
            }
#pragma unroll
            for (int v = 0; v < V; ++v) neven[NC + 1][v] = __shfl_down_sync(0xffffffffu, neven[1][v], 1);
            if (e < Hl) {
                half_row8<IN, 1, 1>(e, odd, neven, nodd, y1, z, own_e, xn);
                store<IN>(1, off, 1, own_e, xn, mu[1], mm[1]);
            }
            sides(neven);
            if (do_o) {
                const int o = e - 1;
                load_y<IN>(2, off - cols, true, y2);
                load_y<IN>(3, off - cols, true, y3);
                load_moments<IN>(2, off - cols, own_o, mu[0], mm[0]);
                load_moments<IN>(3, off - cols, own_o, mu[1], mm[1]);
                normals(o, z);
                coefficients<IN>(o);
                half_row8<IN, 0, 2>(o, even, odd, neven, y2, z, own_o, xn);
                store<IN>(2, off - cols, 0, own_o, xn, mu[0], mm[0]);
                sides(odd);
                half_row8<IN, 1, 3>(o, even, odd, neven, y3, z, own_o, xn);
                store<IN>(3, off - cols, 1, own_o, xn, mu[1], mm[1]);
            }
#pragma unroll
            for (int k = 0; k < NC + 2; ++k)
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    odd[k][v] = nodd[k][v];
                    even[k][v] = neven[k][v];
                }
        }
    }
    __device__ __forceinline__ void march()
    {
        if constexpr (E8) {
            if (inner) march8<true>();
            else march8<false>();
        } else {
            if (inner) march4<true>();
            else march4<false>();
        }
#pragma unroll
        for (int v = 0; v < V; ++v) aA[v] -= aC[v];
    }
};

// The block's sums per chain: a shuffle tree over each warp's lanes, then the warps in
// order, FP32 (compensated terms aside, a few hundred sites); thread chain * 3 + k returns value k.
template <int V>
__device__ __forceinline__ float march_sums(const float (&aS)[V], const float (&aR)[V], const float (&aA)[V],
                                            float (&red)[kMarchWarps][V][3])
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int v = 0; v < V; ++v) {
        float sS = aS[v], sR = aR[v], sA = aA[v];
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) {
            sS += __shfl_xor_sync(0xffffffffu, sS, o);
            sR += __shfl_xor_sync(0xffffffffu, sR, o);
            sA += __shfl_xor_sync(0xffffffffu, sA, o);
        }
        if (lane == 0) {
            red[warp][v][0] = sS;
            red[warp][v][1] = sR;
            red[warp][v][2] = sA;
        }
    }
    __syncthreads();
    float s = 0.0f;
    if (threadIdx.x < V * 3) {
        const int chain = threadIdx.x / 3, k = threadIdx.x - 3 * chain;
#pragma unroll
        for (int w = 0; w < kMarchWarps; ++w) s += red[w][chain][k];
    }
    return s;
}

// One sweep per launch.
template <int KIND, int V, bool PLAIN>
__global__ void __launch_bounds__(kMarchThreads, 1) march_kernel(const MarchArgs a)
{
    __shared__ float red[kMarchWarps][V][3];
    const MarchTile t = a.tiles[blockIdx.x];
    const FieldDev f = a.f.fields[t.field];
    March<KIND, V, PLAIN> m(a, f);
    m.place(t, threadIdx.x >> 5);
    pdl_wait();
    pdl_release();
    const long long sw = a.f.ctl->sweep;
    const bool acc = a.f.acc_enabled && sweep_accumulated(sw, a.f.burn_in, a.f.thin);
    const float *hyp = static_cast<const float *>(a.f.hyp) + (static_cast<int64_t>(t.field) * V) * kHypStride;
#pragma unroll
    for (int v = 0; v < V; ++v) {
        m.tau[v] = hyp[kHypStride * v];
        m.isig[v] = hyp[kHypStride * v + 1];
        m.beta[v] = hyp[kHypStride * v + 2];
    }
    m.start(sw, acc, acc ? 1.0f / static_cast<float>(a.f.ctl->acc_count + 1) : 0.0f);
    if (m.active()) m.march();
    const float s = march_sums<V>(m.aS, m.aR, m.aA, red);
    if (threadIdx.x < V * 3) {
        const int chain = threadIdx.x / 3, k = threadIdx.x - 3 * chain;
        reinterpret_cast<double *>(a.f.partials + static_cast<int64_t>(t.part) * V + chain)[k] = static_cast<double>(s);
    }
}

// A batch of sweeps of a single field (at most kGridChains chains).
template <int KIND, int V, bool PLAIN>
__global__ void __launch_bounds__(kMarchThreads, 1) march_grid_kernel(const MarchArgs a)
{
    extern __shared__ __align__(16) float zsm[];
    __shared__ GridShared sh;
    __shared__ float red[kMarchWarps][V][3];
    const HyperArgs &h = a.h;
    const MarchTile t = a.tiles[blockIdx.x];
    const FieldDev f = a.f.fields[t.field];
    SweepCtl *ctl = a.f.ctl;
    const int tid = threadIdx.x, nblk = gridDim.x;
    March<KIND, V, PLAIN> m(a, f);
    m.place(t, tid >> 5);
    const long long sweep0 = ctl->sweep;
    long long acc_count = ctl->acc_count;
    grid_draws_init(sh, h, a.count, sweep0);
    __syncthreads();
    // The first rows' normals of a sweep, drawn ahead into shared memory.
    auto ahead = [&](long long sw) {
        for (int r = 0; r < a.zrows; ++r) {
            const int i = m.first_row() + r;
            if (i > m.last_row()) break;
            float z[March<KIND, V, PLAIN>::NC][V];
            m.draw(static_cast<uint32_t>(sw), i, z);
#pragma unroll
            for (int k = 0; k < March<KIND, V, PLAIN>::NC * V; ++k)
                zsm[(r * March<KIND, V, PLAIN>::NC * V + k) * kMarchThreads + tid] = z[k / V][k % V];
        }
    };
    if (m.active()) ahead(sweep0);
    m.zs = zsm;
    m.zfirst = m.first_row();
    m.zcount = a.zrows;
    unsigned long long arrivals = a.extra_arrivals;
    for (int it = 0; it < a.count; ++it) {
        const long long sw = sweep0 + it;
        const bool acc = a.f.acc_enabled && sweep_accumulated(sw, a.f.burn_in, a.f.thin);
#pragma unroll
        for (int v = 0; v < V; ++v) {
            m.tau[v] = sh.hs[v][0];
            m.isig[v] = sh.hs[v][1];
            m.beta[v] = sh.hs[v][2];
        }
        m.start(sw, acc, acc ? 1.0f / static_cast<float>(acc_count + 1) : 0.0f);
        if (m.active()) m.march();
        if (acc) ++acc_count;
        const float s = march_sums<V>(m.aS, m.aR, m.aA, red);
        // [chain][S, R, A][block], by the sweep's parity: a block of a few rows ends its next sweep while
        // others, still drawing ahead, have not read this one's sums
        double *const pm = a.pm + (it & 1) * 3 * V * nblk;
        if (tid < V * 3) pm[tid * nblk + blockIdx.x] = static_cast<double>(s);
        __syncthreads();  // the block's stores of this sweep
        if (tid == 0) grid_arrive(ctl);
        arrivals += nblk;
        if (it + 1 < a.count && m.active()) ahead(sw + 1);
        if (tid == 0 && grid_wait(ctl, arrivals, a.wait_ns)) sh.abort = 1;
        __syncthreads();
        if (sh.abort) break;
        grid_draw(sh, h, pm, nblk, f, sw, it, blockIdx.x == 0);
        __syncthreads();
    }
    grid_finish(ctl, sweep0 + a.count, acc_count);
}

// The sums of the draws from the current state, with the blocks of the sweep (gmrf_hyper_update).
template <int KIND, int V>
__global__ void __launch_bounds__(kMarchThreads) march_reduce_kernel(const MarchArgs a)
{
    constexpr bool E8 = KIND == kLat2D8;
    __shared__ float red[kMarchWarps][V][3];
    const MarchTile t = a.tiles[blockIdx.x];
    const FieldDev f = a.f.fields[t.field];
    March<KIND, V, false> m(a, f);
    m.place(t, threadIdx.x >> 5);
    pdl_wait();
    pdl_release();
    const long long sw = a.f.ctl->sweep;
    const float *hyp = static_cast<const float *>(a.f.hyp) + (static_cast<int64_t>(t.field) * V) * kHypStride;
#pragma unroll
    for (int v = 0; v < V; ++v) {
        m.tau[v] = hyp[kHypStride * v];
        m.isig[v] = hyp[kHypStride * v + 1];
        m.beta[v] = hyp[kHypStride * v + 2];
    }
    m.start(sw, false, 0.0f);
    auto colour = [](int i, int j) { return E8 ? 2 * (i & 1) + (j & 1) : (i + j) & 1; };
    auto at = [&](int i, int j) { return (static_cast<int64_t>(colour(i, j)) * m.rows + (E8 ? i >> 1 : i)) * m.cols + (j >> 1); };
    if (m.mine)
        for (int i = m.ra; i < m.rb; ++i)
            for (int k = 0; k < March<KIND, V, false>::NC; ++k) {
                const int j = m.c0 + k;
                if (j < 0 || j >= m.Wl) continue;
                float x[V], e[V];
                Vec<float, V>::ld(m.X + at(i, j) * V, x);
                int deg = 0;
#pragma unroll
                for (int v = 0; v < V; ++v) e[v] = 0.0f;
                for (int di = -1; di <= 1; ++di)
                    for (int dj = -1; dj <= 1; ++dj) {
                        const int ii = i + di, jj = j + dj;
                        if ((di == 0 && dj == 0) || (!E8 && di != 0 && dj != 0) || ii < 0 || ii >= m.Hl || jj < 0 || jj >= m.Wl) continue;
                        ++deg;
                        if (colour(ii, jj) >= colour(i, j)) continue;
                        float nb[V];
                        Vec<float, V>::ld(m.X + at(ii, jj) * V, nb);
                        m.edge(e, x, nb, true);
                    }
                m.add_edges(e);
                const float y = m.Y[at(i, j)];
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    m.aS[v] += m.om * static_cast<float>(deg) * x[v] * x[v];
                    const float r = (y - m.beta[v]) - x[v];
                    m.aR[v] = fmaf(r, r, m.aR[v]);
                    m.aA[v] += r;
                }
            }
    const float s = march_sums<V>(m.aS, m.aR, m.aA, red);
    if (threadIdx.x < V * 3) {
        const int chain = threadIdx.x / 3, k = threadIdx.x - 3 * chain;
        reinterpret_cast<double *>(a.f.partials + static_cast<int64_t>(t.part) * V + chain)[k] = static_cast<double>(s);
    }
}

// The configuration of a sampler (one or two chains) and its model, passed to `use`.
template <int KIND, int V, typename Use>
cudaError_t with_model(bool plain, Use &&use)
{
    std::integral_constant<int, KIND> kd;
    std::integral_constant<int, V> v;
    return plain ? use(kd, v, std::true_type{}) : use(kd, v, std::false_type{});
}
template <typename Use>
cudaError_t with_march(int kind, int Cp, bool plain, Use &&use)
{
    if (kind == kLat2D8) return Cp == 2 ? with_model<kLat2D8, 2>(plain, use) : with_model<kLat2D8, 1>(plain, use);
    return Cp == 2 ? with_model<kLat2D4, 2>(plain, use) : with_model<kLat2D4, 1>(plain, use);
}
bool plain_model(const MarchArgs &a) { return !a.intercept && a.f.rho == 1.0; }
size_t z_row_bytes(int Cp) { return sizeof(float) * march_cols(Cp) * Cp * kMarchThreads; }

}  // namespace

int march_strips(int kind, int Cp, int W)
{
    const int own = march_own(kind, Cp);
    return (W + own - 1) / own;
}

int march_blocks(int kind, int Cp, int H, int W, int rows)
{
    const int64_t q = static_cast<int64_t>((H + rows - 1) / rows) * march_strips(kind, Cp, W);
    return static_cast<int>((q + kMarchWarps - 1) / kMarchWarps);
}

int march_warps() { return kMarchWarps; }

int march_ahead_rows(int Cp, int rows)
{
    const int most = static_cast<int>(kAheadBytes / z_row_bytes(Cp));
    return rows + 2 < most ? rows + 2 : most;
}

cudaError_t plan_march_grid(int kind, int Cp, int blocks, int zrows, bool *fits)
{
    *fits = false;
    if (blocks > 32 * kSumRows) return cudaSuccess;
    int dev = 0, sms = 0, coop = 0, per_sm = 32;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (e == cudaSuccess)
        for (bool plain : {true, false})
            if (e == cudaSuccess)
                e = with_march(kind, Cp, plain, [&](auto kd, auto v, auto pl) {
                    auto *k = march_grid_kernel<decltype(kd)::value, decltype(v)::value, decltype(pl)::value>;
                    const cudaError_t a = allow_smem(k, z_row_bytes(Cp) * zrows);
                    int n = 0;
                    const cudaError_t o = a != cudaSuccess ? a : cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                                                                     &n, k, kMarchThreads, z_row_bytes(Cp) * zrows);
                    per_sm = n < per_sm ? n : per_sm;
                    return o;
                });
    *fits = e == cudaSuccess && coop && static_cast<int64_t>(per_sm) * sms >= blocks;
    return e;
}

cudaError_t launch_march(int kind, const MarchArgs &a, cudaStream_t stream)
{
    if (a.ntiles <= 0) return cudaSuccess;
    return with_march(kind, a.f.Cp, plain_model(a), [&](auto kd, auto v, auto pl) {
        constexpr int KD = decltype(kd)::value, V = decltype(v)::value;
        if (!a.f.update) return launch_sweep_kernel(march_reduce_kernel<KD, V>, dim3(a.ntiles), dim3(kMarchThreads), 0, stream, a);
        return launch_sweep_kernel(march_kernel<KD, V, decltype(pl)::value>, dim3(a.ntiles), dim3(kMarchThreads), 0, stream, a);
    });
}

cudaError_t launch_march_grid(int kind, const MarchArgs &a, cudaStream_t stream)
{
    return with_march(kind, a.f.Cp, plain_model(a), [&](auto kd, auto v, auto pl) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(a.ntiles);
        cfg.blockDim = dim3(kMarchThreads);
        cfg.dynamicSmemBytes = z_row_bytes(a.f.Cp) * a.zrows;
        cfg.stream = stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, march_grid_kernel<decltype(kd)::value, decltype(v)::value, decltype(pl)::value>, a);
    });
}

}  // namespace gmrf
