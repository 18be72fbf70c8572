"""Edges of the rules that choose kernels and of their sizes: Polya-Gamma sites at the ends of a draw's
segments, draws at the number of partial sums from which a block per draw takes over, FP64 tiles and
degree tables, moments pooled over every chain count's vector width, read-backs at the size up to which
they go through pinned memory, and samplers of different sizes alive at once."""
import numpy as np
import pytest

import oracle
from gmrf_testutil import (TOL_FP32_1, TOL_FP32_1000, TOL_FP64, oracle_colors, oracle_graph, relerr, run_oracle,
                           trace_relerr)
from paper_1702_05518_gb300 import gmrf as g
from paper_1702_05518_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1702_05518_gb300 import build

    build.build()


@pytest.mark.parametrize("precision,chains", [(g.FP64, 1), (g.FP64, 3), (g.FP32, 2)])
@pytest.mark.parametrize("trials", [[0], [1], [31, 32, 33], [4095, 0, 1], [1023, 1024, 1025, 0, 0, 5]], ids=str)
def test_polya_gamma_trials(precision, chains, trials):
    dims = (13, 21)
    n = dims[0] * dims[1]
    m = np.resize(np.array(trials, np.int32), n)
    f = {"kind": wl.LATTICE2D_4, "dims": dims, "n": n, "y": wl.rng(4).binomial(m, 0.4).astype(np.float64), "trials": m}
    T, tol = (4, TOL_FP64) if precision == g.FP64 else (1, TOL_FP32_1)
    st = oracle.initial_state(f["y"], chains, x0=np.zeros(n))
    out = oracle.run(oracle_graph(f), oracle_colors(f), f["y"], st, seed=31, nsweeps=T, stream=0, prior="pcar", rho=0.99,
                     a_tau=1.0, b_tau=1.0, trials=m, beta0_prior=(0.0, 1000.0), accumulate=False)
    with g.Sampler([f], precision=precision, chains=chains, seed=31, likelihood=g.LIKELIHOOD_BINOMIAL, prior=g.PRIOR_PCAR,
                   rho=0.99, a_tau=1.0, b_tau=1.0, beta0_prior=(0.0, 1000.0)) as s:
        s.sweep(T)
        for c in range(chains):
            assert relerr(s.fetch(0, c)["x"], st.x[c]) <= tol
            assert relerr(s.fetch_intercept(0, c, trace=T)["beta0_trace"], out["beta0_trace"][c]) <= tol


@pytest.mark.parametrize("chains", [1, 2, 8])
@pytest.mark.parametrize("cols", [120, 127, 128, 129, 136])  # tiles of 8 x 8: 240, 256, 256, 272, 272 partial sums
def test_draws_around_the_wide_kernel(cols, chains):
    f = wl.small_lattice(wl.LATTICE2D_4, (128, cols), 15)
    tuning = {"fused_rows": [8, 8], "fused_cols": [8, 8], "fused_threads": [512, 512]}
    st, out = run_oracle(f, chains, 6, seed=6, stream=0, intercept=True)
    with g.Sampler([f], precision=g.FP32, chains=chains, seed=6, intercept=True, flags=g.FLAG_NO_RESIDENT, tuning=tuning) as s:
        s.sweep(6)
        for c in range(chains):
            r = s.fetch(0, c, trace=6)
            assert relerr(r["x"], st.x[c]) <= TOL_FP32_1000
            assert trace_relerr(r["tau_trace"], out["tau_trace"][c]) <= TOL_FP32_1000
            assert trace_relerr(r["sigma2_trace"], out["sigma2_trace"][c]) <= TOL_FP32_1000


@pytest.mark.parametrize("chains", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("kind,dims", [(wl.LATTICE2D_4, (1, 1)), (wl.LATTICE2D_8, (8, 16)), (wl.LATTICE2D_4, (65, 63)),
                                       (wl.LATTICE2D_8, (130, 97)), (wl.LATTICE3D_6, (2, 3, 5)), (wl.LATTICE3D_6, (33, 17, 20))])
def test_fp64_tiles_and_degrees(kind, dims, chains):
    f = wl.small_lattice(kind, dims, 16)
    st, out = run_oracle(f, chains, 5, seed=8, stream=0, prior="pcar", rho=0.7, burn_in=1)
    with g.Sampler([f], precision=g.FP64, chains=chains, seed=8, prior=g.PRIOR_PCAR, rho=0.7, burn_in=1) as s:
        s.sweep(5)
        for c in range(chains):
            r = s.fetch(0, c, trace=5)
            assert relerr(r["x"], st.x[c]) <= TOL_FP64 and relerr(r["mean"], st.mean[c]) <= TOL_FP64
            assert trace_relerr(r["tau_trace"], out["tau_trace"][c]) <= TOL_FP64


@pytest.mark.parametrize("chains", [20, 40])  # 16 and 32 chain vectors to a warp
@pytest.mark.parametrize("rho", [1.0, 0.7])
@pytest.mark.parametrize("kind,dims,flags", [(wl.LATTICE3D_6, (3, 4, 5), 0), (wl.LATTICE2D_8, (9, 7), g.FLAG_PER_COLOUR),
                                             (wl.LATTICE2D_4, (9, 7), 0)])
def test_fp64_sums_of_many_chains(kind, dims, flags, chains, rho):
    f = wl.small_lattice(kind, dims, 16)
    st, out = run_oracle(f, chains, 4, seed=8, stream=0, prior="icar" if rho == 1.0 else "pcar", rho=rho, burn_in=1,
                         intercept=True)
    with g.Sampler([f], precision=g.FP64, chains=chains, seed=8, prior=g.PRIOR_ICAR if rho == 1.0 else g.PRIOR_PCAR,
                   rho=rho, burn_in=1, intercept=True, flags=flags) as s:
        s.sweep(4)
        for c in (0, 1, chains - 1):
            r = s.fetch(0, c, trace=4)
            assert relerr(r["x"], st.x[c]) <= TOL_FP64 and relerr(r["mean"], st.mean[c]) <= TOL_FP64
            assert trace_relerr(r["tau_trace"], out["tau_trace"][c]) <= TOL_FP64
            assert trace_relerr(r["sigma2_trace"], out["sigma2_trace"][c]) <= TOL_FP64


@pytest.mark.parametrize("precision", [g.FP32, g.FP64])
@pytest.mark.parametrize("chains", [1, 2, 3, 5, 8, 11, 16])
def test_pooled_moments(precision, chains):
    # the same FP64 sums of the same (FP32 or FP64) moments, in another order: a few roundings apart
    f = wl.small_lattice(wl.LATTICE2D_8, (19, 37), 17)
    k = 9
    with g.Sampler([f], precision=precision, chains=chains, seed=9, burn_in=2) as s:
        s.sweep(2 + k)
        m, v = s.fetch_pooled(0)
        parts = [s.fetch(0, c) for c in range(chains)]
    mc, vc = np.stack([p["mean"] for p in parts]), np.stack([p["var"] for p in parts])
    mean = mc.mean(0)
    np.testing.assert_allclose(m, mean, rtol=1e-13, atol=1e-13)
    # var is stored as M2 / (k - 1); an FP32 sampler's fetch divides in FP64
    np.testing.assert_allclose(v, ((k - 1) * vc + k * (mc - mean) ** 2).sum(0) / (chains * k - 1), rtol=1e-12, atol=1e-15)


@pytest.mark.parametrize("n", [8191, 8192, 8193])
def test_fetches_around_the_pinned_size(n):
    # a row of n sites and a trace of n sweeps; the trace's ring wraps at its capacity
    f = wl.small_lattice(wl.LATTICE2D_4, (1, 40), 18)
    with g.Sampler([f], precision=g.FP32, chains=2, seed=10, trace_capacity=n) as s:
        s.sweep(n + 5)
        full = s.fetch(0, 1, trace=n)
        tail = s.fetch(0, 1, trace=7)
        assert len(full["tau_trace"]) == n and np.all(full["tau_trace"] > 0)
        np.testing.assert_array_equal(full["tau_trace"][-7:], tail["tau_trace"])
        assert full["tau_trace"][-1] == full["tau"] and full["sigma2_trace"][-1] == full["sigma2"]
    big = wl.small_lattice(wl.LATTICE2D_4, (1, n), 19)
    st, _ = run_oracle(big, 1, 2, seed=11, stream=0, burn_in=0)
    with g.Sampler([big], precision=g.FP64, chains=1, seed=11) as s:
        s.set_data(0, big["y"])
        s.sweep(2)
        r = s.fetch(0, 0)
        assert relerr(r["x"], st.x[0]) <= TOL_FP64 and relerr(r["mean"], st.mean[0]) <= TOL_FP64
        np.testing.assert_array_equal(s.fetch_pooled(0)[0], r["mean"])


def _graph(n, seed):
    rp, ci, _ = wl.delaunay_graph(n, wl.rng(seed))
    return dict(wl.graph_field(rp, ci, seed=seed), color_seed=seed)


PAIRS = {
    "lattice": (g.FP32, 1, lambda: (wl.small_lattice(wl.LATTICE2D_8, (60, 60), 1), wl.small_lattice(wl.LATTICE2D_8, (12, 9), 2))),
    "tiles": (g.FP32, 2, lambda: (wl.small_lattice(wl.LATTICE2D_4, (400, 380), 1), wl.small_lattice(wl.LATTICE2D_4, (90, 200), 2))),
    "quad": (g.FP32, 1, lambda: (wl.small_lattice(wl.LATTICE2D_8, (1024, 1024), 1), wl.small_lattice(wl.LATTICE2D_8, (300, 300), 2))),
    "march": (g.FP32, 1, lambda: (wl.small_lattice(wl.LATTICE2D_4, (2100, 1999), 1), wl.small_lattice(wl.LATTICE2D_4, (1300, 1300), 2))),
    "graph": (g.FP32, 3, lambda: (_graph(9000, 1), _graph(300, 2))),
    "fp64": (g.FP64, 1, lambda: (wl.small_lattice(wl.LATTICE2D_8, (400, 400), 1), wl.small_lattice(wl.LATTICE2D_8, (20, 33), 2))),
}


@pytest.mark.parametrize("case", list(PAIRS))
def test_samplers_side_by_side(case):
    # a smaller sampler made after a larger one leaves the larger one's shared memory alone
    precision, chains, make = PAIRS[case]
    fields = make()

    def new(f, s):
        return g.Sampler([f], precision=precision, chains=chains, seed=s, graph_sweeps=4)

    alone = []
    for k, f in enumerate(fields):
        with new(f, k) as s:
            s.sweep(6)
            alone.append(s.fetch(0, 0)["x"])
    with new(fields[0], 0) as a, new(fields[1], 1) as b:
        for n in (4, 2):
            a.sweep(n)
            b.sweep(n)
        np.testing.assert_array_equal(a.fetch(0, 0)["x"], alone[0])
        np.testing.assert_array_equal(b.fetch(0, 0)["x"], alone[1])
