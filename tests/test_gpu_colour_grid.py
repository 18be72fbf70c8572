"""Grid sweeps (colour_grid.cu): whole sweeps of a single FP32 field's colour steps in one cooperative
launch, a grid barrier per colour step.  Parity with the oracle (1e-5 after one sweep, 1e-4 on
states, means and traces after more) where its indexing can go wrong, the same results however
the sweeps are cut into launches, agreement with the launch-per-colour path, and the bounded wait.
"""
import numpy as np
import pytest

from gmrf_testutil import TOL_FP32_1, TOL_FP32_1000, relerr, run_oracle, trace_relerr
from paper_1702_05518_gb300 import gmrf as g
from paper_1702_05518_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1702_05518_gb300 import build

    build.build()


def _weighted(rp, ci, seed, color_seed=5):
    f = dict(wl.graph_field(rp, ci, seed=seed), color_seed=color_seed)
    rows = np.repeat(np.arange(f["n"]), np.diff(f["row_ptr"]))
    lo, hi = np.minimum(rows, f["col_idx"]), np.maximum(rows, f["col_idx"])
    f["weights"] = 0.25 + ((lo * 7 + hi * 13) % 17) / 8.0  # symmetric, positive
    return f


def _delaunay(n, seed):
    return wl.delaunay_graph(n, wl.rng(seed))[:2]


# One vertex per class and block, hubs far beyond the neighbours loaded ahead, isolated vertices,
# classes that leave blocks and threads without work, more positions than threads.
FIELDS = {
    "k4": lambda: _weighted(*wl.k4_minus_edge(), 1),
    "star_700": lambda: dict(wl.graph_field(*wl.star_graph(700), seed=2), color_seed=5),
    "isolated": lambda: _weighted(*wl.csr_from_edges(300, np.array([[0, 1], [5, 250]])), 3),
    "dense_90": lambda: _weighted(*wl.random_graph(90, 0.3, wl.rng(4)), 4),
    "delaunay_1000": lambda: _weighted(*_delaunay(1000, 6), 6),
    "delaunay_33000": lambda: dict(wl.graph_field(*_delaunay(33000, 7), seed=7), color_seed=5),
}


# Units of a thread (up to four consecutive sites) across row and plane ends of every parity, single
# rows, columns and planes, a last unit that is not full.
VOLUMES = [(1, 1, 1), (1, 1, 9), (7, 1, 1), (1, 6, 1), (5, 3, 2), (3, 5, 3), (3, 4, 7), (2, 3, 6), (9, 8, 5), (17, 13, 11),
           (20, 24, 28)]
# One, two or four units per thread: (chains, extents) at the sizes where the number grows.
UNITS = [(1, (61, 71, 73)), (1, (89, 85, 83)), (2, (50, 61, 53)), (2, (72, 70, 67)), (4, (55, 54, 53)), (8, (44, 43, 45))]


def _volume(dims):
    return wl.small_lattice(wl.LATTICE3D_6, dims, 8)


def _run(f, chains, calls, intercept=False, **kw):
    with g.Sampler([f], precision=g.FP32, chains=chains, seed=31, trace_capacity=512, intercept=intercept, **kw) as s:
        for n, hyper in calls:
            s.sweep(n, with_hyper=hyper)
        T = sum(n for n, _ in calls)
        out = [s.fetch(0, c, trace=T) for c in range(chains)]
        if intercept:
            for c in range(chains):
                out[c].update(s.fetch_intercept(0, c, trace=T))
        info = s.info()
    return out, info


KEYS = ("x", "mean", "var", "tau_trace", "sigma2_trace")


@pytest.mark.parametrize("chains", [1, 2, 3, 8])
@pytest.mark.parametrize("name", sorted(FIELDS) + VOLUMES, ids=str)
def test_parity_with_the_oracle(name, chains):
    f = FIELDS[name]() if name in FIELDS else _volume(name)
    one, _ = _run(f, chains, [(1, True)])
    st, _ = run_oracle(f, chains, 1, seed=31, stream=0)
    assert max(relerr(one[c]["x"], st.x[c]) for c in range(chains)) <= TOL_FP32_1
    T = 40
    res, info = _run(f, chains, [(T, True)], burn_in=15, prior=g.PRIOR_PCAR, rho=0.9, intercept=chains == 3,
                     graph_sweeps=16)
    assert info["sweeps_done"] == T and info["accumulated"] == T - 15 and info["wait_timeouts"] == 0
    st, out = run_oracle(f, chains, T, seed=31, stream=0, burn_in=15, prior="pcar", rho=0.9, intercept=chains == 3)
    for c in range(chains):
        assert relerr(res[c]["x"], st.x[c]) <= TOL_FP32_1000
        assert relerr(res[c]["mean"], st.mean[c]) <= TOL_FP32_1000
        assert trace_relerr(res[c]["tau_trace"], out["tau_trace"][c]) <= TOL_FP32_1000
        assert trace_relerr(res[c]["sigma2_trace"], out["sigma2_trace"][c]) <= TOL_FP32_1000
        if chains == 3:
            assert relerr(res[c]["beta0_trace"], out["beta0_trace"][c]) <= TOL_FP32_1000


@pytest.mark.parametrize("chains,dims", UNITS)
def test_units_per_thread(chains, dims):
    f = _volume(dims)
    res, _ = _run(f, chains, [(3, True)], intercept=chains == 2)
    st, out = run_oracle(f, chains, 3, seed=31, stream=0, intercept=chains == 2, burn_in=0)
    for c in range(chains):
        assert relerr(res[c]["x"], st.x[c]) <= TOL_FP32_1000
        assert relerr(res[c]["mean"], st.mean[c]) <= TOL_FP32_1000
        assert trace_relerr(res[c]["tau_trace"], out["tau_trace"][c]) <= TOL_FP32_1000


@pytest.mark.parametrize("name", ["delaunay_1000", "star_700", (17, 13, 11)], ids=str)
@pytest.mark.parametrize("thin", [1, 3])
def test_any_cut_into_launches_is_the_same_bit_for_bit(name, thin):
    f = FIELDS[name]() if name in FIELDS else _volume(name)
    ref, _ = _run(f, 3, [(150, True)], burn_in=20, thin=thin)
    for kw in ({"graph_sweeps": 7}, {"graph_sweeps": 128}):
        got, _ = _run(f, 3, [(1, True), (148, True), (1, True)], burn_in=20, thin=thin, **kw)
        for c in range(3):
            for key in KEYS:
                assert np.array_equal(got[c][key], ref[c][key]), key


@pytest.mark.parametrize("name", ["delaunay_1000", "delaunay_33000", (20, 24, 28), (60, 60, 61)], ids=str)
def test_agrees_with_a_launch_per_colour(name):
    f = FIELDS[name]() if name in FIELDS else _volume(name)
    calls = [(5, True), (3, False), (12, True)]
    a, ia = _run(f, 4, calls, burn_in=4, thin=2)
    b, ib = _run(f, 4, calls, burn_in=4, thin=2, flags=g.FLAG_NO_RESIDENT)
    assert ia["accumulated"] == ib["accumulated"] and ia["sweeps_done"] == ib["sweeps_done"]
    for c in range(4):
        for key in KEYS:
            assert relerr(a[c][key], b[c][key]) <= TOL_FP32_1000, key


@pytest.mark.parametrize("name", ["delaunay_1000", (17, 13, 11)], ids=str)
def test_barrier_timeout_reports_and_poisons(name):
    f = FIELDS[name]() if name in FIELDS else _volume(name)
    with g.Sampler([f], precision=g.FP32, chains=2, seed=3, flags=g.FLAG_TEST_STALL) as s:
        s.sweep(10)
        with pytest.raises(g.GmrfError) as e:
            s.fetch(0, 0)
        assert e.value.status == g.E_TIMEOUT
        with pytest.raises(g.GmrfError) as e:
            s.sweep(1)
        assert e.value.status == g.E_STATE
    a, info = _run(f, 2, [(10, True)])
    b, _ = _run(f, 2, [(10, True)], flags=g.FLAG_NO_RESIDENT)
    assert info["wait_timeouts"] == 0
    assert relerr(a[0]["x"], b[0]["x"]) <= TOL_FP32_1000
