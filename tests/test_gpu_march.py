"""Marching warps (lattice_march.cu): sweeps of FP32 2-D lattices with the state in registers, one
launch per sweep or a batch of sweeps per cooperative launch.  Parity with the oracle (1e-5 after
one sweep, 1e-4 on states, means and traces after more) where the decomposition can go wrong: widths
around a strip's columns and their halo, row lengths of every offset to the Philox blocks, chunk ends of
both parities, images of a row or a column, one to sixteen chains; several fields in one sampler; the
sums of an extra draw.  The two forms agree bit for bit.

Single fields of one wave of tiles take the tiled kernels by default; asking for the chains per thread
the sampler would choose anyway sends them to the marching warps.
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


# A strip owns 120 columns (one chain), 60 or 56 (two; 4 and 8 neighbours); chunks of a few rows.
DIMS = [(1, 1), (1, 130), (9, 1), (2, 3), (5, 2), (7, 119), (8, 120), (9, 121), (6, 122), (11, 123), (13, 125), (4, 240),
        (33, 241), (10, 57), (17, 61), (12, 113), (40, 118), (67, 66), (131, 35)]


def _march(chains):
    return {"tuning": {"chains_per_thread": chains}} if chains <= 2 else {}


def _run(fields, chains, calls, extra=False, **kw):
    with g.Sampler(fields, precision=g.FP32, chains=chains, seed=77, trace_capacity=256, **kw) as s:
        for n in calls:
            s.sweep(n)
        if extra:
            s.hyper_update()
        T = sum(calls)
        out = [[s.fetch(f, c, trace=T) for c in range(chains)] for f in range(len(fields))]
        info = s.info()
    return out, info


def _check(f, res, chains, T, tol, stream=0, **kw):
    st, out = run_oracle(f, chains, T, seed=77, stream=stream, **kw)
    for c in range(chains):
        assert relerr(res[c]["x"], st.x[c]) <= tol
        assert trace_relerr(res[c]["tau_trace"], out["tau_trace"][c]) <= tol
        assert trace_relerr(res[c]["sigma2_trace"], out["sigma2_trace"][c]) <= tol
        if kw.get("burn_in") is not None:
            assert relerr(res[c]["mean"], st.mean[c]) <= tol
    return st


@pytest.mark.parametrize("kind", [wl.LATTICE2D_4, wl.LATTICE2D_8], ids=["4nbr", "8nbr"])
@pytest.mark.parametrize("dims", DIMS, ids=str)
@pytest.mark.parametrize("chains", [1, 2, 3, 8])
def test_parity_with_the_oracle(kind, dims, chains):
    # (single-chain 8-neighbour rows of a multiple of four take the quad kernel)
    f = wl.small_lattice(kind, dims, 9)
    one, _ = _run([f], chains, [1], flags=g.FLAG_NO_RESIDENT, **_march(chains))
    _check(f, one[0], chains, 1, TOL_FP32_1)
    kw = dict(prior=g.PRIOR_PCAR, rho=0.9) if chains != 2 else dict(intercept=True)
    res, info = _run([f], chains, [23, 8], burn_in=11, flags=g.FLAG_NO_RESIDENT, graph_sweeps=5, **kw, **_march(chains))
    assert info["accumulated"] == 20
    kw = dict(prior="pcar", rho=0.9) if chains != 2 else dict(intercept=True)
    _check(f, res[0], chains, 31, TOL_FP32_1000, burn_in=11, **kw)


@pytest.mark.parametrize("kind,dims,chains", [(wl.LATTICE2D_4, (200, 363), 1), (wl.LATTICE2D_8, (201, 362), 1),
                                              (wl.LATTICE2D_8, (150, 171), 4), (wl.LATTICE2D_4, (150, 171), 8),
                                              (wl.LATTICE2D_4, (1500, 1999), 1), (wl.LATTICE2D_8, (97, 60), 16),
                                              (wl.LATTICE2D_8, (700, 901), 8)])
def test_batches_of_sweeps_parity(kind, dims, chains):
    f = wl.small_lattice(kind, dims, 10)
    T = 6 if dims[0] >= 700 else 40
    res, info = _run([f], chains, [T], burn_in=T // 2, graph_sweeps=16, **_march(chains))
    assert info["wait_timeouts"] == 0
    _check(f, res[0], chains, T, TOL_FP32_1000, burn_in=T // 2)


@pytest.mark.parametrize("kind,dims,chains", [(wl.LATTICE2D_4, (1500, 1999), 1), (wl.LATTICE2D_8, (901, 1510), 2),
                                              (wl.LATTICE2D_4, (41, 241), 1), (wl.LATTICE2D_8, (70, 123), 1),
                                              (wl.LATTICE2D_8, (90, 61), 2)])
def test_batches_equal_single_sweeps(kind, dims, chains):
    f = wl.small_lattice(kind, dims, 14)
    a, info = _run([f], chains, [7, 2], burn_in=3, **_march(chains))
    assert info["resident"] == 0  # not the small-lattice or tile-resident form
    b, _ = _run([f], chains, [7, 2], burn_in=3, flags=g.FLAG_NO_RESIDENT, **_march(chains))
    for c in range(chains):
        for k in ("x", "mean", "var", "tau_trace", "sigma2_trace"):
            np.testing.assert_array_equal(a[0][c][k], b[0][c][k], err_msg=k)


@pytest.mark.parametrize("chains", [1, 3])
def test_several_fields_and_graphs(chains):
    rp, ci, _ = wl.delaunay_graph(400, wl.rng(3))
    fields = [wl.small_lattice(wl.LATTICE2D_4, (37, 150), 1), wl.small_lattice(wl.LATTICE2D_8, (61, 59), 2),
              dict(wl.graph_field(rp, ci, seed=4), color_seed=5), wl.small_lattice(wl.LATTICE2D_4, (1, 9), 5),
              wl.small_lattice(wl.LATTICE2D_4, (140, 33), 6)]
    res, _ = _run(fields, chains, [20], burn_in=8, graph_sweeps=6)
    for k, f in enumerate(fields):
        _check(f, res[k], chains, 20, TOL_FP32_1000, stream=k, burn_in=8)


@pytest.mark.parametrize("kind", [wl.LATTICE2D_4, wl.LATTICE2D_8], ids=["4nbr", "8nbr"])
@pytest.mark.parametrize("chains", [1, 2, 8])
def test_sums_of_an_extra_draw(kind, chains):
    # the draw after hyper_update uses the sums of the current state: the tiled kernel's agree
    f = wl.small_lattice(kind, (45, 131), 12)
    out = []
    for tuning in (_march(chains).get("tuning"), {"fused_rows": [16, 16], "fused_cols": [32, 32], "fused_threads": [512, 512]}):
        with g.Sampler([f], precision=g.FP32, chains=chains, seed=5, flags=g.FLAG_NO_RESIDENT, prior=g.PRIOR_PCAR, rho=0.8,
                       tuning=tuning) as s:
            s.sweep(4)
            s.hyper_update()
            out.append([(s.fetch(0, c)["tau"], s.fetch(0, c)["sigma2"]) for c in range(chains)])
    assert np.allclose(out[0], out[1], rtol=1e-5, atol=0)


def test_barrier_timeout_reports_and_poisons():
    f = wl.small_lattice(wl.LATTICE2D_4, (41, 241), 13)
    with g.Sampler([f], precision=g.FP32, chains=1, seed=3, flags=g.FLAG_TEST_STALL, **_march(1)) as s:
        assert s.info()["resident"] == 0
        s.sweep(10)
        with pytest.raises(g.GmrfError) as e:
            s.fetch(0, 0)
        assert e.value.status == g.E_TIMEOUT
        with pytest.raises(g.GmrfError) as e:
            s.sweep(1)
        assert e.value.status == g.E_STATE
    res, info = _run([f], 1, [10], **_march(1))
    assert info["wait_timeouts"] == 0
    _check(f, res[0], 1, 10, TOL_FP32_1000)
