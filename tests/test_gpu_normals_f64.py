"""FP64 normals (fixed point, normals_f64.cuh) against Box-Muller in extended precision."""
import numpy as np
import pytest

from paper_1702_05518_gb300 import gmrf as g

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1702_05518_gb300 import build

    build.build()


def _box_muller(a, b):
    ld = np.longdouble
    pi = ld("3.14159265358979323846264338327950288419716939937510")
    u = (a.astype(ld) + ld(0.5)) / ld(2) ** 32
    v = ((~a).astype(ld) + ld(0.5)) / ld(2) ** 32  # 1 - u
    r = np.sqrt(-2 * np.where(u > ld(0.5), np.log1p(-v), np.log(u)))
    s = b + np.uint32(0x20000000)
    d = ((s & np.uint32(0x3FFFFFFF)).astype(ld) + ld(0.5)) / ld(2) ** 30 - ld(0.5)
    c, n = np.cos(d * pi / 2), np.sin(d * pi / 2)
    q = s >> np.uint32(30)
    return (r * np.choose(q, [c, -n, -c, n]), r * np.choose(q, [n, c, -n, -c]))


@pytest.mark.parametrize("seed", [1, 2])
def test_fp64_normals_to_the_last_place(seed):
    # every intermediate value has a relative error below 2^-57 (a sixteenth of a last place), one
    # rounding (half a last place) at the end
    n = 1 << 18
    w = np.asarray(g.philox_words(seed, 3, 5, 0, n), np.uint32).reshape(n, 4)
    want = [*_box_muller(w[:, 0], w[:, 1]), *_box_muller(w[:, 2], w[:, 3])]
    for chain in range(4):
        got = g.site_normals(seed, 3, 5, chain, n, g.FP64, lanes=4)
        ulp = np.spacing(np.abs(want[chain]).astype(np.float64))
        assert np.max(np.abs(got.astype(np.longdouble) - want[chain]) / ulp) <= 0.75
