"""Initial states of lattices whose rows are short (several to a warp) or few and long (several warps
to a row), on both sides of the sizes from which the axes are tabulated and the buffer is cleared
by a memset: against the oracle's populations, and not much slower than a square lattice of as
many nodes."""
import time

import numpy as np
import pytest

import lbw_workloads as W
import oracle

pytestmark = pytest.mark.gpu

CART = dict(kind=W.KIND_CARTESIAN, h=(1, 1, 1), x0=(0, 0, 0), c=0.4)
WALLS, PERIODIC = (1, 2, 2, 1, 3, 1), (0,) * 6


def _cart(n, bc=WALLS):
    return W.GridSpec(n=n, bc=bc, **CART)


SPECS = {
    "n2=1": _cart((17, 1, 23)), "n2=3": _cart((20, 3, 35), PERIODIC), "n2=15": _cart((9, 15, 11)),
    "n2=16": _cart((7, 16, 5)), "n2=17": _cart((7, 17, 5)), "n2=33": _cart((3, 33, 2)),
    "line": _cart((1, 5000, 1), PERIODIC), "two lines": _cart((2, 40001, 1)), "long": _cart((2, 300000, 2)),
    "disk": W.disk(9, 3000), "cylinder": W.cylinder(60, 1100, 3), "torus": W.torus(5, 3, 90),
    "short": W.cylinder(300, 3, 200), "horn": W.bessel_horn(0.2, (3, 5, 700)),
}


@pytest.mark.parametrize("name", list(SPECS))
def test_initial_state_matches_oracle(name):
    """FP64: sums of up to 70 exponentials, 1e-13 of the largest population (their arguments, up to
    80, carry some 1e-14)."""
    from paper_1705_01801_gb300 import lbw
    spec = SPECS[name].with_(prec=W.PREC_F64)
    g, o = lbw.Grid(spec), oracle.OracleGrid(spec)
    for pl in (W.pulses(spec, 1, 1, margin=0), W.pulses(spec, 2, 70, sigma=1.2, margin=0, random_phase=True)):
        g.init(W.pulses(spec, 9, 3, sigma=9.0, margin=0))  # an earlier state leaves nothing behind
        g.step(3)
        g.init(pl)
        o.init(pl)
        fo = o.get_f()
        np.testing.assert_allclose(g.get_f(), fo, rtol=0, atol=1e-13 * np.abs(fo).max())
    g.close()


def _seconds(spec, pulses):
    from paper_1705_01801_gb300 import lbw
    g = lbw.Grid(spec)
    pl = W.pulses(spec, 1, pulses, margin=0)
    best = 1e9
    for _ in range(6):
        t = time.perf_counter()
        g.init(pl)  # synchronises
        best = min(best, time.perf_counter() - t)
    g.close()
    return best


@pytest.mark.parametrize("n", [(1, 1 << 20, 1), (4, 1 << 16, 4), (1000, 3, 350)])
def test_shape_does_not_set_the_time(n):
    """A warp per row would take 40 to 430 times as long on the first two and 3 times on the third."""
    assert _seconds(_cart(n), 2) < 2.5 * _seconds(_cart((1024, 1024, 1)), 2)
