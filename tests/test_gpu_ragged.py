"""Single lattices whose q2 extent is no multiple of the tile width, large enough to leave the
multi-step kernel: they step on the ensemble's tile kernels.  Odd, even and ragged extents on
both sides of the full-row tile's limit, tiles that start at q1 = -1, every q1 and q3 face rule,
sources next to the periodic wrap, probes, checkpoints.

Tolerances as in the other parity tests: FP64 1e-11, FP32 2e-5 of the largest population."""
import numpy as np
import pytest

import lbw_workloads as W
import oracle

pytestmark = pytest.mark.gpu

SPECS = {
    "narrow": W.cylinder(60, 37, 300),              # tall full-row tiles, an odd row
    "row100": W.cylinder(91, 100, 80),              # (n1 - 1) a multiple of the tile rows
    "wide": W.cylinder(71, 130, 75),                # 64-column tiles with a 2-column remainder
    "trumpet": W.trumpet(43, 150, 106),             # coupled q1 and q3
    "torus": W.torus(50, 90, 150),                  # periodic q3
    "damped": W.cylinder(64, 101, 105).with_(damping=0.65, bc=(1, 3, 0, 0, 3, 1)),
}


@pytest.mark.parametrize("prec,tol", [(W.PREC_F64, 1e-11), (W.PREC_F32, 2e-5)], ids=["f64", "f32"])
@pytest.mark.parametrize("name", list(SPECS))
def test_matches_oracle(name, prec, tol):
    from paper_1705_01801_gb300 import lbw
    spec = SPECS[name].with_(prec=prec)
    assert spec.nodes > 640000
    n1, n2, n3 = spec.n
    pl, pr = W.pulses(spec, 5, 3), np.array([[0, 0, 0], [n1 - 1, n2 - 1, n3 - 1], [n1 // 2, n2 // 2, n3 // 3]])
    src = [[n1 // 3, q2, n3 // 2] for q2 in (0, 1, n2 // 2, n2 - 2, n2 - 1)]
    g, o = lbw.Grid(spec), oracle.OracleGrid(spec)
    for s in (g, o):
        s.init(pl)
        s.set_probes(pr, 12)
        s.set_sources(src, kind=0, amp=0.3, omega=0.3)
        s.step(7)
    f = g.get_f()
    g.set_f(f)                       # a checkpoint goes back into the padded rows
    assert np.array_equal(g.get_f(), f)
    g.step(5)
    o.step(5)
    fo, so = o.get_f(), o.read_probes()
    np.testing.assert_allclose(g.get_f(), fo, rtol=0, atol=tol * np.abs(fo).max())
    np.testing.assert_allclose(g.read_probes(), so, rtol=0, atol=10 * tol * np.abs(fo).max())
    Po = o.get_P()
    np.testing.assert_allclose(g.get_P(), Po, rtol=0, atol=10 * tol * np.abs(Po).max())
    g.close()
    o.close()


def test_chains_equal_single_steps():
    from paper_1705_01801_gb300 import lbw
    spec = SPECS["wide"]
    out = []
    for counts in ((130,), (1,) * 130):
        g = lbw.Grid(spec)
        g.init(W.pulses(spec, 5, 1))
        for n in counts:
            g.step(n)
        out.append(g.get_f())
        g.close()
    assert np.array_equal(*out)
