"""The tall full-row tile of FP32 ensembles and ragged lattices (one block per SM): row counts on
both sides of one tile (34 rows at most), (n1 - 1) a multiple of the rows, two rows, odd and narrow
q2 extents, segments of one to all planes, every q1 and q3 face, probes.

FP32: 2e-5 of the largest population and ten times that for the probes, as in the other parity
tests.  Single ragged lattices of 720,000 nodes, past the multi-step kernel, on both sides of
the tall tile's widest row (242 columns)."""
import numpy as np
import pytest

import lbw_workloads as W
import oracle

pytestmark = pytest.mark.gpu


def _box(n, bc):
    return W.GridSpec(kind=W.KIND_CARTESIAN, n=n, h=(1, 1, 1), x0=(0, 0, 0), c=0.4, bc=bc, prec=W.PREC_F32)


SPECS = [
    _box((2, 32, 20), (1, 2, 0, 0, 3, 1)),
    _box((34, 33, 30), (2, 1, 0, 0, 0, 0)),                       # one tile
    W.cylinder(35, 37, 25).with_(prec=W.PREC_F32),                # two tiles
    W.cylinder(61, 16, 9).with_(prec=W.PREC_F32, bc=(1, 3, 0, 0, 1, 3), damping=0.7),
    W.torus(21, 96, 40).with_(prec=W.PREC_F32),
    _box((41, 95, 17), (3, 1, 0, 0, 2, 2)),
]


@pytest.mark.parametrize("lz", [1, 7, 64])
def test_matches_oracle(lz):
    from paper_1705_01801_gb300 import lbw
    b = lbw.Batch(SPECS)
    pulses = [W.pulses(s, 4, 2) for s in SPECS]
    probes = np.stack([[[0, 0, 0], [s.n[0] - 1, s.n[1] - 1, s.n[2] - 1], [s.n[0] // 2, 5, s.n[2] // 2]] for s in SPECS])
    b.init(pulses)
    b.set_probes(probes, 10)
    b.set_shape(0, lz, 1)
    b.step(3)
    b.step(7)
    series = np.asarray(b.read_probes())
    for m, s in enumerate(SPECS):
        o = oracle.OracleGrid(s)
        o.init(pulses[m])
        o.set_probes(probes[m], 10)
        o.step(10)
        fo, so = o.get_f(), o.read_probes()
        np.testing.assert_allclose(b.get_f(m), fo, rtol=0, atol=2e-5 * np.abs(fo).max())
        np.testing.assert_allclose(series[m], so, rtol=0, atol=2e-4 * np.abs(fo).max())
        o.close()
    b.close()


@pytest.mark.parametrize("n", [(90, 200, 40), (75, 242, 40), (75, 244, 40)])
def test_wide_rows(n):
    from paper_1705_01801_gb300 import lbw
    spec = W.cylinder(*n).with_(prec=W.PREC_F32, bc=(1, 3, 0, 0, 2, 1), damping=0.8)
    g, o = lbw.Grid(spec), oracle.OracleGrid(spec)
    for s in (g, o):
        s.init(W.pulses(spec, 5, 3))
        s.step(8)
    fo = o.get_f()
    np.testing.assert_allclose(g.get_f(), fo, rtol=0, atol=2e-5 * np.abs(fo).max())
    g.close()
    o.close()
