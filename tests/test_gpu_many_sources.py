"""Plate sources: more source nodes than a box of the multi-step kernel keeps on chip.  The fields are
those of the kernels that launch once per step (equal in 32- and 16-bit storage, FP64 within
1e-11 of the largest population, as in the other comparisons of these kernels), and four planes of
sources do not make it slower than they are."""
import time

import numpy as np
import pytest

import lbw_workloads as W

pytestmark = pytest.mark.gpu


def _grid(spec, sources, kind):
    from paper_1705_01801_gb300 import lbw
    g = lbw.Grid(spec)
    g.init(W.pulses(spec, 1, 1, margin=0))
    n1, n2, _ = spec.n
    g.set_sources([[i % n1, i // n1 % n2, 3 + i // (n1 * n2)] for i in range(sources)], kind, 0.7, 0.13)
    return g


@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("prec", [W.PREC_F64, W.PREC_F32, W.PREC_F16S, W.PREC_BF16S])
@pytest.mark.parametrize("n,sources", [((40, 50, 30), 65), ((40, 50, 30), 4000), ((33, 64, 20), 2112), ((5, 7, 9), 200)])
def test_fields_are_those_of_single_steps(n, sources, prec, kind):
    out = []
    for mode in (W.GEOM_AUTO, W.GEOM_TABLE):
        g = _grid(W.cylinder(*n).with_(prec=prec, geom_mode=mode), sources, kind)
        for k in (1, 2, 70):
            g.step(k)
        out.append(g.get_f())
        g.close()
    tol = 1e-11 if prec == W.PREC_F64 else 0.0
    np.testing.assert_allclose(out[0], out[1], rtol=0, atol=tol * np.abs(out[1]).max())


@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("prec", [W.PREC_F64, W.PREC_F32, W.PREC_F16S, W.PREC_BF16S])
@pytest.mark.parametrize("n,members", [((24, 130, 30), 3), ((12, 64, 40), 4), ((9, 33, 50), 2)])
def test_ensembles_with_plates_that_come_and_go(n, members, prec, kind):
    """Where a plate makes launches per step the faster way, the ensemble changes to them (and their
    ghost columns) and back again."""
    from paper_1705_01801_gb300 import lbw
    spec = W.cylinder(*n).with_(prec=prec)
    plate = [[[i % n[0], i // n[0] % n[1], 3 + i // (n[0] * n[1])] for i in range(9 * n[0] * n[1])]] * members
    out = []
    for shape in (None, (7, 16, 1)):
        b = lbw.Batch([spec] * members)
        if shape:
            b.set_shape(*shape)
        b.init([W.pulses(spec, m, 2, margin=0) for m in range(members)])
        for sources in (0, 9 * n[0] * n[1], 0, 7):
            b.set_sources(np.array(plate)[:, :sources], 0.1 + 0.01 * np.arange(members), kind, 0.7)
            b.step(5)
        out.append([b.get_f(m) for m in range(members)])
        b.close()
    tol = 1e-11 if prec == W.PREC_F64 else 0.0
    for x, y in zip(*out):
        np.testing.assert_allclose(x, y, rtol=0, atol=tol * np.abs(y).max())


@pytest.mark.parametrize("n", [(128, 128, 30), (64, 128, 70), (64, 64, 100)])
def test_four_planes_of_sources_do_not_slow_it_down(n):
    """us per step, FP32, with a sine per source and one SM per box: 41 against 23 for a launch per
    step, 59 against 21, 34 against 17."""
    took = []
    for mode in (W.GEOM_AUTO, W.GEOM_TABLE):
        g = _grid(W.cylinder(*n).with_(geom_mode=mode), 4 * n[0] * n[1], 0)
        g.step(256)
        g.get_P()
        best = 1e9
        for _ in range(5):
            t = time.perf_counter()
            g.step(1024)
            g.set_probes(np.zeros((0, 3), np.int32), 0)  # synchronises
            best = min(best, time.perf_counter() - t)
        took.append(best)
        g.close()
    assert took[0] < 1.3 * took[1], took
