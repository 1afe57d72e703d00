"""The multi-step kernel of small lattices (the AUTO geometry source takes it where a lattice or
ensemble fits) against the kernels that launch once per step (geom_mode TABLE; an ensemble with
a launch shape of the caller's) and the FP64 oracle, at the sizes where its boxes can go wrong:
axes one or two nodes long, boxes that span a periodic axis or end ragged, the largest lattice
that fits and the first that does not, ensembles that take several turns, sources in and
between boxes, captured and concurrent launches.

Tolerances: FP64 1e-11 of the largest population, as in the other parity tests (reordered sums
over at most 140 steps); 32- and 16-bit storage repeats the per-step kernels' operations, so its
populations are equal."""
import math
import threading

import numpy as np
import pytest

import lbw_workloads as W
import oracle

pytestmark = pytest.mark.gpu

CART = dict(kind=W.KIND_CARTESIAN, h=(1, 1, 1), x0=(0, 0, 0), c=0.4)
SPECS = {
    "disk": W.disk(37, 181),                       # ragged boxes in two directions
    "disk64": W.disk(33, 128),                     # a tile kernel's lattice
    "cylinder": W.cylinder(30, 57, 41),
    "trumpet": W.trumpet(20, 70, 40),              # coupled q1 and q3
    "torus": W.torus(20, 50, 33),                  # periodic q3
    "damped": W.cylinder(20, 40, 30).with_(damping=0.65, bc=(1, 3, 0, 0, 1, 3)),
    "walls": W.GridSpec(n=(24, 41, 20), bc=(1, 2, 2, 1, 3, 1), **CART),
    "periodic": W.GridSpec(n=(25, 40, 21), bc=(0,) * 6, **CART),
    "point": W.GridSpec(n=(1, 1, 1), bc=(0,) * 6, **CART),
    "line": W.GridSpec(n=(1, 70, 1), bc=(0,) * 6, **CART),
    "two": W.cylinder(2, 33, 2),
}
PRECS = {"f64": W.PREC_F64, "f32": W.PREC_F32, "f16": W.PREC_F16S, "bf16": W.PREC_BF16S}


def _run(spec, steps, source=None, mode=W.GEOM_AUTO):
    from paper_1705_01801_gb300 import lbw
    g = lbw.Grid(spec.with_(geom_mode=mode))
    g.init(W.pulses(spec, 1, 2, margin=0))
    g.set_probes(W.probes(spec, 1, 3, margin=0), 140)
    if source is not None:
        n1, n2, n3 = spec.n
        g.set_sources([[n1 // 2, j, n3 // 2] for j in range(n2)], kind=source, amp=0.7, omega=0.13)
    for n in steps:
        g.step(n)
    out = g.get_f(), g.read_probes()
    g.close()
    return out


@pytest.mark.parametrize("prec", list(PRECS))
@pytest.mark.parametrize("name", list(SPECS))
def test_matches_the_step_by_step_kernels(name, prec):
    spec = SPECS[name].with_(prec=PRECS[prec])
    tol = {"f64": 1e-11}.get(prec, 0.0)
    for source in (None, 0, 1) if name in ("cylinder", "damped", "disk64") else (None,):
        f, p = _run(spec, (1, 2, 130), source)
        ft, pt = _run(spec, (133,), source, W.GEOM_TABLE)
        np.testing.assert_allclose(f, ft, rtol=0, atol=tol * np.abs(ft).max())
        np.testing.assert_allclose(p, pt, rtol=0, atol=10 * tol * np.abs(pt).max())


@pytest.mark.parametrize("name", list(SPECS))
def test_matches_the_oracle(name):
    spec = SPECS[name]
    f, _ = _run(spec.with_(prec=W.PREC_F64), (40,))
    o = oracle.OracleGrid(spec)
    o.init(W.pulses(spec, 1, 2, margin=0))
    o.step(40)
    fo = o.get_f()
    np.testing.assert_allclose(f, fo, rtol=0, atol=1e-11 * np.abs(fo).max())


@pytest.mark.parametrize("n", [(64, 128, 72), (64, 128, 76), (80, 120, 64), (80, 120, 66)])
def test_at_the_capacity(n):
    """Lattices around the 152 x 4096 FP32 nodes that the SMs hold."""
    spec = W.cylinder(*n)
    f, _ = _run(spec, (20,))
    ft, _ = _run(spec, (20,), mode=W.GEOM_TABLE)
    np.testing.assert_array_equal(f, ft)


@pytest.mark.parametrize("prec", list(PRECS))
def test_ensemble_in_several_turns(prec):
    """Members and sources of their own over more nodes than one turn holds, then the same
    ensemble on the kernel that launches once per step."""
    from paper_1705_01801_gb300 import lbw
    pipe = W.GridSpec(kind=W.KIND_CYLINDRICAL, n=(20, 3, 100), h=(1.2, 2 * math.pi / 3, 1.0), x0=(1.0, 0, 0), c=0.1,
                      damping=0.9, prec=PRECS[prec], bc=(1, 1, 0, 0, 1, 3))
    specs = [pipe.with_(n=(20, 3, 100 - m % 7)) for m in range(130)]
    src = np.array([[[0, j, 0] for j in range(3)] + [[5, 1, 80]]] * len(specs))
    omega = np.linspace(0.01, 0.2, len(specs))
    probes = np.array([[[3, 0, 10], [19, 2, 60]]] * len(specs))
    out = []
    for shape in (None, (16, 16, 2)):
        b = lbw.Batch(specs)
        if shape:
            b.set_shape(*shape)
        b.init([np.zeros((0, 5))] * len(specs))
        b.set_probes(probes, 90)
        b.set_sources(src, omega)
        b.step(3)
        b.step(87)
        out.append((b.read_probes(), b.get_f(0), b.get_f(77), b.get_f(129)))
        b.close()
    tol = {"f64": 1e-11}.get(prec, 0.0)
    for x, y in zip(*out):
        np.testing.assert_allclose(x, y, rtol=0, atol=tol * np.abs(y).max())


def test_captured_and_concurrent_launches():
    """A user's graph around a few steps replays them, and lattices stepped from several threads
    on streams of their own keep the results of a lone run."""
    import torch
    from paper_1705_01801_gb300 import lbw
    spec = W.cylinder(40, 57, 41)
    pl = W.pulses(spec, 2, 1)
    alone, _ = _run_plain(spec, pl, 600)
    s = torch.cuda.Stream()
    g = lbw.Grid(spec, stream=lbw.ctypes.c_void_p(s.cuda_stream))
    g.init(pl)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        g.step(20)
    g.init(pl)
    with torch.cuda.stream(s):
        for _ in range(30):
            graph.replay()
    assert np.array_equal(g.get_f(), alone)
    g.close()
    got = [None] * 6

    def work(k):
        got[k] = _run_plain(spec, pl, 600)[0]

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(got))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert all(np.array_equal(f, alone) for f in got)


def _run_plain(spec, pl, steps):
    from paper_1705_01801_gb300 import lbw
    g = lbw.Grid(spec)
    g.init(pl)
    for _ in range(steps // 50):
        g.step(50)
    out = g.get_f(), g.step_count()
    g.close()
    return out
