"""The kernels that launch once per step, on lattices that the multi-step kernel would take
(geom_mode TABLE keeps them): parity with the oracle, graph chains against single launches, sources,
thin lattices, checkpoints, the Cartesian schemes and the injected timeout of the tile kernel's
waits; and single ragged lattices on the ensemble kernels, which TABLE does not decide.

Tolerances as in the tests of the same names without "per step": FP64 1e-11 of the largest
population, FP32 2e-5, probes ten times that; equal bits where only the launches differ."""
import numpy as np
import pytest

import lbw_workloads as W
import oracle
from test_gpu_parity import DEGENERATE, SPECS, _run_both

pytestmark = pytest.mark.gpu

STORAGE = {"f64": W.PREC_F64, "f32": W.PREC_F32, "f16s": W.PREC_F16S, "bf16s": W.PREC_BF16S}
# beyond what the SMs hold at a time, with a q2 extent that no tile width divides
RAGGED = {"rows": W.cylinder(66, 100, 100), "columns": W.cylinder(40, 250, 66), "tall": W.cylinder(60, 200, 54)}
# tall tiles and blocks cut into pieces (see test_gpu_tile_cuts.py)
TALL = {"16 rows": W.cylinder(100, 128, 64), "12 rows": W.torus(61, 256, 24).with_(prec=W.PREC_F16S)}


def _table(spec, prec):
    return spec.with_(prec=prec, geom_mode=W.GEOM_TABLE)


@pytest.mark.parametrize("prec,tol", [(W.PREC_F64, 1e-11), (W.PREC_F32, 2e-5)], ids=["f64", "f32"])
@pytest.mark.parametrize("name", list(SPECS))
def test_populations_match_oracle_per_step(name, prec, tol):
    g, o, _, _ = _run_both(_table(SPECS[name], prec), 150, seed=11)
    fo, so = o.get_f(), o.read_probes()
    np.testing.assert_allclose(g.get_f(), fo, rtol=0, atol=tol * np.abs(fo).max())
    np.testing.assert_allclose(g.read_probes(), so, rtol=0, atol=10 * tol * np.abs(so).max())


@pytest.mark.parametrize("storage", list(STORAGE))
@pytest.mark.parametrize("name", ["cylinder", "cylinder_wide", "cylinder_unstaged", "torus", "rows", "columns", "tall"])
def test_graph_chain_equals_single_launches_per_step(name, storage):
    """131 steps: two chains of 64 and three launches against 131 launches."""
    from paper_1705_01801_gb300 import lbw
    spec = _table({**SPECS, **RAGGED}[name], STORAGE[storage])
    pl, pr = W.pulses(spec, 3, 1, sigma=2.5), W.probes(spec, 3, 4, margin=0)
    out = []
    for steps in ((131,), (1,) * 131):
        g = lbw.Grid(spec)
        g.init(pl)
        g.set_probes(pr, 131)
        for n in steps:
            g.step(n)
        out.append((g.get_f(), g.read_probes()))
        g.close()
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("prec,tol", [(W.PREC_F64, 1e-11), (W.PREC_F32, 2e-5)], ids=["f64", "f32"])
@pytest.mark.parametrize("kind", [0, 1], ids=["P", "Jz"])
@pytest.mark.parametrize("name", ["cylinder", "cylinder_unstaged", "cylinder_wide", "rows", "columns"])
def test_sources_match_oracle_per_step(name, kind, prec, tol):
    from paper_1705_01801_gb300 import lbw
    large = name in RAGGED
    spec = _table({**SPECS, **RAGGED}[name], prec)
    src = [[i, j, 2] for i in (range(spec.n[0]) if kind else (0,)) for j in range(spec.n[1])]
    pl, pr, steps = W.pulses(spec, 5, 1, sigma=2.5, margin=2), W.probes(spec, 5, 4, margin=0), 66 if large else 130
    g, o = lbw.Grid(spec), oracle.OracleGrid(spec)
    for s in (g, o):
        s.init(pl)
        s.set_sources(src, kind=kind, amp=0.8, omega=0.21)
        s.set_probes(pr, steps)
        s.step(steps)
    fo, so = o.get_f(), o.read_probes()
    np.testing.assert_allclose(g.get_f(), fo, rtol=0, atol=tol * np.abs(fo).max())
    np.testing.assert_allclose(g.read_probes(), so, rtol=0, atol=10 * tol * np.abs(so).max())
    g.close()


@pytest.mark.parametrize("name", list(DEGENERATE))
def test_degenerate_extents_match_oracle_per_step(name):
    from paper_1705_01801_gb300 import lbw
    n, bc = DEGENERATE[name]
    spec = W.GridSpec(kind=W.KIND_CARTESIAN, n=n, h=(1, 1, 1), x0=(0, 0, 0), c=0.4, bc=bc, damping=0.8,
                      prec=W.PREC_F64, geom_mode=W.GEOM_TABLE)
    f = np.random.default_rng(sum(n)).standard_normal((7, n[2], n[0], n[1]))
    q = [[n[0] - 1, n[1] - 1, n[2] - 1], [0, 0, 0]]
    g, o = lbw.Grid(spec), oracle.OracleGrid(spec)
    for s in (g, o):
        s.set_f(f)
        s.set_probes(q, 40)
        s.step(40)
    fo, so = o.get_f(), o.read_probes()
    np.testing.assert_allclose(g.get_f(), fo, rtol=0, atol=1e-11 * np.abs(fo).max())
    np.testing.assert_allclose(g.read_probes(), so, rtol=0, atol=1e-11 * np.abs(so).max())
    g.close()


@pytest.mark.parametrize("storage", list(STORAGE))
@pytest.mark.parametrize("name", ["cylinder", "cylinder_wide", "cylinder_unstaged", "rows", "columns"])
def test_split_run_equals_straight_run_per_step(name, storage):
    from paper_1705_01801_gb300 import lbw
    spec = _table({**SPECS, **RAGGED}[name], STORAGE[storage])
    pl, pr = W.pulses(spec, 5, 2, sigma=2.5, margin=3), W.probes(spec, 5, 3)
    a = lbw.Grid(spec)
    a.init(pl)
    a.step(37)
    ckpt = a.get_f()
    a.set_probes(pr, 53)
    a.step(53)
    c = lbw.Grid(spec)
    c.set_f(ckpt)
    c.set_probes(pr, 53)
    c.step(53)
    np.testing.assert_array_equal(c.get_f(), a.get_f())
    np.testing.assert_array_equal(c.read_probes(), a.read_probes())
    a.close()
    c.close()


@pytest.mark.parametrize("prec,tol", [(W.PREC_F64, 1e-11), (W.PREC_F32, 2e-5)], ids=["f64", "f32"])
@pytest.mark.parametrize("eq", [W.EQ_MOMENT_MATCHING, W.EQ_HERMITE], ids=["moment-matching", "hermite"])
@pytest.mark.parametrize("n,q2", [((9, 40, 11), (2, 3)), ((9, 128, 11), (2, 3)), ((66, 100, 100), (0, 0)),
                                  ((40, 250, 66), (0, 0))],
                         ids=["pipelined", "tiled", "ragged rows", "ragged columns"])
def test_cartesian_equilibria_match_oracle_per_step(n, q2, eq, prec, tol):
    from paper_1705_01801_gb300 import lbw
    spec = W.GridSpec(kind=W.KIND_CARTESIAN, n=n, h=(1, 1, 1), x0=(0, 0, 0), c=0.35, equilibrium=eq, prec=prec,
                      damping=0.9, bc=(W.BC_FREE, W.BC_BOUNCE, *q2, W.BC_BOUNCE, W.BC_ANTIBOUNCE), geom_mode=W.GEOM_TABLE)
    steps = 140 if spec.nodes < 10 ** 5 else 30
    pl, pr = W.pulses(spec, 33, 2, sigma=2.0, random_phase=True, margin=2), W.probes(spec, 33, 3, margin=0)
    g, o = lbw.Grid(spec), oracle.OracleGrid(spec)
    for s in (g, o):
        s.init(pl)
        s.set_sources([[4, n[1] // 2, 5]], kind=0, amp=0.3, omega=0.2)
        s.set_probes(pr, steps)
        s.step(steps)
    fo, so = o.get_f(), o.read_probes()
    np.testing.assert_allclose(g.get_f(), fo, rtol=0, atol=tol * np.abs(fo).max())
    # of the populations, not of the series: after 30 steps some probes have seen 1e-30 and less, where the
    # pulses' cut-off at 2e-35 shows
    np.testing.assert_allclose(g.read_probes(), so, rtol=0, atol=10 * tol * np.abs(fo).max())
    g.close()


@pytest.mark.parametrize("spec", [_table(W.cylinder(13, 128, 10), p) for p in STORAGE.values()]
                         + [s.with_(geom_mode=W.GEOM_TABLE) for s in TALL.values()],
                         ids=list(STORAGE) + list(TALL))
def test_injected_wait_timeout_per_step(spec):
    """The tile kernel's consumers wait on a barrier that nothing completes, for a few hundred tries; the
    producer stops and its copies land, launches behind it (a graph chain too) find the flag, the calls
    that synchronise report it, and lbw_init brings back a state that runs like a fresh one."""
    from paper_1705_01801_gb300 import lbw
    pl, pr = W.pulses(spec, 4, 1, sigma=2.5, margin=3), W.probes(spec, 4, 2)
    fresh = lbw.Grid(spec)
    fresh.init(pl)
    fresh.step(80)
    want = fresh.get_f()
    fresh.close()
    g = lbw.Grid(spec)
    g.init(pl)
    g.set_probes(pr, 100)
    g.step(4)
    g.read_probes()  # no flag before the injection
    lbw.lbw_inject_wait_timeout(g.handle)
    g.step(70)  # a chain of 64 and six launches
    for call in (g.read_probes, lambda: g.spectrum(-1, 2), g.get_P, g.get_f):
        with pytest.raises(lbw.LbwError) as e:
            call()
        assert e.value.status == lbw.LBW_ETIMEOUT, str(e.value)
    g.init(pl)
    g.step(80)
    np.testing.assert_array_equal(g.get_f(), want)
    g.close()


@pytest.mark.parametrize("prec,tol", [(W.PREC_F64, 1e-11), (W.PREC_F32, 2e-5)], ids=["f64", "f32"])
@pytest.mark.parametrize("spec", [
    W.disk(1000, 701), W.disk(2700, 250),
    W.GridSpec(kind=W.KIND_CARTESIAN, n=(900, 801, 1), h=(1, 1, 1), x0=(0, 0, 0), c=0.4, bc=(1, 2, 0, 0, 1, 3)),
    W.GridSpec(kind=W.KIND_CARTESIAN, n=(130, 2601, 2), h=(1, 1, 1), x0=(0, 0, 0), c=0.4, bc=(3, 1, 0, 0, 2, 1)),
    W.GridSpec(kind=W.KIND_CARTESIAN, n=(2, 300, 1200), h=(1, 1, 1), x0=(0, 0, 0), c=0.4, bc=(3, 1, 0, 0, 0, 0))],
    ids=["disk", "disk rows", "plane", "two planes", "two rows"])
def test_large_thin_ragged_lattices_match_oracle(spec, prec, tol):
    """Ragged lattices of one or two planes (or rows) beyond the multi-step kernel's capacity."""
    from paper_1705_01801_gb300 import lbw
    spec = spec.with_(prec=prec)
    pl, pr = W.pulses(spec, 7, 6, sigma=9.0, random_phase=True, margin=0), W.probes(spec, 7, 5, margin=0)
    g, o = lbw.Grid(spec), oracle.OracleGrid(spec)
    for s in (g, o):
        s.init(pl)
        s.set_probes(pr, 25)
        s.step(25)
    fo, so = o.get_f(), o.read_probes()
    np.testing.assert_allclose(g.get_f(), fo, rtol=0, atol=tol * np.abs(fo).max())
    np.testing.assert_allclose(g.read_probes(), so, rtol=0, atol=10 * tol * np.abs(fo).max())
    g.close()
