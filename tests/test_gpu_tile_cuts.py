"""The tile kernel's tiles and their division into blocks: tile heights 5, 7, 12, 13 and 16,
sizes whose last blocks are pieces of the remaining (tile, segment) items, a halo row on the
q1 = n1 - 1 face ((n1 - 1) a multiple of a 16-bit tile's rows), a last tile of few lattice rows,
every kind of face.

One device step from a shared state that the storage holds exactly against one FP64 oracle step
at every node; FP32: 1e-6 of the largest population, 16-bit: half an ulp of the stored value more
(FP16 2^-11, BF16 2^-8), as in the full-size parity test."""
import numpy as np
import pytest

import lbw_workloads as W
import oracle

pytestmark = pytest.mark.gpu

RTOL = {W.PREC_F32: 0.0, W.PREC_F16S: 2.0 ** -11, W.PREC_BF16S: 2.0 ** -8}
BOX = dict(h=(1, 1, 1), x0=(0, 0, 0), c=0.4, damping=0.7)
SPECS = {
    "torus-bf16": W.torus(101, 1024, 16).with_(prec=W.PREC_BF16S),
    "cylinder-f16": W.cylinder(161, 640, 16).with_(prec=W.PREC_F16S),
    "walls-f16": W.GridSpec(kind=W.KIND_CARTESIAN, n=(161, 640, 16), bc=(3, 1, 1, 2, 2, 3), prec=W.PREC_F16S, **BOX),
    "free-f16": W.GridSpec(kind=W.KIND_CARTESIAN, n=(101, 1024, 16), bc=(2, 3, 3, 3, 0, 0), prec=W.PREC_F16S, **BOX),
    "torus-f32": W.torus(192, 768, 5).with_(prec=W.PREC_F32),
    "walls-f32": W.GridSpec(kind=W.KIND_CARTESIAN, n=(121, 640, 13), bc=(1, 3, 3, 1, 2, 2), prec=W.PREC_F32, **BOX),
    "rows5-f16": W.cylinder(157, 512, 16).with_(prec=W.PREC_F16S),
    "rows12-face-f16": W.GridSpec(kind=W.KIND_CARTESIAN, n=(61, 128, 24), bc=(2, 1, 2, 3, 1, 1), prec=W.PREC_F16S, **BOX),
    "rows12-pieces-bf16": W.torus(196, 640, 16).with_(prec=W.PREC_BF16S),
    "rows13-f16": W.cylinder(37, 128, 40).with_(prec=W.PREC_F16S),
    "rows13-face-bf16": W.GridSpec(kind=W.KIND_CARTESIAN, n=(196, 128, 9), bc=(1, 3, 0, 0, 3, 2), prec=W.PREC_BF16S, **BOX),
    "rows16-face-f16": W.GridSpec(kind=W.KIND_CARTESIAN, n=(145, 192, 5), bc=(3, 2, 1, 1, 0, 0), prec=W.PREC_F16S, **BOX),
    "rows16-pieces-f32": W.cylinder(197, 384, 16).with_(prec=W.PREC_F32),
    "rows16-f32": W.GridSpec(kind=W.KIND_CARTESIAN, n=(29, 64, 5), bc=(2, 1, 3, 2, 3, 1), prec=W.PREC_F32, **BOX),
}


@pytest.mark.parametrize("name", list(SPECS))
def test_one_step(name):
    from paper_1705_01801_gb300 import lbw
    spec = SPECS[name].with_(geom_mode=1)  # a launch per step
    rng = np.random.default_rng(3)
    shape = (7, spec.n[2], spec.n[0], spec.n[1])
    if spec.prec == W.PREC_F32:
        f = rng.standard_normal(shape, dtype=np.float32).astype(np.float64)
    else:
        w = np.array([0.25] + [0.125] * 6)[:, None, None, None]
        f = rng.integers(-64, 65, size=shape).astype(np.float64) / 64.0 * w
    g, o = lbw.Grid(spec), oracle.OracleGrid(spec)
    for s in (g, o):
        s.set_f(f)
        s.step(1)
    fo = o.get_f()
    np.testing.assert_allclose(g.get_f(), fo, rtol=RTOL[spec.prec], atol=1e-6 * np.abs(fo).max())
    g.close()
    o.close()


@pytest.mark.parametrize("n2", [64, 40], ids=["tile", "full-row"])
def test_many_probes_of_a_tile(n2):
    """64 probes in the tile and ensemble kernels: several in a plane, planes 256 apart, both ends
    of a row, every row; FP32 as in the other parity tests (2e-5, probes ten times that)."""
    from paper_1705_01801_gb300 import lbw
    spec = W.GridSpec(kind=W.KIND_CARTESIAN, n=(9, n2, 600), bc=(1, 2, 0, 0, 3, 1), prec=W.PREC_F32, **BOX)
    q = np.array([[k % 9, (0, n2 - 1, 17, 18)[k % 4], (3, 259, 515, 599)[k // 16] - (k % 3 == 0)] for k in range(64)])
    o = oracle.OracleGrid(spec)
    o.init(W.pulses(spec, 5, 4))
    o.set_probes(q, 8)
    o.step(10)
    so, fmax = o.read_probes(), np.abs(o.get_f()).max()
    o.close()
    if n2 == 64:
        g = lbw.Grid(spec.with_(geom_mode=1))
        g.init(W.pulses(spec, 5, 4))
        g.set_probes(q, 8)
        g.step(10)
        series = [g.read_probes()]
        g.close()
    else:
        b = lbw.Batch([spec, spec])
        b.init([W.pulses(spec, 5, 4)] * 2)
        b.set_probes(np.stack([q, q]), 8)
        series = []
        for cps in (1, 2):
            b.init([W.pulses(spec, 5, 4)] * 2)
            b.set_shape(0, 300, cps)
            b.step(10)
            series += list(b.read_probes())
        b.close()
    for s in series:
        assert np.asarray(s).shape == np.asarray(so).shape
        np.testing.assert_allclose(s, so, rtol=0, atol=2e-4 * fmax)
