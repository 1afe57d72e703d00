"""Initial states and read-outs: pulses that reach no row, one row or all of them, rows and axes of
one node, more pulses than one warp tests at a time, against the oracle's initial populations and
field; the field's finite check where only one value is not."""
import numpy as np
import pytest

import lbw_workloads as W
import oracle

pytestmark = pytest.mark.gpu

CART = dict(kind=W.KIND_CARTESIAN, h=(1, 1, 1), x0=(0, 0, 0), c=0.4)
SPECS = {
    "disk": W.disk(37, 181), "cylinder": W.cylinder(40, 33, 120), "trumpet": W.trumpet(30, 40, 60),
    "torus": W.torus(30, 40, 90), "horn": W.bessel_horn(0.2, (12, 16, 64)),
    "walls": W.GridSpec(n=(40, 21, 60), bc=(1, 2, 2, 1, 3, 1), **CART),
    "point": W.GridSpec(n=(1, 1, 1), bc=(0,) * 6, **CART),
}


@pytest.mark.parametrize("name", list(SPECS))
def test_initial_state_matches_oracle(name):
    """FP64: sums of up to 70 exponentials, 1e-13 of the largest population (their arguments, up to
    80, carry some 1e-14)."""
    from paper_1705_01801_gb300 import lbw
    spec = SPECS[name].with_(prec=W.PREC_F64)
    far = np.array([[1e4, -3e3, 500.0, 3.0, 1.0]])
    for pl in (W.pulses(spec, 1, 1, margin=0), W.pulses(spec, 2, 70, sigma=1.2, margin=0, random_phase=True),
               W.pulses(spec, 3, 2, sigma=40.0, margin=0), far, np.zeros((0, 5))):
        g, o = lbw.Grid(spec), oracle.OracleGrid(spec)
        g.init(W.pulses(spec, 9, 3, margin=0))  # an earlier state leaves nothing behind
        g.step(3)
        g.init(pl)
        o.init(pl)
        fo, Po = o.get_f(), o.get_P()
        np.testing.assert_allclose(g.get_f(), fo, rtol=0, atol=1e-13 * np.abs(fo).max())
        np.testing.assert_allclose(g.get_P(), Po, rtol=0, atol=1e-13 * np.abs(Po).max())
        g.close()


@pytest.mark.parametrize("prec", [W.PREC_F64, W.PREC_F32, W.PREC_F16S, W.PREC_BF16S])
def test_read_out_goes_through_any_storage(prec):
    """Written populations come back exactly, run on, and one infinite value is reported once."""
    from paper_1705_01801_gb300 import lbw
    spec = W.cylinder(30, 50, 40, prec=prec)
    rng = np.random.default_rng(0)
    f = np.round(rng.normal(size=(7, 40, 30, 50)), 1).astype(np.float16).astype(np.float64)
    f = np.round(f * 8) / 64  # exact in every format
    g = lbw.Grid(spec)
    g.set_f(f)
    np.testing.assert_array_equal(g.get_f(), f)
    P = g.get_P()
    assert np.isfinite(P).all()
    f[3, 39, 29, 49] = np.inf
    g.set_f(f)
    with pytest.raises(lbw.LbwError) as e:
        g.get_P()
    assert e.value.status == lbw.LBW_EUNSTABLE
    f[3, 39, 29, 49] = 0.125
    g.set_f(f)
    g.get_P()
