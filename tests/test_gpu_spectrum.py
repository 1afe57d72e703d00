"""The device estimator against the oracle's at the lengths where its transform, segments and
batching can go wrong: every remainder radix (M / 2 = 8 .. 1024 points), odd lengths, fewer
samples than segments, more estimates than one pass holds.

Tolerances: the search compares powers whose rounding is a few 1e-16, flat to second order at the
maximum, so it determines a frequency to about 1e-8 of the line width 2 pi / T: 1e-7 of it here;
amplitudes to 1e-9.  The oracle's sums over a long series round more coarsely (the phase omega t
alone to 1e-12 at t = 4000, which moves its search by 1e-7 of the width), so its frequencies are
polished by Newton steps in extended precision."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _series(T, n, seed):
    rng = np.random.default_rng(seed)
    t = np.arange(T)
    x = np.zeros((n, T))
    for _ in range(5):
        x += rng.uniform(0.1, 1.0, (n, 1)) * np.cos(rng.uniform(0.2, 2.8, (n, 1)) * t + rng.uniform(0, 6, (n, 1)))
    return x + 1e-3 * rng.normal(size=(n, T)) + rng.normal()


def _polish(x, f):
    """The maximum of the windowed power next to f: two Newton steps on its derivative."""
    L = np.longdouble
    T = x.size
    t = np.arange(T).astype(L)
    w = L(0.5) - L(0.5) * np.cos(2 * np.arccos(L(-1)) * t / (T - 1))
    xw, u = w * (x.astype(L) - x.astype(L).mean()), t - L(T) / 2
    out = []
    for om in f.astype(L):
        for _ in range(2):
            c, s = np.cos(om * u), np.sin(om * u)
            X = [(np.sum(xw * u ** m * c), -np.sum(xw * u ** m * s)) for m in range(3)]
            # X' = -i sum x u e, X'' = -sum x u^2 e; P' = 2 Re(conj X X'), P'' = 2 (|X'|^2 + Re(conj X X''))
            (a, b), (a1, b1), (a2, b2) = X
            d1 = a * b1 - b * a1
            d2 = a1 * a1 + b1 * b1 - a * a2 - b * b2
            om = om - d1 / d2
        out.append(float(om))
    return np.array(out)


@pytest.mark.parametrize("T", [5, 8, 9, 16, 17, 31, 33, 64, 65, 100, 129, 255, 256, 257, 1000, 4097])
@pytest.mark.parametrize("k", [1, 64])
def test_matches_oracle(T, k):
    from paper_1705_01801_gb300 import lbw
    x = _series(T, 3, T)
    for (f, a), row in zip(lbw.lbw_spectrum_series(x, k), x):
        fo, ao = oracle.spectrum(row, k)
        assert len(f) == len(fo)
        np.testing.assert_allclose(f, _polish(row, fo), rtol=0, atol=1e-7 * 2 * np.pi / T)
        np.testing.assert_allclose(a, ao, rtol=1e-9)


def test_more_series_than_one_pass_and_a_zero_one():
    """At 20,000 samples 256 MB hold fewer than 80 workspaces: rows of a call of 150 equal the same
    rows alone, a constant row has no peaks, and a NaN is reported."""
    from paper_1705_01801_gb300 import lbw
    x = _series(20000, 150, 7)
    x[3] = 2.5
    got = lbw.lbw_spectrum_series(x, 4)
    assert len(got[3][0]) == 0
    for r in (0, 75, 149):
        (f, a), = lbw.lbw_spectrum_series(x[r:r + 1], 4)
        assert np.array_equal(f, got[r][0]) and np.array_equal(a, got[r][1]) and len(f) == 4
    x[140, 5] = np.nan
    with pytest.raises(lbw.LbwError) as e:
        lbw.lbw_spectrum_series(x, 4)
    assert e.value.status == lbw.LBW_EUNSTABLE
