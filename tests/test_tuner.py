"""The autotuner's choices, on a fake CUDA runtime whose clock the test sets: no GPU."""
import ctypes
import json

import pytest

import lbw_workloads as W
from host import load

SMALL = [W.cylinder(20, 33, 10)] * 3  # starts on the multi-step kernel
LARGE = [W.cylinder(60, 90, 150 + 3 * m) for m in range(9)]  # on full-row tiles


@pytest.fixture(scope="module")
def fake():
    return load()


def _tune(fake, batch, clock, **kw):
    """tune() with `clock(shape, resident)` for the milliseconds of each trial."""
    L = fake.lib()
    counts = [0]

    def elapsed():
        many = L.fake_launches(b"15resident_kernel")
        resident, counts[0] = many > counts[0], many
        return float(clock(batch.info(), resident))

    counts[0] = L.fake_launches(b"15resident_kernel")
    f = ctypes.CFUNCTYPE(ctypes.c_float)(elapsed)
    L.fake_elapsed(f)
    try:
        return batch.tune(trial_steps=2, **kw)
    finally:
        L.fake_elapsed(ctypes.cast(None, ctypes.CFUNCTYPE(ctypes.c_float)))


def _steps_on(fake, batch, kernel):
    L = fake.lib()
    batch.init([W.pulses(s, 1, 1, margin=0) for s in batch.specs])
    before = L.fake_launches(kernel)
    batch.step(2)
    return L.fake_launches(kernel) > before


def test_the_shape_it_starts_with_is_among_those_timed(fake):
    """best_shape has more lengths than the tuner: where its choice is the fastest, it stays."""
    for specs in (LARGE, [s.with_(n=(s.n[0], s.n[1], 8 * k + 9)) for k, s in enumerate(LARGE)]):
        b = fake.Batch(specs)
        start = b.info()
        _tune(fake, b, lambda info, resident: 1.0 if info == start else 2.0)
        assert b.info() == start
        b.close()


def test_cache_lines_of_other_kernels_are_not_taken(fake, tmp_path):
    """A line of the same sizes written before there was a multi-step kernel (no field for it, another
    signature), or for an ensemble that does not offer it, says nothing about this one."""
    cache = tmp_path / "tune.jsonl"
    table = fake.Batch([s.with_(geom_mode=W.GEOM_TABLE) for s in SMALL])
    _tune(fake, table, lambda info, resident: 1.0, cache_path=str(cache))
    line = json.loads(cache.read_text())
    old = dict(line, signature=line["signature"].split("-k")[0])
    cache.write_text(json.dumps(old) + "\n" + json.dumps(line) + "\n")
    table.close()
    b = fake.Batch(SMALL)
    report = _tune(fake, b, lambda info, resident: 0.1 if resident else 1.0, cache_path=str(cache))
    assert "cached" not in report and "resident" in report
    assert _steps_on(fake, b, b"15resident_kernel")
    b.close()
    b = fake.Batch(SMALL)  # its own line is
    assert "cached resident" in _tune(fake, b, lambda info, resident: 1.0, cache_path=str(cache))
    assert _steps_on(fake, b, b"15resident_kernel")
    b.close()
    assert fake.lib().fake_errors() == b""
