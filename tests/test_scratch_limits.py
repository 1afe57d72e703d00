"""What is launched after an allocation or a launch has failed, on a fake CUDA runtime (tests/host):
every pointer that the next launch of a step kernel is given has to be a live allocation.  No GPU."""
import ctypes

import numpy as np
import pytest

import lbw_workloads as W
from host import load

SMALL = W.cylinder(20, 33, 10)           # on the multi-step kernel
RAGGED = W.cylinder(100, 100, 70)        # on the ensemble kernels, as a single lattice
TILED = W.cylinder(20, 64, 10).with_(geom_mode=W.GEOM_TABLE)


@pytest.fixture(scope="module")
def fake():
    return load()


@pytest.fixture(autouse=True)
def _reset(fake):
    yield
    L = fake.lib()
    L.fake_fail_allocation(0)
    L.fake_largest_allocation(2 ** 63)
    L.fake_fail_launch(b"")
    L.fake_errors()


def _until_it_succeeds(fake, call, after, all_behind=False):
    """`call` with its first, second, ... allocation failing (and all behind it) until none is left to
    fail; `after` runs behind each failure."""
    for n in range(1, 50):
        fake.lib().fake_fail_allocation(-n if all_behind else n)
        try:
            call()
        except fake.LbwError:
            failed = True
        else:
            failed = False
        fake.lib().fake_fail_allocation(0)
        after()
        assert fake.lib().fake_errors() == b"", n
        if not failed:
            return n
    raise AssertionError("the call never succeeded")


def _grid(fake, spec):
    g = fake.Grid(spec)
    g.init(W.pulses(spec, 1, 1, margin=0))
    return g


def _batch(fake, specs):
    b = fake.Batch(specs)
    b.init([W.pulses(s, 1, 1, margin=0) for s in specs])
    return b


@pytest.mark.parametrize("spec", [SMALL, TILED], ids=["small", "tiled"])
def test_a_failed_allocation_is_no_later_calls_error(fake, spec):
    """The runtime hands a failed allocation's error to the next look at its last error, which every
    launch takes: the call that failed clears it."""
    g = _grid(fake, spec)
    fake.lib().fake_fail_allocation(1)
    with pytest.raises(fake.LbwError):
        g.set_sources([[1, 1, 1]])
    g.init(W.pulses(spec, 1, 1, margin=0))
    g.close()


@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("spec", [SMALL, RAGGED, TILED], ids=["small", "ragged", "tiled"])
def test_sources_after_a_failed_allocation(fake, spec, kind):
    g = _grid(fake, spec)
    nodes = [[1, j, 2] for j in range(30)]
    g.set_sources(nodes, kind)
    assert _until_it_succeeds(fake, lambda: g.set_sources(nodes[:9], kind), lambda: g.step(3)) > 1
    g.close()
    assert fake.lib().fake_errors() == b""


@pytest.mark.parametrize("specs", [[SMALL] * 3, [RAGGED] * 2], ids=["small", "large"])
def test_ensemble_sources_after_a_failed_allocation(fake, specs):
    b = _batch(fake, specs)
    nodes = np.array([[[1, j, 2] for j in range(30)]] * len(specs))
    b.set_sources(nodes, np.ones(len(specs)))
    assert _until_it_succeeds(fake, lambda: b.set_sources(nodes[:, :9], np.ones(len(specs))), lambda: b.step(3)) > 1
    b.close()
    assert fake.lib().fake_errors() == b""


@pytest.mark.parametrize("spec", [SMALL, RAGGED, TILED], ids=["small", "ragged", "tiled"])
def test_probes_after_a_failed_allocation(fake, spec):
    g = _grid(fake, spec)
    g.set_probes([[1, 1, 1]] * 4, 100)
    assert _until_it_succeeds(fake, lambda: g.set_probes([[2, 2, 2]] * 3, 50), lambda: g.step(3)) > 1
    g.close()
    assert fake.lib().fake_errors() == b""


@pytest.mark.parametrize("shape", [None, (7, 16, 2)], ids=["created", "set"])
@pytest.mark.parametrize("specs", [[SMALL] * 3, [RAGGED] * 2], ids=["small", "large"])
def test_ensemble_probes_after_a_failed_allocation(fake, specs, shape):
    b = _batch(fake, specs)
    if shape:
        b.set_shape(*shape)
    b.set_probes([[[1, 1, 1]] * 4] * len(specs), 100)
    assert _until_it_succeeds(fake, lambda: b.set_probes([[[2, 2, 2]] * 3] * len(specs), 50), lambda: b.step(3)) > 1
    b.close()
    assert fake.lib().fake_errors() == b""


@pytest.mark.parametrize("all_behind", [False, True], ids=["one", "all"])
@pytest.mark.parametrize("call", [lambda b: b.set_shape(7, 16, 2), lambda b: b.set_shape(0, 16, 2),
                                  lambda b: b.tune(1)], ids=["columns", "rows", "tune"])
@pytest.mark.parametrize("specs", [[SMALL] * 3, [RAGGED] * 2], ids=["small", "large"])
def test_ensemble_shapes_after_a_failed_allocation(fake, specs, call, all_behind):
    """A change of shape that fails leaves the last one, or an ensemble that refuses to step."""
    b = _batch(fake, specs)
    b.set_sources([[[1, j, 2] for j in range(30)]] * len(specs), np.ones(len(specs)))
    before, refused = b.info(), []

    def after():
        try:
            b.step(3)
        except fake.LbwError as e:
            refused.append(e.status)
        else:
            assert refused or fake.lib().fake_launches(b"kernel") > 0

    assert _until_it_succeeds(fake, lambda: call(b), after, all_behind) > 1
    assert set(refused) <= {fake.LBW_ESTATE}
    assert before["nodes"] == b.info()["nodes"]
    b.step(3)  # the change that went through
    b.close()
    assert fake.lib().fake_errors() == b""


def test_weights_are_packed_again_after_a_failed_launch(fake):
    L = fake.lib()
    net = fake.MLP(7, 16, 4, 8)
    x = np.zeros((5, 7), np.float32)
    L.fake_fail_launch(b"pack_kernel")
    with pytest.raises(fake.LbwError):
        net.forward(x)
    L.fake_fail_launch(b"")
    before = L.fake_launches(b"pack_kernel")
    net.forward(x)
    assert L.fake_launches(b"pack_kernel") - before == 4
    net.forward(x)  # still those of the last change of the parameters
    assert L.fake_launches(b"pack_kernel") - before == 4
    net.close()


@pytest.mark.parametrize("hidden", [16, 18], ids=["one launch", "layer by layer"])
def test_training_after_a_failed_allocation(fake, hidden):
    """A call that could not train leaves the count of Adam's steps, frees what it took and names no
    sample that it has freed."""
    L = fake.lib()
    x, t = np.zeros((20, 7), np.float32), np.zeros((20, 8), np.float32)
    order = np.zeros((3, 8), np.int32)
    grads = []
    for n in range(1, 40):
        net = fake.MLP(7, hidden, 4, 8)
        net.train(x[:10], t[:10], order, 8, 1e-3)
        net.set_params(net.get_params())  # counts from 0
        L.fake_fail_allocation(n)
        try:
            net.train(x, t, order, 8, 1e-3)
            done = 3
        except fake.LbwError:
            done = 0
        L.fake_fail_allocation(0)
        if not done:
            net.train(x[:10], t[:10], order, 8, 1e-3)
            done = 3
        net.adam_step(np.zeros(net.nparam, np.float32), 1e-3)
        grads.append(L.fake_adam_correction())
        net.close()
        assert L.fake_errors() == b"", n
        assert abs(grads[-1] - (1 - 0.9 ** (done + 1))) < 1e-6, n


def test_a_failed_training_call_frees_what_it_took(fake):
    L = fake.lib()
    net = fake.MLP(7, 16, 4, 8)
    x, t, order = np.zeros((20, 7), np.float32), np.zeros((20, 8), np.float32), np.zeros((3, 8), np.int32)
    net.train(x, t, order, 8, 1e-3)
    live = L.fake_live()
    for n in (1, 2, 3):
        L.fake_fail_allocation(n)
        with pytest.raises(fake.LbwError):
            net.train(x, t, order, 8, 1e-3)
        assert L.fake_live() == live, n
    net.close()


@pytest.mark.parametrize("n", [1, 16, 200])
def test_spectra_in_smaller_passes_where_memory_is_short(fake, n):
    """The estimates of a call share a workspace, but need no more memory than one after the other."""
    T = 4096
    fake.lib().fake_largest_allocation(max(8 * T * n, 5 * 10 ** 6))  # the series, or four estimates' workspace
    assert len(fake.lbw_spectrum_series(np.zeros((n, T)), 4)) == n
    fake.lib().fake_largest_allocation(8 * T * n - 1)
    with pytest.raises(fake.LbwError):
        fake.lbw_spectrum_series(np.zeros((n, T)), 4)


@pytest.mark.parametrize("failing", range(1, 9))
@pytest.mark.parametrize("spec", [SMALL, RAGGED, TILED], ids=["small", "ragged", "tiled"])
def test_creation_needs_no_more_memory_than_the_lattice(fake, spec, failing):
    """Of a lattice's allocations only its populations, table and counters have to succeed: without the
    rest (or the longer rows of the ensemble kernels) it runs on the kernels that need none of it."""
    L = fake.lib()
    L.fake_fail_allocation(failing)
    try:
        g = fake.Grid(spec)
    except fake.LbwError:
        assert failing <= 4  # f, f, table, counters
        return
    finally:
        L.fake_fail_allocation(0)
    g.init(W.pulses(spec, 1, 1, margin=0))
    g.set_probes([[1, 1, 1]], 100)
    g.step(3)
    g.close()
    assert L.fake_errors() == b""


def test_ragged_lattice_without_room_for_its_padding(fake):
    """350 columns are stored in rows of 360 with ghost columns; where only the lattice itself fits it is
    stored densely."""
    L = fake.lib()
    spec = W.cylinder(40, 350, 60)
    L.fake_largest_allocation(7 * 4 * spec.nodes)
    g = fake.Grid(spec)
    L.fake_largest_allocation(2 ** 63)
    g.init(W.pulses(spec, 1, 1, margin=0))
    before = L.fake_launches(b"11step_kernel")
    g.step(3)
    assert L.fake_launches(b"11step_kernel") == before + 3
    g.close()
    assert L.fake_errors() == b""
