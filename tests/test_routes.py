"""Which kernels lattices are stepped by, on a fake CUDA runtime (tests/host): no GPU."""
import pytest

import lbw_workloads as W
from host import load

CART = dict(kind=W.KIND_CARTESIAN, h=(1, 1, 1), x0=(0, 0, 0), c=0.4, bc=(1, 2, 0, 0, 1, 3))


@pytest.fixture(scope="module")
def fake():
    return load()


def _kernels(fake, spec):
    """The names of the step kernels that three steps launch."""
    L = fake.lib()
    names = (b"15step_tma_kernel", b"11step_kernel", b"16batch_tma_kernel", b"16batch_row_kernel", b"15resident_kernel")
    g = fake.Grid(spec)
    g.init(W.pulses(spec, 1, 1, margin=0))
    before = [L.fake_launches(n) for n in names]
    g.step(3)
    took = {n[2:].decode() for n, b in zip(names, before) if L.fake_launches(n) > b}
    g.close()
    assert L.fake_errors() == b""
    return took


@pytest.mark.parametrize("prec,n,kernel", [
    # FP64 tiles of two and three rows are mostly halo
    (W.PREC_F64, (2, 200, 3193), "step_kernel"), (W.PREC_F64, (2, 33, 6060), "step_kernel"),
    (W.PREC_F64, (2, 100, 19560), "batch_row_kernel"), (W.PREC_F64, (3, 120, 1483), "step_kernel"),
    (W.PREC_F64, (3, 200, 2500), "batch_tma_kernel"), (W.PREC_F64, (3, 100, 1333), "batch_row_kernel"),
    (W.PREC_F64, (4, 200, 1000), "batch_tma_kernel"), (W.PREC_F32, (2, 200, 3193), "batch_row_kernel"),
    (W.PREC_F32, (100, 64, 250), "step_tma_kernel"), (W.PREC_F32, (40, 50, 100), "resident_kernel"),
])
def test_kernel_of_a_lattice(fake, prec, n, kernel):
    assert _kernels(fake, W.GridSpec(n=n, prec=prec, **CART)) == {kernel}


@pytest.mark.parametrize("rows,kernel", [(1, b"14forward_kernel"), (2432, b"14forward_kernel"),
                                         (2433, b"19forward_rows_kernel"), (50000, b"19forward_rows_kernel")])
def test_kernel_of_a_forward_pass(fake, rows, kernel):
    """Splitting every layer's inputs over 512 threads made narrow networks of many rows 1.6 times
    slower than a product per layer."""
    import numpy as np
    L = fake.lib()
    net = fake.MLP(7, 16, 4, 8)
    before = L.fake_launches(kernel), L.fake_launches(b"forward")
    net.forward(np.zeros((rows, 7), np.float32))
    assert (L.fake_launches(kernel) - before[0], L.fake_launches(b"forward") - before[1]) == (1, 1)
    net.close()


def test_the_injected_timeout_says_where_it_is_built(fake):
    """It is refused on ragged lattices, but not because their kernels had no waits."""
    for n in ((20, 33, 10), (100, 100, 70)):
        g = fake.Grid(W.cylinder(*n))
        g.init(W.pulses(g.spec, 1, 1, margin=0))
        with pytest.raises(fake.LbwError) as e:
            fake.lbw_inject_wait_timeout(g.handle)
        assert e.value.status == fake.LBW_EINVAL and "tile width" in str(e.value) and "no device waits" not in str(e.value)
        g.close()
