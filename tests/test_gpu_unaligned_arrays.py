"""Host arrays that are no multiple of 8 bytes off their start, page-locked or not,
pass through every transfer with the values of aligned ones."""
import numpy as np
import pytest

from paper_1505_02037_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1505_02037_gb300 import lbnr
    lbnr.library()
    return lbnr


def unaligned(values, offset, pinned):
    import torch
    raw = torch.empty(values.nbytes + 16, dtype=torch.uint8, pin_memory=pinned).numpy()
    a = np.frombuffer(raw.data, dtype=np.float64, count=values.size,
                      offset=offset).reshape(values.shape)
    a[...] = values
    return a


@pytest.mark.parametrize("pinned", [True, False])
@pytest.mark.parametrize("offset", [1, 4])
def test_unaligned(L, pinned, offset):
    shape = (19, 7, 5)
    cells = 19 * 7 * 5
    fields = W.smooth_modes(shape, 1 / 19, 0.01, seed=3).reshape(16, cells)
    lat = L.Lattice(3, shape, 2.0, 1 / 19)
    lat.init(fields)
    lat.step(2)
    want = lat.moments(), lat.distributions()
    L.lbnr_init(lat.ctx, unaligned(fields, offset, pinned))
    lat.step(2)
    m = unaligned(np.zeros((16, cells)), offset, pinned)
    L.lbnr_moments(lat.ctx, m)
    f = unaligned(np.zeros((16, 19, cells)), offset, pinned)
    L.lbnr_get_distributions(lat.ctx, f)
    assert m.ctypes.data % 8 and f.ctypes.data % 8
    assert np.array_equal(m, want[0]) and np.array_equal(f, want[1])
    L.lbnr_set_distributions(lat.ctx, f)
    assert np.array_equal(lat.distributions(), want[1])
    lat.close()
