"""The bounded wait of the one-launch step (FP32 storage, D3Q19): when it runs
out no cell is stored, the steps behind it do nothing, every read-back of the
state says so, and a new initial state runs as if nothing had happened."""
import ctypes

import numpy as np
import pytest

from paper_1505_02037_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TIMEOUT = -5


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1505_02037_gb300 import lbnr
    lbnr.library()
    return lbnr


@pytest.mark.parametrize("shape", [(8, 4, 2), (64, 40, 9), (96, 60, 7)])
@pytest.mark.parametrize("streaming", [1, 2])
@pytest.mark.parametrize("shift", [False, True])
def test_wait_that_runs_out(L, shape, streaming, shift):
    cells = shape[0] * shape[1] * shape[2]
    fields = W.smooth_modes(shape, 1 / shape[0], 0.01, seed=3)

    def lattice():
        lat = L.Lattice(3, shape, 4.5, 1 / shape[0], storage="f32", streaming=streaming)
        if shift:
            lat.set_shift((0.05, 0.02, -0.02))
        lat.init(fields)
        return lat

    lat = lattice()
    lat.step(4)
    want = lat.distributions()

    lat.init(fields)
    start = lat.distributions()
    L.lbnr_set_step_wait(lat.ctx, 1_000_000, True)
    lat.step(4)
    with pytest.raises(L.LbnrError) as e:
        lat.status()
    assert e.value.code == TIMEOUT
    got = np.full((16, 19, cells), np.nan)
    p = got.ctypes.data_as(ctypes.POINTER(ctypes.c_double))
    assert L.library().lbnr_get_distributions(lat.ctx, p) == TIMEOUT
    # four steps lead back to the first buffer and layout, which nothing has changed
    assert np.array_equal(got, start)
    for call in (lat.moments, lat.constraints, lambda: lat.cells_distributions([0])):
        with pytest.raises(L.LbnrError) as e:
            call()
        assert e.value.code == TIMEOUT

    # the hook taken back, the state is still refused and not stepped further
    L.lbnr_set_step_wait(lat.ctx, 2_000_000_000)
    lat.step(2)
    assert L.library().lbnr_get_distributions(lat.ctx, p) == TIMEOUT
    assert np.array_equal(got, start)
    lat.init(fields)
    lat.step(4)
    lat.status()
    assert np.array_equal(lat.distributions(), want)
    with pytest.raises(L.LbnrError):
        L.lbnr_set_step_wait(lat.ctx, 0)
    lat.close()
