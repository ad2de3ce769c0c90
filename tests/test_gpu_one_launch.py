"""The SYNC step with both passes in one launch (FP32 storage, D3Q19) on
lattices that its work list cuts into several units, strips and ragged tiles:
two single steps (in place: both layouts) from the stored state against the
oracle's step, within the derived one-step bound; and the same bits whichever
blocks claim the items."""
import numpy as np
import pytest

from onestep_bound import field_max_err, first_order_max, one_step_bound
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


SHAPES = [(64, 40, 9), (96, 60, 7), (67, 131, 5), (131, 37, 6), (33, 8, 96)]


@pytest.mark.parametrize("storage", ["f32", "dev_f32"])
@pytest.mark.parametrize("streaming", [1, 2])
@pytest.mark.parametrize("shape", SHAPES)
def test_one_launch_step(L, oracle_mod, shape, streaming, storage):
    c, w = oracle_mod.velocity_set(3)
    tau, dx = 0.8, 1 / shape[0]
    o = oracle_mod.Oracle(3, shape, tau, dx)
    lat = L.Lattice(3, shape, tau, dx, storage=storage, streaming=streaming)
    bits = []
    for name in ("P1-reread-64x4", "P1-reread", "P1-reread-64x4"):
        lat.set_variant(lat.variants.index(name))
        lat.set_distributions(W.random_distributions(19, w, shape, seed=77))
        f_in = lat.distributions()
        for n in range(2):
            lat.step(1)
            got = lat.distributions()
            if not bits or name == "P1-reread":
                ref = o.step(f_in)
                rho = o.moments(f_in)
                m1 = first_order_max(rho.reshape(16, *shape[::-1]), dx, 3)
                b = one_step_bound(storage, c, w, tau, dx, f_in, ref, rho[0].max(), m1)
                err = field_max_err(got, ref)
                bad = np.flatnonzero(err > b)
                assert bad.size == 0, (name, n, [(int(F), err[F], b[F]) for F in bad])
            f_in = got
        lat.status()
        bits.append(f_in)
        # the odd step count would change the in-place layout of the next form
        assert lat.steps_done % 2 == 0
    assert np.array_equal(bits[0], bits[1]) and np.array_equal(bits[0], bits[2])
    lat.close()
