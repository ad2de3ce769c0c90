"""Combinations of launch form and term that the other files leave out: every FP64
form (a thread or several lanes per cell) with matter and each slicing against
the oracle, and the one-launch step's shift forms on lattices that its work
list cuts into strips and many units."""
import numpy as np
import pytest

from paper_1505_02037_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL64 = 1e-12


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1505_02037_gb300 import lbnr
    lbnr.library()
    return lbnr


def dist_err(g, o):
    """Per field, relative to the field's size, at least 1 for lapse and metric
    and the noise amplitude of the random states for K and V."""
    g, o = g.reshape(16, -1), o.reshape(16, -1)
    floor = np.array([1.0] * 7 + [1e-3] * 9) / 3
    return (np.abs(g - o).max(axis=1) / np.maximum(np.abs(o).max(axis=1), floor)).max()


@pytest.mark.parametrize("slicing", [0, 1, 2])
@pytest.mark.parametrize("vset,shape", [(1, (77, 1, 1)), (2, (19, 7, 1)), (3, (9, 7, 5))])
def test_fp64_forms_with_matter_and_slicing(L, oracle_mod, vset, shape, slicing):
    Q = {1: 3, 2: 9, 3: 19}[vset]
    _, w = oracle_mod.velocity_set(vset)
    tau, dx, fluid = 0.8, 1 / shape[0], (0.2, 1 / 3, 1.5)
    f0 = W.random_distributions(Q, w, shape, seed=500 + vset)
    o = oracle_mod.Oracle(vset, shape, tau, dx, slicing=slicing, fluid=fluid)
    ref, spread = [], []
    # the bar of the other FP64 tests: 1e-12, or 4 x what one ulp in the initial
    # state moves the oracle
    rng = np.random.default_rng(0)
    f, fp = f0, f0 * (1 + rng.choice([-1.0, 1.0], size=f0.shape) * 2.2e-16)
    for n in range(3):
        f, fp = (o.run(x, 1, t=1.5 + n * dx) for x in (f, fp))
        ref.append(f)
        spread.append(dist_err(fp, f))
    names = L.Lattice(vset, shape, tau, dx).variants
    for v, name in enumerate(names):
        lat = L.Lattice(vset, shape, tau, dx, slicing=slicing)
        lat.set_variant(v)
        lat.set_fluid(*fluid)
        lat.set_distributions(f0)
        for n in range(3):
            lat.step(1)
            err = dist_err(lat.distributions(), ref[n])
            assert err <= max(TOL64, 4 * spread[n]), (name, n, err)
        lat.close()


@pytest.mark.parametrize("storage", ["f32", "dev_f32"])
@pytest.mark.parametrize("streaming", [1, 2])
@pytest.mark.parametrize("shift", ["none", "constant", "field"])
@pytest.mark.parametrize("base,times", [((16, 20, 7), (6, 3, 1)), ((67, 65, 5), (1, 2, 1)),
                                        ((33, 8, 12), (1, 1, 8))])
def test_one_launch_shift_forms_on_tiled_lattices(L, oracle_mod, base, times, shift, streaming,
                                                  storage):
    """A periodic lattice repeated along its axes does what the lattice does, bit
    for bit, whatever its work list looks like."""
    _, w = oracle_mod.velocity_set(3)
    beta = W.smooth_shift(base, 1 / base[0], 0.05, seed=9).reshape(3, *base[::-1])

    def tile(a, shape):  # [..., cells] of the base lattice to the repeated one
        a = a.reshape(*a.shape[:-1], *shape[::-1])
        return np.tile(a, (1,) * (a.ndim - 3) + times[::-1]).reshape(*a.shape[:-3], -1)

    f0 = W.random_distributions(19, w, base, seed=77).reshape(16, 19, -1)
    got = {}
    for name, shape, f, b in (
            ("base", base, f0, beta),
            ("tiled", tuple(n * t for n, t in zip(base, times)), tile(f0, base),
             np.tile(beta, (1,) + times[::-1]))):
        lat = L.Lattice(3, shape, 0.8, 1 / base[0], storage=storage, streaming=streaming)
        assert lat.launches_per_step == 1
        if shift != "none":
            lat.set_shift((0.05, -0.03, 0.02))
        if shift == "field":
            lat.set_shift_field(b)
        lat.set_distributions(f)
        out = []
        for _ in range(3):
            lat.step(1)
            out.append(lat.distributions())
        lat.status()
        got[name] = out
        lat.close()
    for n in range(3):
        assert np.array_equal(got["tiled"][n], tile(got["base"][n], base)), n
