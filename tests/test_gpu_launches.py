"""lbnr_launches_per_step against what a step of each kind of context launches."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1505_02037_gb300 import lbnr
    lbnr.library()
    return lbnr


@pytest.mark.parametrize("vset,storage,streaming,deriv,form,want", [
    (3, "f32", 1, "sync", None, 1),                 # both passes in one launch
    (3, "dev_f32", 2, "sync", "P1-reread", 1),
    (3, "f32", 1, "sync", "tma-p1-nc4-k1-t32", 2),  # a moment pass of its own
    (3, "f32", 1, "lag", "tma-p1-nc4-k1-t32", 1),   # none
    (3, "dev_f16", 1, "sync", None, 2),
    (3, "dev_f16", 1, "lag", None, 1),
    (3, "f64", 1, "sync", "lanes16", 1),
    (3, "f64", 2, "sync", "lanes16", 2),            # in place form 0 runs instead
    (3, "f64", 1, "sync", "P1-reread", 2),
    (1, "f64", 1, "sync", None, 1),                 # lanes by default
    (2, "f32", 1, "sync", None, 2),
])
def test_launches(L, vset, storage, streaming, deriv, form, want):
    shape = {1: (48, 1, 1), 2: (16, 12, 1), 3: (8, 6, 5)}[vset]
    lat = L.Lattice(vset, shape, 2.0, 0.1, storage=storage, streaming=streaming, deriv_mode=deriv)
    if form:
        lat.set_variant(lat.variants.index(form))
    assert lat.launches_per_step == want
    # a shift runs its own form: one launch for FP32 storage on D3Q19
    lat.set_shift((0.05, 0.0, 0.0))
    fused = vset == 3 and storage in ("f32", "dev_f32")
    assert lat.launches_per_step == (1 if fused or deriv == "lag" else 2)
    lat.set_shift((0.0, 0.0, 0.0))
    lat.set_fluid(0.1, 0.3)
    assert lat.launches_per_step == want + 1
    lat.close()
    assert L.library().lbnr_launches_per_step(None) == -1
