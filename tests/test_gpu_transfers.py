"""Transfers between the state and host arrays: page-locked arrays (read and
written by a kernel, 16 or 8 bytes a word by their alignment) and pageable ones
(copied) give the same values, over odd sizes and offsets; and the
distributions of every set, storage and layout come back plane by plane."""
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


@pytest.mark.parametrize("vset,shape", [(1, (1, 1, 1)), (1, (333, 1, 1)), (2, (19, 7, 1)),
                                        (3, (17, 9, 5)), (3, (64, 32, 40))])
@pytest.mark.parametrize("offset", [0, 1])
def test_pinned_and_pageable_arrays(L, vset, shape, offset):
    import torch
    cells = shape[0] * shape[1] * shape[2]
    f = W.smooth_modes(shape, 1 / shape[0], 0.01, seed=3).reshape(16, cells) if cells > 1 \
        else W.flat(shape).reshape(16, cells)
    pin = torch.empty(16 * cells + 3, dtype=torch.float64, pin_memory=True)
    fields = pin[offset:offset + 16 * cells].view(16, cells)  # 16-byte aligned or 8 off
    fields.copy_(torch.from_numpy(np.ascontiguousarray(f)))
    out = torch.full((16 * cells + 3,), 7.0, dtype=torch.float64).pin_memory()
    lat = L.Lattice(vset, shape, 2.0, 1 / shape[0])
    lat.init(f)
    lat.step(3)
    ref = lat.moments()
    lat.init(fields)
    lat.step(3)
    got = lat.moments(out[offset:offset + 16 * cells].view(16, cells))
    assert np.array_equal(got.numpy(), ref)
    rest = torch.cat([out[:offset], out[offset + 16 * cells:]])
    assert bool((rest == 7.0).all())  # nothing written beside the array
    lat.close()


@pytest.mark.parametrize("vset,shape", [(1, (77, 1, 1)), (2, (19, 7, 1)), (3, (9, 7, 5))])
@pytest.mark.parametrize("storage", ["f64", "f32", "dev_f32", "dev_bf16", "dev_f16"])
@pytest.mark.parametrize("streaming", [1, 2])
def test_distributions_round_trip(L, oracle_mod, vset, shape, storage, streaming):
    """Distributions set and read back at both step parities, every plane its
    own values; the sampled cells agree with the planes."""
    Q = {1: 3, 2: 9, 3: 19}[vset]
    _, w = oracle_mod.velocity_set(vset)
    lat = L.Lattice(vset, shape, 2.0, 1 / shape[0], storage=storage, streaming=streaming)
    f0 = W.random_distributions(Q, w, shape, seed=5)
    unit = {"f64": 2.0 ** -52, "f32": 2.0 ** -23, "dev_f32": 2.0 ** -22, "dev_bf16": 2.0 ** -8,
            "dev_f16": 2.0 ** -10}[storage]  # of a stored value below 1, FP64 decoding included
    lat.set_distributions(f0)
    for _ in range(2):
        lat.set_distributions(f0)
        got = lat.distributions()
        assert np.abs(got - f0).max() <= unit
        idx = np.arange(0, lat.cells, 3)
        assert np.array_equal(lat.cells_distributions(idx), got[:, :, idx].transpose(2, 0, 1))
        lat.step(1)
    lat.close()
