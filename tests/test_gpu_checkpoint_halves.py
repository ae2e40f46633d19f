"""A checkpoint holds both halves of the label double buffer: the current
labels and those of the sweep before, whichever kernel form ran the sweeps."""
import numpy as np
import pytest

from paper_1611_06684_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1611_06684_gb300 import build
    build.build()
    torch.cuda.set_device(0)


def _halves(path, h):
    """x[2][N][C] of a checkpoint without free slots: the file ends with it and the counts [N][L]."""
    raw = np.fromfile(path, np.uint8)
    end = raw.size - 4 * h.N * h.L
    return raw[end - 2 * h.N * h.C:end].reshape(2, h.N, h.C)


def _dirty_memory():
    """Device memory full of 0xFF, returned to the driver for the next allocations."""
    import torch
    x = [torch.full((2 << 20,), 255, dtype=torch.uint8, device="cuda") for _ in range(32)]
    torch.cuda.synchronize()
    del x
    torch.cuda.empty_cache()


@pytest.mark.parametrize("sweeps", [0, 1, 2, 5, 100])
@pytest.mark.parametrize("name,make,C", [
    ("resident", lambda: wl.ising_grid(32, 32, seed=1), 1),
    ("resident_groups", lambda: wl.tiny_random(20, 4, 30, seed=5), 700),
    ("small", lambda: wl.ising_grid(60, 70, seed=3), 5),
    ("separate", lambda: wl.potts_grid3d(12, 12, 12, L=8, seed=4), 32)])
def test_both_label_halves_are_saved(name, make, C, sweeps, tmp_path):
    from paper_1611_06684_gb300 import mrf as M
    model = make()
    _dirty_memory()
    h = M.MRF(model.n_vars, model.n_labels, C, seed=3, schedule=1)
    h.set_factors(model.unary, model.src, model.dst, model.pair)
    h.sweep(sweeps)
    path = str(tmp_path / "ckpt.mrf")
    h.save(path)
    x = _halves(path, h)
    assert np.array_equal(x[sweeps & 1].T, h.get_labels())
    if sweeps:                                             # the other half: the labels one sweep earlier
        before = M.MRF(model.n_vars, model.n_labels, C, seed=3, schedule=1)
        before.set_factors(model.unary, model.src, model.dst, model.pair)
        before.sweep(sweeps - 1)
        assert np.array_equal(x[(sweeps + 1) & 1].T, before.get_labels())
    r = M.MRF.load(path)
    for hh in (h, r):
        hh.sweep(3)
    assert np.array_equal(h.get_labels(), r.get_labels())
    assert np.array_equal(h.counts(), r.counts())
