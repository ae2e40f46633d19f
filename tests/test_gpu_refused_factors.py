"""A refused set_factors leaves the handle's model as it was: later edits and
sweeps equal those of a handle that never saw the refused model."""
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


def _refused(model, kind):
    """Another model of the same sites that set_factors refuses."""
    bad = wl.tiny_random(model.n_vars, model.n_labels, 90, seed=8)
    bad.unary += 3.0
    if kind == "range":
        bad.dst[7] = model.n_vars
    elif kind == "negative":
        bad.src[0] = -1
    elif kind == "self_loop":
        bad.dst[7] = bad.src[7]
    elif kind == "unary":
        bad.unary[2, 1] = np.inf
    else:
        bad.pair[3, 1, 1] = np.nan
    return bad


@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("kind", ["range", "negative", "self_loop", "unary", "pair"])
def test_a_refused_model_leaves_no_trace(kind, device):
    import torch
    from paper_1611_06684_gb300 import mrf as M
    N, L, C = 200, 4, 6
    model = wl.ferro_potts_graph(N, L, 500, seed=5)
    bad = _refused(model, kind)
    arrays = (bad.unary, bad.src, bad.dst, bad.pair)
    if device:
        arrays = tuple(torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in arrays)
        torch.cuda.synchronize()
    h, clean = (M.MRF(N, L, C, seed=9, schedule=1) for _ in range(2))
    for g in (h, clean):
        g.set_factors(model.unary, model.src, model.dst, model.pair)
        g.sweep(2)
    with pytest.raises(M.MrfError) as err:
        h.set_factors(*arrays)
    assert err.value.status == (M.MRF_ENONFINITE if kind in ("unary", "pair") else M.MRF_ERANGE)
    for g in (h, clean):
        g.sweep(1)
        g.edit_factors(np.array([5, 6, 40]), np.array([1, 7], np.int32), np.array([150, 9], np.int32),
                       np.stack([np.eye(L, dtype=np.float32) * 0.3] * 2))      # folds the touched sites again
        g.sweep(2)
        g.sweep(2, M.MODE_SW)
        g.sweep(1, M.MODE_HIGDON)
    for x, y in zip(h.debug_tables(), clean.debug_tables()):
        assert np.array_equal(x, y)
    assert np.array_equal(h.get_labels(), clean.get_labels())
    assert np.array_equal(h.counts(), clean.counts())
