"""The label draw's short form on fields of any finite size, against the oracle
(tolerance: the parity protocol's 1e-6 around a decision boundary), in every
kernel form that draws labels, and the device's count of draws near a boundary."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle import decompose as dc, sampler
from paper_1611_06684_gb300 import workloads as wl
from paper_1611_06684_gb300 import mrf as M
from tests.gpu_helpers import make_handle, compare_sweep


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1611_06684_gb300 import build
    build.build()
    torch.cuda.set_device(0)


def _star(n, L, seed):
    rng = np.random.default_rng(seed)
    return wl.Model(n, L, rng.normal(size=(n, L)).astype(np.float32), np.zeros(n - 1, np.int32),
                    np.arange(1, n, dtype=np.int32), rng.normal(0, 0.3, (n - 1, L, L)).astype(np.float32))


# name: (model, chains, schedule), one per kernel form of the primal step
FORMS = {
    "site": (lambda: wl.potts_grid3d(6, 5, 3, L=4, seed=1), 64, 1),
    "pipe": (lambda: wl.potts_grid3d(6, 5, 3, L=8, seed=2), 64, 1),
    "warp": (lambda: wl.potts_grid3d(6, 5, 3, L=8, seed=3), 32, 1),
    "warp_chunks": (lambda: wl.tiny_random(60, 5, 400, w_std=0.4, seed=4), 32, 1),
    "low": (lambda: wl.potts_grid3d(6, 5, 3, L=4, seed=5), 5, 1),
    "thread": (lambda: wl.tiny_random(60, 4, 400, w_std=0.4, seed=6), 5, 1),
    "label_lanes": (lambda: wl.potts_grid3d(6, 5, 3, L=8, seed=7), 5, 1),
    "hub": (lambda: _star(301, 3, 8), 5, 1),
    "cta": (lambda: wl.dense_potts(60, L=4, seed=9), 16, 2),
    "partial": (lambda: wl.random_graph(60, k=2, L=16, seed=10, w_std=0.3), 2, 1),
}
SIZES = [5e9, -5e9, 1e10, 1e11, -1e11, 1e12, 1e20, 1e30, 3e38]


def _clamped(model, seed):
    """One label of every other site clamped by a potential of each size in turn (alone at the top where it
    is positive, alone at the bottom where it is negative)."""
    rng = np.random.default_rng(seed)
    for i, v in enumerate(range(0, model.n_vars, 2)):
        model.unary[v, rng.integers(model.n_labels)] = SIZES[i % len(SIZES)]
    return model


def _tied(model, seed):
    """Fields that are the unaries alone (no couplings but one edge's, which keeps the full tables), each
    site's labels all at one of the sizes, or some of them there and the others at zero."""
    rng = np.random.default_rng(seed)
    keep = {int(model.src[-1]), int(model.dst[-1])}
    model.pair[:-1] = 0.0
    for i, v in enumerate(v for v in range(model.n_vars) if v not in keep):
        size = SIZES[i % len(SIZES)]
        model.unary[v] = size
        if i % 3 == 0 and size > 0:
            model.unary[v, rng.permutation(model.n_labels)[:model.n_labels // 2]] = 0.0
    return model


def _shifted(model):
    """The model with every site's largest unary at zero (the same softmax): the oracle adds the maximum
    back to log sums, which loses them beside 1e12 and more."""
    u = model.unary.astype(np.float64)
    return dc.decompose(wl.Model(model.n_vars, model.n_labels, u - u.max(axis=1, keepdims=True), model.src, model.dst,
                                 model.pair))


def _check(model, C, seed, schedule, t=3):
    h = make_handle(model, C, seed, use_graphs=False, schedule=schedule)
    x0 = h.get_labels()
    h.set_sweep_index(t)
    h.sweep(1, M.MODE_PLAIN)
    dec = _shifted(model)
    ref = sampler.sweep(dec, x0.astype(np.int64), t, seed)
    x = h.get_labels()
    assert x.max() < model.n_labels
    compare_sweep(dec, ref, x, theta_gpu=M.unpack_theta(h.debug_theta(), dec.ell.shape[1]))
    h.close()


@pytest.mark.parametrize("kind", [_clamped, _tied])
@pytest.mark.parametrize("form", list(FORMS))
def test_labels_of_large_finite_fields(form, kind):
    make, C, schedule = FORMS[form]
    _check(kind(make(), 20), C, 7000, schedule)


@pytest.mark.parametrize("kind", [_clamped, _tied])
@pytest.mark.parametrize("name,make,C", [
    ("resident", lambda: wl.potts_grid3d(6, 5, 3, L=8, seed=11), 5),
    ("small", lambda: wl.ising_grid(60, 70, seed=12), 5),
    ("small_one_cta", lambda: wl.dense_potts(60, L=4, seed=13), 2)])
def test_one_launch_labels_of_large_finite_fields(name, make, C, kind):
    model = kind(make(), 21)
    many, single = (make_handle(model, C, 78, schedule=1, use_graphs=False) for _ in range(2))
    many.sweep(4)
    for _ in range(4):
        single.sweep(1)
    assert many.get_labels().max() < model.n_labels
    assert np.array_equal(many.get_labels(), single.get_labels())
    assert np.array_equal(many.counts(), single.counts())
    assert many.counts().sum() == 4 * C * model.n_vars


@pytest.mark.parametrize("L,C", [(2, 128), (8, 64), (5, 24)])
def test_draws_near_a_boundary_are_counted(L, C):
    # the device's CDF is within 7e-7 of the exact one (L <= 8: float32 terms and sums), so it counts
    # every draw within 0.3e-6 of a boundary and none beyond 2e-6
    model = wl.potts_grid3d(30, 30, 30, L=L, seed=30 + L)
    model.pair[:] = 0.0                                    # the fields are the unaries: no dual draw matters
    h = make_handle(model, C, 9, use_graphs=False, schedule=1)
    h.sweep(1)
    cdf = np.cumsum(np.exp(sampler.log_softmax(model.unary.astype(np.float64))), axis=-1)
    u = sampler.site_uniforms(model.n_vars, C, 0, 9)
    dist = np.abs(u[..., None] - cdf[None]).min(axis=-1)
    low, high = int((dist < 0.3e-6).sum()), int((dist < 2e-6).sum())
    assert 0 < low <= h.boundary_draws() <= high, (low, h.boundary_draws(), high)
    h.close()
