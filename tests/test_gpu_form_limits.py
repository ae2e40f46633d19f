"""A chain's labels do not depend on the kernel form that the number of chains
selects: its draws depend on its own index only, and every form adds in the
same order."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_1611_06684_gb300 import workloads as wl
from tests.gpu_helpers import make_handle


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1611_06684_gb300 import build
    build.build()
    torch.cuda.set_device(0)


def _same_first_chains(model, few, many, seed=5, sweeps=3):
    a, b = make_handle(model, few, seed, use_graphs=False, schedule=1), make_handle(model, many, seed, use_graphs=False, schedule=1)
    for _ in range(sweeps):
        a.sweep(1)
        b.sweep(1)
    assert np.array_equal(a.get_labels(), b.get_labels()[:few])


# sites such that `few` chains take a lane per label and `many` the thread form
@pytest.mark.parametrize("L,sites,few,many", [(5, 2000, 5, 7), (6, 2500, 5, 7), (7, 3600, 5, 7), (8, 5000, 5, 7),
                                              (9, 2400, 5, 6), (9, 6400, 3, 4)])
@pytest.mark.parametrize("k", [2, 12])
def test_label_lanes_and_thread_form_draw_the_same_labels(L, sites, few, many, k):
    _same_first_chains(wl.random_graph(sites, k=k, L=L, seed=L, w_std=0.3), few, many)


# chains on both sides of the limits of the low-degree form (items, chains) and of the groups per warp of the dual step
@pytest.mark.parametrize("L,side,few,many", [(2, 28, 14, 18), (3, 28, 14, 18), (4, 28, 14, 18), (5, 40, 4, 6), (6, 52, 7, 9),
                                             (8, 20, 6, 9), (8, 20, 9, 12), (8, 20, 12, 15), (7, 20, 6, 12), (9, 20, 9, 15)])
def test_low_degree_and_dual_group_limits_draw_the_same_labels(L, side, few, many):
    _same_first_chains(wl.potts_grid3d(side, L=L, seed=L), few, many, sweeps=2)


@pytest.mark.parametrize("L,side,few,many", [(3, 40, 4, 6), (4, 40, 4, 6), (8, 20, 3, 5)])
def test_low_degree_form_of_diagonal_tables(L, side, few, many):
    _same_first_chains(wl.ferro_potts_grid3d(side, L=L, seed=L), few, many, sweeps=2)


# largest lists of 119, 199 and 299 incidences: on both sides of the hub launch's limits for up to 32 chains and more
@pytest.mark.parametrize("sites,few,many", [(120, 3, 40), (200, 3, 40), (200, 32, 33), (300, 3, 40)])
def test_hub_limits_draw_the_same_labels(sites, few, many):
    _same_first_chains(wl.dense_potts(sites, L=4, seed=sites), few, many, sweeps=2)


# a CTA's hubs from 97 incidences on, from 193 on with two million items, no hub launch with many chains
@pytest.mark.parametrize("sites,few,many", [(20000, 3, 96), (40000, 3, 64), (20000, 3, 320), (20000, 32, 330)])
def test_hub_rules_of_large_models_draw_the_same_labels(sites, few, many):
    _same_first_chains(wl.ba_potts(sites, m=5, L=4, seed=sites), few, many, sweeps=2)


@pytest.mark.parametrize("device", [False, True])
def test_incidence_lists_of_every_length_are_in_order(device):
    # lists of 0 to 700 incidences, long ones next to each other: folded unaries (summed in list order) and
    # labels equal those of a handle whose lists were rebuilt by an edit that changes nothing
    import torch
    from paper_1611_06684_gb300 import mrf as M
    rng = np.random.default_rng(3)
    hub = rng.integers(0, 40, 6000)
    other = 40 + rng.integers(0, 900, 6000)
    hub[:700], other[:700] = 7, 40 + np.arange(700)
    hub[700:733], other[700:733] = 990, 1000 + np.arange(33)           # 33 and 32: the sorts' border
    hub[733:765], other[733:765] = 991, 1000 + np.arange(32)
    m = wl.Model(1100, 3, rng.normal(size=(1100, 3)).astype(np.float32), hub.astype(np.int32), other.astype(np.int32),
                 rng.normal(0, 0.1, (6000, 3, 3)).astype(np.float32))
    h, e = (M.MRF(m.n_vars, 3, 5, seed=2, schedule=1) for _ in range(2))
    arrays = (m.unary, m.src, m.dst, m.pair)
    h.set_factors(*(tuple(torch.from_numpy(x).cuda() for x in arrays) if device else arrays))
    e.set_factors(*arrays)
    e.edit_factors(np.array([11]), m.src[11:12], m.dst[11:12], m.pair[11:12])
    for x, y in zip(h.debug_tables(), e.debug_tables()):
        assert np.array_equal(x, y)
    fold = m.unary.astype(np.float64)
    assert not np.array_equal(h.debug_tables()[2], fold)
    for g in (h, e):
        g.sweep(3)
    assert np.array_equal(h.get_labels(), e.get_labels())
