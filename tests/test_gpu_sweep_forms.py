"""Forms of the sweep kernels that are chosen by size, against the oracle: one
plain sweep's labels without the log-probability record (so the label draw
takes its short form first), tolerance the parity protocol's 1e-6 around a
decision boundary."""
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


def _check(model, C, seed, t=3, **kw):
    h = make_handle(model, C, seed, use_graphs=False, schedule=kw.pop("schedule", 1), **kw)
    x0 = h.get_labels()
    h.set_sweep_index(t)
    h.sweep(1, M.MODE_PLAIN)
    dec = dc.decompose(model)
    ref = sampler.sweep(dec, x0.astype(np.int64), t, seed)
    W = (dec.ell.shape[1] + 31) // 32
    theta = M.unpack_theta(h.debug_theta(), dec.ell.shape[1]) if model.n_edges else None
    stats = compare_sweep(dec, ref, h.get_labels(), theta_gpu=theta)
    seen, expect = h.boundary_draws(), stats["site_boundary"]
    h.close()
    # the device's count uses its float32 CDF: a draw at the edge of the 1e-6 band may differ
    assert abs(int(seen) - expect) <= 3 + expect, (seen, expect)


def _wide_fields(L, seed):
    """Unaries from 0 to 3e4 in magnitude, exact ties among them."""
    m = wl.potts_grid3d(5, 4, 3, L=L, seed=seed)
    rng = np.random.default_rng(seed)
    m.unary *= np.float32(10.0) ** rng.integers(-1, 5, (m.n_vars, 1)).astype(np.float32)
    m.unary[::3] = np.round(m.unary[::3, :1])
    return m


@pytest.mark.parametrize("L,C,shape", [(2, 64, (7, 5, 3)), (3, 128, (9, 1, 1)), (4, 64, (5, 5, 1)), (6, 64, (6, 3, 2)),
                                       (7, 64, (5, 4, 3)), (8, 192, (4, 3, 3)), (10, 64, (5, 3, 2)), (12, 64, (4, 3, 2)),
                                       (11, 32, (4, 3, 3)), (12, 96, (3, 3, 3)), (14, 32, (4, 3, 2)), (8, 32, (5, 4, 3)),
                                       (16, 64, (3, 3, 2)), (5, 24, (5, 4, 3))])
def test_lattice_forms_match_the_oracle(L, C, shape):
    _check(wl.potts_grid3d(*shape, L=L, seed=40 + L), C, 1000 + L)


@pytest.mark.parametrize("L,C,E,N", [(5, 1, 900, 200), (6, 7, 400, 150), (7, 2, 600, 40), (8, 1, 1500, 70), (9, 3, 300, 90)])
def test_label_lanes_match_the_oracle(L, C, E, N):
    # a lane per label: odd item counts, degrees on both sides of a two-sum flush (32)
    _check(wl.tiny_random(N, L, E, w_std=0.3, seed=110 + L), C, 5000 + L)


@pytest.mark.parametrize("L,C", [(4, 64), (8, 64), (8, 32), (16, 64)])
def test_diagonal_tables_match_the_oracle(L, C):
    _check(wl.ferro_potts_grid3d(5, 4, 3, L=L, seed=50 + L), C, 2000 + L)


@pytest.mark.parametrize("L,C,E", [(8, 64, 150), (5, 64, 400), (12, 32, 120)])
def test_sites_of_uneven_degree_match_the_oracle(L, C, E):
    # isolated sites and degrees on both sides of the one-batch and pipelined forms' limits
    _check(wl.tiny_random(60, L, E, w_std=0.4, seed=60 + L), C, 3000 + L)


@pytest.mark.parametrize("L,C", [(2, 64), (8, 64), (8, 5), (16, 32)])
def test_label_draw_of_wide_fields_matches_the_oracle(L, C):
    _check(_wide_fields(L, 70 + L), C, 4000 + L)


SMALL = {
    "one_chain_L2": (lambda: wl.ising_grid(32, 32, seed=1), 1),                 # eight CTAs per cluster
    "ten_chains_L2": (lambda: wl.ising_grid(50, 50, seed=2), 10),               # 640 threads per CTA
    "too_many_items_per_chain": (lambda: wl.ising_grid(60, 70, seed=3), 5),     # more than 8 x 640
    "tiny": (lambda: wl.tiny_random(3, 3, 2, seed=4), 1),
    "single_site": (lambda: wl.Model(1, 5, np.zeros((1, 5), np.float32), np.zeros(0, np.int32), np.zeros(0, np.int32),
                                     np.zeros((0, 5, 5), np.float32)), 3),
    "several_chains_per_cluster": (lambda: wl.tiny_random(20, 4, 30, seed=5), 700),   # the last cluster is part full
    "odd_chains": (lambda: wl.tiny_random(70, 3, 100, seed=6), 37),
    "degree_79_L4": (lambda: wl.dense_potts(80, L=4, seed=7), 5),               # two-sum flushes
    # sites of more than 96 incidences: one CTA each in the separate launches
    "star_C32": (lambda: wl.Model(701, 3, np.random.default_rng(1).normal(size=(701, 3)).astype(np.float32),
                                  np.zeros(700, np.int32), np.arange(1, 701, dtype=np.int32),
                                  np.random.default_rng(2).normal(0, 0.3, (700, 3, 3)).astype(np.float32)), 32),
    "dense_L3_C5": (lambda: wl.dense_potts(129, L=3, seed=11), 5),
    "dense_L6_C1": (lambda: wl.dense_potts(161, L=6, seed=12), 1),
    "wide_L16": (lambda: wl.random_graph(60, k=2, L=16, seed=8, w_std=0.3), 7), # table rows of 225 entries
    "diag_L16": (lambda: wl.tiny_potts(90, 16, 200, seed=9), 9),
    "lattice_L8": (lambda: wl.potts_grid3d(6, 6, 6, L=8, seed=10), 32),
}


@pytest.mark.parametrize("name", list(SMALL))
def test_small_models_run_the_same_chain_in_one_launch(name):
    make, C = SMALL[name]
    model = make()
    many, single = (make_handle(model, C, 77, schedule=1, use_graphs=False) for _ in range(2))
    if model.n_edges > 3:                                  # free slots inside the edge list
        for h in (many, single):
            h.edit_factors(np.array([1, 3]), np.zeros(0, np.int32), np.zeros(0, np.int32),
                           np.zeros((0, model.n_labels, model.n_labels), np.float32))
            h.reset_marginals(2)
    many.set_kernel_timing(True)
    many.sweep(5)
    assert list(many.kernel_times()) == ["k_sweep_small"]
    for _ in range(5):
        single.sweep(1)
    assert np.array_equal(many.get_labels(), single.get_labels())
    assert np.array_equal(many.counts(), single.counts())
    assert many.boundary_draws() == single.boundary_draws()
    for h in (many, single):                               # the sweep index advanced alike
        h.sweep(1)
    assert np.array_equal(many.get_labels(), single.get_labels())
    assert many.info().sweep_index == single.info().sweep_index == 6


@pytest.mark.parametrize("mode,L,C,label_dependent", [(M.MODE_SW, 8, 64, False), (M.MODE_SW, 5, 64, True), (M.MODE_SW, 2, 128, False),
                                                      (M.MODE_SW, 16, 36, True), (M.MODE_HIGDON, 8, 64, True),
                                                      (M.MODE_HIGDON, 3, 68, False)])
def test_cluster_sweeps_do_not_depend_on_the_scan_form(mode, L, C, label_dependent):
    # four chains per lane (many items) and one per lane (three chains): a chain's
    # draws depend on its own index only, so the first three chains are the same
    model = wl.ferro_potts_grid3d(23, 22, 21, L=L, seed=80 + L)
    if label_dependent:
        rng = np.random.default_rng(L)
        model.pair[:, np.arange(L), np.arange(L)] = rng.uniform(0, 1.2, (model.n_edges, L)) * (rng.random((model.n_edges, L)) > 0.2)
    many, few = make_handle(model, C, 5, use_graphs=False), make_handle(model, 3, 5, use_graphs=False)
    for h in (many, few):
        h.set_labels(np.zeros((h.C, h.N), np.uint8))          # equal labels: the first sweep bonds most
        for _ in range(3):
            h.sweep(1, mode)
    assert np.array_equal(many.get_labels()[:3], few.get_labels())


@pytest.mark.parametrize("C", [64, 45])
def test_hub_potentials_do_not_depend_on_the_chain_count(C):
    # Higdon's potentials of a complete graph of 300 sites (299 incidences each): the hub CTAs'
    # slices and rounds differ between 3 chains and C
    model = wl.ferro_potts_graph(300, 4, 44850, beta_lo=0.0, beta_hi=0.02, seed=90)
    many, few = make_handle(model, C, 6, use_graphs=False), make_handle(model, 3, 6, use_graphs=False)
    for h in (many, few):
        for _ in range(3):
            h.sweep(1, M.MODE_HIGDON)
    assert np.array_equal(many.get_labels()[:3], few.get_labels())


def _set(h, m, device):
    import torch
    arrays = (m.unary, m.src, m.dst, m.pair)
    if device:
        arrays = tuple(torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in arrays)
        torch.cuda.synchronize()
    h.set_factors(*arrays)


@pytest.mark.parametrize("device", [False, True])
def test_set_factors_again_equals_a_new_handle(device):
    """New potentials, then models of other edges, degrees, sizes and layouts on one handle (its arrays
    and captured sweeps are kept where they fit), and a refused model in between."""
    import torch
    N, L, C = 360, 4, 6
    models = [wl.potts_grid3d(10, 9, 4, L=L, seed=1), wl.potts_grid3d(10, 9, 4, L=L, seed=2),
              wl.tiny_random(N, L, 900, w_std=0.4, seed=3), wl.tiny_random(N, L, 700, w_std=0.4, seed=4),
              wl.ferro_potts_graph(N, L, 800, seed=5), wl.tiny_random(N, L, 5000, w_std=0.2, seed=6),
              wl.Model(N, L, np.zeros((N, L), np.float32), np.zeros(0, np.int32), np.zeros(0, np.int32),
                       np.zeros((0, L, L), np.float32)),
              wl.potts_grid3d(10, 9, 4, L=L, seed=7)]
    bad = wl.tiny_random(N, L, 50, seed=8)
    bad.dst[7] = N
    stream = torch.cuda.Stream()
    h = M.MRF(N, L, C, seed=9, stream=stream.cuda_stream, schedule=1)
    for i, m in enumerate(models):
        _set(h, m, device)
        if i == 3:
            with pytest.raises(M.MrfError) as err:
                _set(h, bad, device)
            assert err.value.status == M.MRF_ERANGE and "edge 7" in str(err.value)
            bad.dst[7] = 0 if bad.src[7] else 1
            bad.pair[3, 1, 1] = np.inf
            with pytest.raises(M.MrfError) as err:
                _set(h, bad, device)
            assert err.value.status == M.MRF_ENONFINITE
            _set(h, m, device)
        fresh = M.MRF(N, L, C, seed=9, stream=stream.cuda_stream, schedule=1)
        _set(fresh, m, False)
        fresh.set_labels(h.get_labels())
        fresh.set_sweep_index(h.info().sweep_index)
        for g in (h, fresh):
            g.reset_marginals(0)
            g.sweep(1)
            g.sweep(3)
        assert np.array_equal(h.get_labels(), fresh.get_labels())
        assert np.array_equal(h.counts(), fresh.counts())
        for x, y in zip(h.debug_tables(), fresh.debug_tables()):
            assert np.array_equal(x, y)
        assert abs(h.info().log_const - fresh.info().log_const) <= 1e-9 * max(1.0, abs(fresh.info().log_const))
        if i == 2:                                         # edits after a second model
            for g in (h, fresh):
                g.edit_factors(np.array([5, 6]), np.array([1], np.int32), np.array([300], np.int32),
                               np.full((1, L, L), 0.1, np.float32))
                g.sweep(2)
            assert np.array_equal(h.get_labels(), fresh.get_labels())
        fresh.close()


def test_set_factors_sorts_long_incidence_lists():
    # a site of 3,000 incidences (the CTA sort) beside short lists, against the oracle
    rng = np.random.default_rng(0)
    n = 3001
    m = wl.Model(n, 3, rng.normal(size=(n, 3)).astype(np.float32), np.zeros(n - 1, np.int32), np.arange(1, n, dtype=np.int32),
                 rng.normal(0, 0.1, (n - 1, 3, 3)).astype(np.float32))
    _check(m, 3, 6000)
