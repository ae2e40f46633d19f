"""Small models: what several sweeps in one call leave behind equals what the
same sweeps one at a time leave behind."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from tests.gpu_helpers import make_handle
from tests.test_gpu_sweep_forms import SMALL


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1611_06684_gb300 import build
    build.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("name", [n for n in SMALL if n != "single_site"])
def test_dual_words_of_the_last_sweep(name):
    make, C = SMALL[name]
    model = make()
    many, single = (make_handle(model, C, 77, schedule=1, use_graphs=False) for _ in range(2))
    for sweeps in (2, 5):
        many.sweep(sweeps)
        for _ in range(sweeps):
            single.sweep(1)
        assert np.array_equal(many.debug_theta(), single.debug_theta())
    if model.n_edges > 3:                                  # free slots have no bits
        for h in (many, single):
            h.edit_factors(np.array([1, 3]), np.zeros(0, np.int32), np.zeros(0, np.int32),
                           np.zeros((0, model.n_labels, model.n_labels), np.float32))
        many.sweep(3)
        for _ in range(3):
            single.sweep(1)
        assert np.array_equal(many.debug_theta(), single.debug_theta())
        assert not many.debug_theta()[[1, 3]].any()


# sites, edges, chains at the edges of the forms: part-full last groups, one and several CTAs per group,
# more groups than fit at once, dual words on both sides of 200 KB
@pytest.mark.parametrize("L,N,E,C", [(2, 20, 30, 305), (3, 9, 12, 700), (4, 70, 300, 33), (5, 300, 700, 17),
                                     (8, 40, 400, 7), (8, 500, 1300, 40), (10, 60, 150, 9), (11, 30, 60, 13),
                                     (16, 40, 90, 11), (2, 1000, 3000, 16), (2, 1000, 3200, 17)])
def test_several_sweeps_in_one_call_equal_single_sweeps(L, N, E, C):
    from paper_1611_06684_gb300 import workloads as wl
    model = wl.tiny_random(N, L, E, w_std=0.3, seed=100 * L + C)
    many, single = (make_handle(model, C, 31, schedule=1, use_graphs=False) for _ in range(2))
    many.sweep(4)
    many.sweep(3)
    for _ in range(7):
        single.sweep(1)
    assert np.array_equal(many.get_labels(), single.get_labels())
    assert np.array_equal(many.counts(), single.counts())
    assert np.array_equal(many.debug_theta(), single.debug_theta())
