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
