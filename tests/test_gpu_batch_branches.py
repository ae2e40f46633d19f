"""Captured batch rounds run the classes in parallel branches where they are
small and one after another where each fills the GPU: both equal the rounds of
direct launches."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_1611_06684_gb300 import workloads as wl


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1611_06684_gb300 import build
    build.build()
    torch.cuda.set_device(0)


# 2 x 10^4 edges per graph: 4.5 and 18.5 million dual words, on both sides of 2^24
@pytest.mark.parametrize("C", [32, 132])
def test_captured_rounds_equal_direct_launches(C):
    import torch
    from paper_1611_06684_gb300 import mrf as M
    models = [wl.random_graph(10000, k=2, L=L, seed=s, w_std=0.3) for s, L in enumerate((2, 4, 2, 4, 3, 6, 3))]
    stream = torch.cuda.Stream()
    batches = []
    for graphs in (True, False):
        b = M.MRFBatch([m.n_vars for m in models], [m.n_labels for m in models], C, seed=4, use_graphs=graphs,
                       stream=stream.cuda_stream, schedule=1)
        b.set_factors(models)
        b.queue_create(2000, 2000, 2000 * 36, extra_slots=64)
        batches.append((b, wl.ErBatchEdits(models, [b.graph(g).first_edge_slot for g in range(len(models))], seed=1)))
    for n_sweeps in (2, 2, 3):
        slots = []
        for b, ed in batches:
            arrays = ed.edit(0.01)
            b.queue_load(*arrays)
            b.round(n_sweeps)
            status, new = b.queue_result(len(arrays[3]))
            assert status == 0
            ed.apply(new)
            slots.append(new)
        assert np.array_equal(*slots)
    for g in range(len(models)):
        assert np.array_equal(batches[0][0].get_labels(g), batches[1][0].get_labels(g))
        assert np.array_equal(batches[0][0].counts(g), batches[1][0].counts(g))
