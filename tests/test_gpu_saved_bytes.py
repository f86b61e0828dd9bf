"""What leaves the library as bytes: a checkpoint depends on the run alone."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pa():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_02146_gb300 import build, pa as pa_mod
    build.build()
    return pa_mod


def test_gaussian_checkpoint_holds_no_stale_memory(pa):
    """Two equal runs save the same bytes, whatever the runs before them left in the memory they take."""
    saved = []
    for model in (pa.PA_MODEL_PM1, pa.PA_MODEL_GAUSS):
        before = pa.Run(10, 3000, 1, 2, np.linspace(0.0, 1.0, 40), n_sweeps=1, model=model)
        before.run()
        before.close()
        run = pa.Run(6, 500, 5, 7, np.linspace(0.0, 1.0, 6), n_sweeps=2, n_pop=2, model=pa.PA_MODEL_GAUSS)
        run.step()
        run.step()
        saved.append(run.checkpoint())
        run.close()
    assert saved[0] == saved[1]
