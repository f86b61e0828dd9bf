"""A step's sweep launches (two populations, a split last wave) run over each other's ends;
the fused batch advances the same runs with one launch per step: everything is equal."""
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


# fewer tiles than SMs, a little over one wave, a split last wave, and less than one tile
@pytest.mark.parametrize("L,R,n_pop", [(8, 100_000, 2), (10, 170_000, 2), (10, 170_000, 1), (6, 31, 2)])
def test_overlapped_launches_equal_fused_rounds(pa, L, R, n_pop):
    from paper_1711_02146_gb300.workloads import Workload
    w = Workload("overlap", L=L, R=R, disorder_seed=3, run_seed=4, betas=np.linspace(0.0, 1.5, 6), n_temps=6,
                 n_sweeps=1, n_pop=n_pop)
    run = pa.Run.from_workload(w)
    for _ in range(5):  # issued without a wait, so that every step meets the one before
        run.step()
    batch = pa.Batch([w])
    batch.run()
    view = batch.run_view(0)
    for p in range(n_pop):
        for t in range(6):
            assert run.obs(t, p) == view.obs(t, p)
            assert np.array_equal(run.energy_hist(t, p), view.energy_hist(t, p))
        for a, b in zip(run.population(p), view.population(p)):
            assert np.array_equal(a, b)
    if n_pop == 2:
        assert np.array_equal(run.q_hist(5), view.q_hist(5))
    run.close()
    batch.close()
