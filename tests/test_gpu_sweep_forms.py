"""The forms of the sweep's eight-plane comparison: the thresholds' leading zero bits
choose the form of a step, so a schedule that steps across each line (beta about 0.347,
0.693 and 1.386, and beyond where thresholds vanish) is checked against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BETAS = np.array([0.0, 0.2, 0.346, 0.347, 0.6931, 0.6932, 1.386, 1.387, 1.85, 2.78, 4.2, 5.6])


@pytest.fixture(scope="module")
def pa():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_02146_gb300 import build, pa as pa_mod
    build.build()
    return pa_mod


@pytest.mark.parametrize("L,R", [(2, 500), (4, 900), (8, 600), (10, 140), (14, 70), (18, 40)])
def test_every_form_matches_the_oracle(pa, oracle_lib, L, R):
    gpu = pa.Run(L, R, 3, 4, BETAS, n_sweeps=3)
    ref = oracle_lib.Run(oracle_lib.RunConfig(L=L, R=R, disorder_seed=3, run_seed=4, betas=BETAS, n_sweeps=3))
    for t in range(1, len(BETAS)):
        assert gpu.step() == 0
        ref.step()
        for a, b in zip(gpu.population(0), ref.population(0)):
            assert np.array_equal(a, b), f"L={L} beta={BETAS[t]}"
    gpu.close()
