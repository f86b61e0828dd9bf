"""The Gaussian sweep's comparison of 16 random bits with the upper halves of the
thresholds, where it can go wrong: thresholds whose upper half is zero or all ones (dE
just above zero, beta near zero) or that vanish (large beta), and enough updates that
uniforms equal the threshold's upper half many times.  Spins, labels and energies are the
oracle's bit for bit."""
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


@pytest.mark.parametrize("L,R,n_sweeps", [(2, 1100, 40), (4, 1300, 20), (6, 530, 10), (8, 300, 8), (10, 270, 5),
                                          (12, 260, 3), (14, 129, 2), (16, 65, 2)])
def test_comparison_edges_match_the_oracle(pa, oracle_lib, L, R, n_sweeps):
    betas = np.array([0.0, 1e-9, 1e-4, 0.5, 1.0, 2.0, 40.0])
    gpu = pa.Run(L, R, 11, 12, betas, n_sweeps=n_sweeps, model=pa.PA_MODEL_GAUSS)
    ref = oracle_lib.GRun(oracle_lib.RunConfig(L=L, R=R, disorder_seed=11, run_seed=12, betas=betas,
                                                   n_sweeps=n_sweeps))
    for t in range(1, len(betas)):
        assert gpu.step() == 0
        ref.step()
        for a, b, what in zip(gpu.population(0), ref.population(0), ("spins", "labels", "energies")):
            assert np.array_equal(a, b), f"beta={betas[t]}: {what}"
    gpu.close()
