"""Populations of more words than the sizes of the parity tests reach: large lattices over several
blocks of the level count (32 words), of the transposes (8 words) and more words than a warp has
lanes, and Gaussian pairs over more than one wave of tiles, whose second sweep starts while the
first runs.  Populations, histograms and counts are the oracle's."""
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


def pair(pa, oracle_lib, L, R, betas, n_sweeps, n_pop, model):
    gpu = pa.Run(L, R, L, 7 + R, betas, n_sweeps=n_sweeps, n_pop=n_pop, model=model)
    make = oracle_lib.GRun if model == pa.PA_MODEL_GAUSS else oracle_lib.Run
    return gpu, make(oracle_lib.RunConfig(L=L, R=R, disorder_seed=L, run_seed=7 + R, betas=betas, n_sweeps=n_sweeps,
                                          n_pop=n_pop))


def assert_populations(gpu, ref, n_pop, t):
    for p in range(n_pop):
        assert np.array_equal(gpu.copy_counts(p), ref.last_counts(p)), f"t={t} pop {p}: copy numbers"
        for a, b, what in zip(gpu.population(p), ref.population(p), ("spins", "labels", "energies")):
            assert np.array_equal(a, b), f"t={t} pop {p}: {what}"


@pytest.mark.parametrize("L,R,T,n_pop", [(18, 1100, 3, 2), (18, 2100, 3, 2), (24, 1055, 2, 1), (18, 20_001, 2, 1)])
def test_large_lattices(pa, oracle_lib, L, R, T, n_pop):
    gpu, ref = pair(pa, oracle_lib, L, R, np.linspace(0.0, 1.0, T), 2 if R < 10_000 else 1, n_pop, pa.PA_MODEL_PM1)
    for t in range(1, T):
        assert gpu.step() == 0
        ref.step()
        assert_populations(gpu, ref, n_pop, t)
        for p in range(n_pop):
            assert np.array_equal(gpu.energy_hist(t, p), ref.energy_hist(t, p))
            for k in ("R_tilde", "sum_E", "sum_E2", "E_min", "sum_eta2", "n_families"):
                assert gpu.obs(t, p)[k] == ref.obs(t, p)[k], k
        if n_pop == 2:
            assert np.array_equal(gpu.q_hist(t), ref.q_hist(t))
    gpu.close()


# a little more than the 311 296 slots of one wave of tiles on 152 SMs
@pytest.mark.parametrize("L,R", [(2, 320_000), (4, 330_000)])
def test_gaussian_pairs(pa, oracle_lib, L, R):
    betas = np.linspace(0.0, 1.0, 3)
    gpu, ref = pair(pa, oracle_lib, L, R, betas, 1, 2, pa.PA_MODEL_GAUSS)
    for _ in betas[1:]:  # issued without a wait, so that every step meets the one before
        gpu.step()
        ref.step()
    assert_populations(gpu, ref, 2, gpu.t)
    for t in range(len(betas)):
        for p in range(2):
            for k in ("R_tilde", "sum_E", "E_min", "sum_eta2", "n_families", "ql_sum"):
                assert gpu.gobs(t, p)[k] == ref.obs(t, p)[k], (t, p, k)
        assert np.array_equal(gpu.q_hist(t), ref.q_hist(t))
        assert np.array_equal(gpu.ql_hist(t), ref.q_hist(t, link=True))
    gpu.close()
