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


@pytest.mark.parametrize("L,R", [(2, 3000), (6, 200), (10, 60), (16, 30)])
@pytest.mark.parametrize("model", [0, 1])
def test_few_replicas_equal_the_population(pa, L, R, model):
    """Read-outs of up to 16384 spins cross the link as rows of bits, larger ones as bytes."""
    run = pa.Run(L, R, 3, 4, np.linspace(0.0, 0.4, 3), n_sweeps=1, model=model)
    run.run()
    spins, labels, _ = run.population()
    N, most = L ** 3, 16384 // L ** 3
    assert len(spins) > most + 4
    out, lab = np.zeros((most + 1, N), dtype=np.int8), np.zeros(most + 1, dtype=np.int32)
    for n in (1, 3, most, most + 1):  # most is 4 at the least
        run.stats_reset()
        rc = pa.lib().pa_get_replicas(run._h, 0, 3, n, pa._p(out, pa.ctypes.c_int8), pa._p(lab, pa.ctypes.c_int32), None)
        assert rc == pa.PA_OK
        assert np.array_equal(out[:n], spins[3:3 + n]) and np.array_equal(lab[:n], labels[3:3 + n])
        row = 4 * ((N + 31) // 32) if N <= 64 else 32 * ((N + 255) // 256)
        assert run.stats()["d2h_bytes"] - 4 * n - 8 == (n * row if n <= most else n * N)  # labels; size and status
    run.close()
