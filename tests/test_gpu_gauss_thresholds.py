"""The Metropolis thresholds of the Gaussian model, entry by entry: the device computes them and
lists those whose floor the last bits of its exponential could decide, the host evaluates the
listed ones.  Every entry is compared with its definition, min(floor(2^32 exp(-beta dE)), 2^32 - 2)
with the C library's exponential, where NumPy's leaves it open (both are within an ulp), and with
NumPy's elsewhere.  Lists that fill, overflow or find no pinned memory give the same tables."""
import ctypes
import math

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


def flip_costs(L, Jq):
    """dE (units of 2^-20) of flipping site n under pattern b, [N, 64]."""
    J = Jq.astype(np.int64).reshape(L, L, L, 3)  # z, y, x, direction
    bonds = [J[..., 0], np.roll(J[..., 0], 1, 2), J[..., 1], np.roll(J[..., 1], 1, 1), J[..., 2],
             np.roll(J[..., 2], 1, 0)]
    sign = 1 - 2 * ((np.arange(64)[None, :] >> np.arange(6)[:, None]) & 1)  # [6, 64]
    return 2 * np.stack([b.reshape(-1) for b in bonds], 1) @ sign


def expected(dE, beta):
    """The table of beta, and its entries that 2^-50 of v (as the device lists them) leaves open."""
    v = np.exp(-(beta * (np.maximum(dE, 0) * 2.0 ** -20))) * 2.0 ** 32
    tol = v * 2.0 ** -50
    top = 4294967294.0
    lo, hi = (np.minimum(np.floor(v + s * tol), top) for s in (-1, 1))
    want = np.where(dE > 0, lo, 4294967295.0)
    is_open = np.argwhere((dE > 0) & (lo != hi))
    for n, b in is_open:
        want[n, b] = min(math.floor(math.exp(-(beta * (float(dE[n, b]) * 2.0 ** -20))) * 2.0 ** 32), top)
    return want.astype(np.uint32), len(is_open)


def table(pa, run, t):
    out = np.zeros(64 * run.N, dtype=np.uint32)
    rc = pa.lib().pa_get_thresholds(run._h, t, out.ctypes.data_as(ctypes.POINTER(ctypes.c_uint32)), out.size)
    assert rc == pa.PA_OK
    return out.reshape(run.N, 64)


@pytest.mark.parametrize("L,T,beta_max", [(2, 3001, 0.1), (6, 101, 0.3), (10, 41, 0.3), (16, 9, 0.1)])
@pytest.mark.parametrize("cap", [-1, 0, 1])
def test_explicit_schedule(pa, L, T, beta_max, cap):
    betas = np.concatenate([[0.0, 0.0, 1e-9], np.linspace(0.0, beta_max, T)[1:], [40.0]])
    run = pa.Run(L, 10, 7, 8, betas, n_sweeps=1, model=pa.PA_MODEL_GAUSS)
    dE = flip_costs(L, run.gcouplings())
    if cap >= 0:
        assert pa.lib().pa_debug_thresholds(run._h, cap, 1) == pa.PA_OK
    n_open = 0
    for t in range(1, len(betas)):
        want, k = expected(dE, betas[t])
        n_open += k
        assert np.array_equal(table(pa, run, t), want), f"t={t}"
    assert n_open > 1  # so that caps of 0 and 1 overflow
    run.close()


def test_list_of_a_long_schedule(pa):
    """More open entries than one step's list holds: all of them are settled one by one, and no
    whole table (442 KB each, 442 MB in all) comes from the host."""
    L, betas = 12, np.linspace(0.0, 1.0, 1001)
    run = pa.Run(L, 10, 5, 7, betas, n_sweeps=1, model=pa.PA_MODEL_GAUSS)
    assert run.stats()["h2d_bytes"] < 64 << 20
    dE = flip_costs(L, run.gcouplings())
    n_open = 0
    for t in range(1, len(betas)):
        want, k = expected(dE, betas[t])
        n_open += k
        if k or t % 50 == 0:
            assert np.array_equal(table(pa, run, t), want), f"t={t}"
    assert n_open > 127
    run.close()


@pytest.mark.parametrize("cap,pinned", [(-1, 1), (-1, 0), (0, 1), (0, 0)])
def test_adaptive_steps(pa, cap, pinned):
    L = 14
    run = pa.Run(L, 400, 9, 10, None, n_temps=100, beta_max=1.0, eps_target=0.05, n_sweeps=1,
                 model=pa.PA_MODEL_GAUSS)
    assert pa.lib().pa_debug_thresholds(run._h, cap, pinned) == pa.PA_OK
    dE = flip_costs(L, run.gcouplings())
    n_open = 0
    for t in range(1, 31):
        assert run.step() == pa.PA_OK
        want, k = expected(dE, run.beta(t))
        n_open += k
        assert np.array_equal(table(pa, run, t), want), f"t={t}"
    assert n_open > 1
    out = np.zeros(64 * run.N, dtype=np.uint32)
    ptr = out.ctypes.data_as(ctypes.POINTER(ctypes.c_uint32))
    assert pa.lib().pa_get_thresholds(run._h, 29, ptr, out.size) == pa.PA_ERR_STATE
    run.close()


def test_wrong_calls_are_refused(pa):
    pm1 = pa.Run(4, 100, 1, 1, np.linspace(0, 1, 3))
    run = pa.Run(4, 100, 1, 1, np.linspace(0, 1, 3), model=pa.PA_MODEL_GAUSS)
    out = np.zeros(64 * 64, dtype=np.uint32)
    ptr = out.ctypes.data_as(ctypes.POINTER(ctypes.c_uint32))
    f, g = pa.lib().pa_debug_thresholds, pa.lib().pa_get_thresholds
    for args in ((pm1._h, -1, 1), (run._h, -2, 1), (run._h, -1, 2)):
        assert f(*args) == pa.PA_ERR_INVALID
    for args in ((pm1._h, 1, ptr, out.size), (run._h, 0, ptr, out.size), (run._h, 3, ptr, out.size)):
        assert g(*args) == pa.PA_ERR_INVALID
    assert g(run._h, 1, ptr, out.size - 1) == pa.PA_ERR_CAPACITY
    for r in (pm1, run):
        r.close()
