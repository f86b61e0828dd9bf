"""The population as one bit per spin in replica rows: whatever reads or rewrites the
rows agrees with numpy on the spins handed out, at sizes whose rows end inside a word
(L = 2, 6, 10, 14, 18) or in padding words (L = 6, 12, 14), for ragged populations."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [(2, 37), (4, 1100), (6, 333), (8, 257), (10, 1057), (12, 70), (14, 131), (16, 65), (18, 300)]


@pytest.fixture(scope="module")
def pa():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_02146_gb300 import build, pa as pa_mod
    build.build()
    return pa_mod


def lattice(s, L):
    return s.reshape(len(s), L, L, L).astype(np.int64)  # [replica, z, y, x]


def bond_products(s, L):
    """s_n s_m of every forward bond, [replica, n, d] with n = x + L (y + L z)."""
    c = lattice(s, L)
    return np.stack([(c * np.roll(c, -1, axis=ax)).reshape(len(s), -1) for ax in (3, 2, 1)], axis=2)


def overlap_hist(v, full, bins):
    b = ((v + full) * (bins - 1) + full) // (2 * full)
    return np.bincount(b, minlength=bins)


@pytest.mark.parametrize("model", [0, 1])
@pytest.mark.parametrize("L,R", SIZES)
def test_rows_agree_with_the_spins_read_out(pa, L, R, model):
    if model and L > 16:
        pytest.skip("Gaussian couplings go up to L = 16")
    kw = dict(n_sweeps=1, n_pop=2, model=model)
    betas = np.array([0.0, 0.4, 0.8])
    run = pa.Run(L, R, 5, 9, betas, **kw)
    for t in range(3):
        if t:
            assert run.step() == 0
        pops = [run.population(p) for p in (0, 1)]
        for s, _, E in pops:
            assert set(np.unique(s)) <= {-1, 1}
            J = (run.gcouplings() if model else run.couplings().astype(np.int64)).astype(np.int64).reshape(-1, 3)
            assert np.array_equal(-(bond_products(s, L) * J).sum(axis=(1, 2)), E)
        n = min(len(pops[0][0]), len(pops[1][0]))
        c = pops[0][0][:n].astype(np.int64) * pops[1][0][:n]
        assert np.array_equal(overlap_hist(c.sum(axis=1), L ** 3, 65), run.q_hist(t))
        if model:
            ql = bond_products(c, L).sum(axis=(1, 2))
            assert np.array_equal(overlap_hist(ql, 3 * L ** 3, 65), run.ql_hist(t))
            assert run.gobs(t)["ql_sum"] == ql.sum()
        else:
            first = len(pops[1][0]) // 3
            part = run.replicas(1, first, len(pops[1][0]) - first - 1)
            for a, b in zip(part, pops[1]):
                assert np.array_equal(a, b[first:-1])
        if t == 1:
            saved = run.checkpoint()
    resumed = pa.Run(L, R, 5, 9, betas, checkpoint=saved, **kw)
    assert resumed.checkpoint() == saved
    assert resumed.step() == 0
    for p in (0, 1):
        for a, b in zip(resumed.population(p), pops[p]):
            assert np.array_equal(a, b)
    assert np.array_equal(resumed.q_hist(2), run.q_hist(2))
    run.close()
    resumed.close()
