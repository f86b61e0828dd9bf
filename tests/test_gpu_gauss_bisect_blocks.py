"""The one-launch bisection of the Gaussian model against the form of a launch per halving, where
a warp has one chunk of 256 replicas, two, and more (their energies in registers for the first
two, read again for the others): as many blocks as the device holds reach the second only beyond
6e5 replicas and the third beyond 1.2e6, so their number is bounded here.  Also populations so
small that |R~ / R - 1| rules the shortcut out (its condition on the culling fraction needs
0.8 sqrt|R~ / R - 1| below the target).  Every temperature and observable is the same to the bit."""
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


@pytest.mark.parametrize("L,R,eps,bmax,blocks", [
    (4, 3, 0.5, 1.0, 0), (4, 40, 0.1, 1.5, 0), (6, 257, 0.3, 1.5, 0),  # less than a chunk, and two
    (4, 3000, 0.2, 2.0, 1),            # 12 chunks: the warps of one block have one or none
    (4, 5500, 0.272, 2.0, 1),          # 22: one or two
    (4, 12_000, 0.05, 1.0, 1),         # 47: two or three
    (4, 8192, 0.272, 1.0, 1),          # 32: two, the last one full at first
    (4, 60_000, 0.272, 2.0, 2),        # 235 over 32 warps
    (6, 300_000, 0.2, 0.6, 5),         # 1172 over 80 warps, two levels of sums
    (2, 1_300_000, 0.3, 1.0, 0),       # more than two chunks a warp with all blocks of the device
])
def test_chunks_of_a_warp(pa, L, R, eps, bmax, blocks):
    runs = []
    for one_launch in (1, 0):
        r = pa.Run(L, R, 5, 70 + L, None, n_temps=400, beta_max=bmax, eps_target=eps, n_sweeps=1,
                   model=pa.PA_MODEL_GAUSS)
        assert pa.lib().pa_debug_bisect(r._h, one_launch, -1) == pa.PA_OK
        assert pa.lib().pa_debug_bisect_blocks(r._h, blocks) == pa.PA_OK
        runs.append(r)
    t = 0
    while True:
        a, b = runs[0].step(), runs[1].step()
        assert a == b
        if a == pa.PA_DONE:
            break
        t += 1
        for k, v in runs[0].gobs(t).items():
            w = runs[1].gobs(t)[k]
            assert v == w or (v != v and w != w), (t, k, v, w)
    assert t >= 2
    for x, y in zip(runs[0].population(), runs[1].population()):
        assert np.array_equal(x, y)
    assert pa.lib().pa_debug_bisect_blocks(runs[0]._h, -1) == pa.PA_ERR_INVALID
    for r in runs:
        r.close()
