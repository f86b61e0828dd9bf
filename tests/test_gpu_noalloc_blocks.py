"""pa_resample_counts_noalloc at the sizes where its second kernel's split of the slots changes:
a counting block of 1024 slots to a block up to 2048 of them, two to a block beyond, with and
without a remainder, up to the largest population accepted."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EDGE = 2048 * 1024


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_02146_gb300 import build, pa
    build.build()
    return torch, pa


@pytest.mark.parametrize("n_old", [1, 1024, EDGE - 1, EDGE, EDGE + 1, EDGE + 1024, EDGE + 1025, 2 * EDGE - 1023, 2 * EDGE])
@pytest.mark.parametrize("invalid", [False, True])
def test_every_split_against_the_oracle(env, oracle_lib, n_old, invalid):
    torch, pa = env
    rng = np.random.default_rng(n_old)
    n_levels, run_seed, t = 301, 77, 5
    levels = rng.integers(0, n_levels - 1, n_old).astype(np.int32)
    fl = rng.integers(0, 3, n_levels).astype(np.int32)
    thr = rng.integers(0, 2 ** 32, n_levels, dtype=np.uint64).astype(np.uint32)
    want = oracle_lib.copy_counts(run_seed, 0, t, levels, fl, thr)
    total, n_new_want = int(want.astype(np.int64).sum()), int(want.astype(np.int64).sum())
    if invalid:  # the last slot's level lies above the tables
        levels[-1] = n_levels
        n_new_want = -1
    dev = [torch.from_numpy(a).cuda() for a in (levels, fl, thr.view(np.int32))]
    counts = torch.full((n_old,), -7, dtype=torch.int32, device="cuda")
    cap = total + 100
    parents = torch.full((cap,), -1, dtype=torch.int32, device="cuda")
    n_new = torch.zeros(1, dtype=torch.int64, device="cuda")
    rc = pa.resample_counts_noalloc(dev[0].data_ptr(), n_old, dev[1].data_ptr(), dev[2].data_ptr(), n_levels, run_seed,
                                    0, t, counts.data_ptr(), parents.data_ptr(), cap, n_new.data_ptr(),
                                    torch.cuda.current_stream())
    assert rc == pa.PA_OK
    p, c = parents.cpu().numpy(), counts.cpu().numpy()
    assert int(n_new.item()) == n_new_want
    if invalid:
        assert np.all(p == -1) and c[-1] == 0 and np.array_equal(c[:-1], want[:-1])
    else:
        assert np.array_equal(c, want)
        assert np.array_equal(p[:total], np.repeat(np.arange(n_old, dtype=np.int32), want))
        assert np.all(p[total:] == -1)
