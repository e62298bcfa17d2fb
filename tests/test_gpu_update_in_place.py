"""The in-place update writes the near sites and no other byte, at every alignment of the
two arrays and every length of the last group."""
import numpy as np
import pytest

import oracle
from paper_1405_1931_gb300 import hk

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3, 4, 5, 31, 4096, 100003])
@pytest.mark.parametrize("density", [0.0, 0.02, 1.0])
def test_in_place(n, density):
    rng = np.random.default_rng(n)
    near = np.array([-0.5, -0.25, -0.0, 0.0, 0.25, 0.5, np.nan, np.inf], np.float32)
    I = np.where(rng.random(n) < density, rng.choice(near, size=n), np.float32(-1.0)).astype(np.float32)
    prev = rng.integers(-1, 2, size=n).astype(np.int8)
    want = oracle.interior_update(prev.reshape(1, 1, n), I.reshape(1, 1, n)).reshape(-1)
    for off_i in (0, 1):
        for off_s in range(5):
            index = torch.full((n + 8,), 0.25, device="cuda")
            state = torch.full((n + 16,), 9, dtype=torch.int8, device="cuda")
            index[off_i:off_i + n] = torch.from_numpy(I).cuda()
            state[off_s:off_s + n] = torch.from_numpy(prev).cuda()
            hk.interior_update(state[off_s:off_s + n], index[off_i:off_i + n])
            got = state.cpu().numpy()
            np.testing.assert_array_equal(got[off_s:off_s + n], want)
            assert (got[:off_s] == 9).all() and (got[off_s + n:] == 9).all()


@pytest.mark.parametrize("off_i,off_s", [(0, 0), (1, 0), (0, 4)])
def test_in_place_large(off_i, off_s):
    """From 2^25 sites on, with stretches full of near sites, sparse ones and a ragged end."""
    n = (1 << 25) + 45
    rng = np.random.default_rng(off_i + off_s)
    density = np.repeat(rng.choice([0.0, 0.01, 0.3, 1.0], size=n // 5000 + 1), 5000)[:n]
    I = np.where(rng.random(n, dtype=np.float32) < density, np.where(rng.random(n) < 0.5, -0.25, 0.25), -1.0)
    I = I.astype(np.float32)
    prev = rng.integers(-1, 2, size=n).astype(np.int8)
    want = oracle.interior_update(prev.reshape(1, 1, n), I.reshape(1, 1, n)).reshape(-1)
    index = torch.full((n + 8,), 0.25, device="cuda")
    state = torch.full((n + 16,), 9, dtype=torch.int8, device="cuda")
    index[off_i:off_i + n] = torch.from_numpy(I).cuda()
    state[off_s:off_s + n] = torch.from_numpy(prev).cuda()
    hk.interior_update(state[off_s:off_s + n], index[off_i:off_i + n])
    got = state.cpu().numpy()
    np.testing.assert_array_equal(got[off_s:off_s + n], want)
    assert (got[:off_s] == 9).all() and (got[off_s + n:] == 9).all()
