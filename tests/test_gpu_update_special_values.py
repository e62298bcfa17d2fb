"""The in-place update of large fields, whose far sectors are left alone: what makes a sector
near is one site that is not below -0.5, whatever it holds -- NaN, -0.5 itself, zeros of
either sign, infinities -- and what keeps it far may be any value below."""
import numpy as np
import pytest

import oracle
from paper_1405_1931_gb300 import hk

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BELOW = np.nextafter(np.float32(-0.5), np.float32(-1.0))
NEAR = np.array([np.nan, -0.5, -0.25, -0.0, 0.0, 0.25, 0.5, 1e-30, np.inf], np.float32)
FAR = np.array([-1.0, BELOW, -3e38, -np.inf], np.float32)


@pytest.mark.parametrize("off_i,off_s", [(0, 0), (4, 16), (1, 0), (0, 3)])
def test_special_values(off_i, off_s):
    n = (1 << 25) + 77
    rng = np.random.default_rng(11 + off_i + off_s)
    index = np.full(n, -1.0, np.float32)
    alone = rng.choice(n // 32, size=20000, replace=False) * 32 + rng.integers(0, 32, 20000)   # one near site a sector
    index[alone] = rng.choice(NEAR, size=alone.size)
    index[: 1 << 20] = rng.choice(np.concatenate([NEAR, FAR]), size=1 << 20)
    index[1 << 21: (1 << 21) + 100000] = rng.choice(NEAR, size=100000)
    index[3 << 20: (3 << 20) + 100000] = rng.choice(FAR, size=100000)
    prev = rng.integers(-1, 2, size=n).astype(np.int8)
    want = oracle.interior_update(prev.reshape(1, 1, n), index.reshape(1, 1, n)).reshape(-1)
    d_index = torch.full((n + 8,), 0.25, device="cuda")
    d_state = torch.full((n + 32,), 9, dtype=torch.int8, device="cuda")
    d_index[off_i:off_i + n] = torch.from_numpy(index).cuda()
    d_state[off_s:off_s + n] = torch.from_numpy(prev).cuda()
    hk.interior_update(d_state[off_s:off_s + n], d_index[off_i:off_i + n])
    got = d_state.cpu().numpy()
    np.testing.assert_array_equal(got[off_s:off_s + n], want)
    assert (got[:off_s] == 9).all() and (got[off_s + n:] == 9).all()
