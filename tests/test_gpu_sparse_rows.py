"""Ranks of rows whose first tiles are empty: flatten looks a row's rank up in the first tile where
one of its warp's rows has a run, and carries it on along x from there.  Sparse sites on long
rows, whole rows and planes left empty, every tile shape, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1405_1931_gb300 import hk

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [(8, 8), (16, 8), (16, 16), (32, 8)])
@pytest.mark.parametrize("dims", [(3200, 40, 9), (1037, 33, 20), (70000, 3, 2), (160, 100, 64)])
def test_sparse_rows(dims, tile):
    nx, ny, nz = dims
    rng = np.random.default_rng(nx + tile[0])
    phi = np.full((nz, ny, nx), -1.0, np.float32)
    n = phi.size
    phi.reshape(-1)[rng.choice(n, size=n // 700, replace=False)] = 1.0
    phi[:, :, : nx // 3] = -1.0                       # no run in the first tiles of any row
    phi[:, 1::3, :] = -1.0                            # nor in these rows
    phi[nz // 2] = -1.0
    phi[:, ny - 1, nx // 2:] = 1.0                    # one long run a plane, late in its row
    lab = hk.Labeller(0, tile=tile)
    lab.set_small_path(False)
    for per in ((1, 1, 1), (0, 0, 0)):
        want = oracle.label(phi, per)
        labels, sizes, hist, ncl = lab.label(torch.from_numpy(phi).cuda(), per)
        lab.sync_status()
        assert int(ncl.item()) == want[3]
        np.testing.assert_array_equal(labels.cpu().numpy(), want[0])
        np.testing.assert_array_equal(sizes[:want[3]].cpu().numpy(), want[1])
        np.testing.assert_array_equal(hist.cpu().numpy(), want[2])
    lab.close()
