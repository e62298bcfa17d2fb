"""Ranks on lattices of very many rows: past a number of scan blocks their sums get a
pass of their own, below it every block adds up those before it."""
import numpy as np
import pytest

import oracle
from paper_1405_1931_gb300 import fields, hk

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROWS, DIRECT = 1024, 2048   # rows of a scan block; blocks up to which no pass of their own is needed


@pytest.mark.parametrize("ny,nz", [(ROWS, DIRECT - 1), (ROWS, DIRECT), (1025, 2049), (ROWS - 1, 1), (ROWS, 1)])
def test_ranks_of_many_rows(ny, nz):
    phi_np = fields.iid_field(2, ny, nz, seed=9, occupancy=0.3)
    want = oracle.label(phi_np, (0, 1, 1))
    lab = hk.Labeller(0)
    lab.set_small_path(False)
    labels, sizes, hist, ncl = lab.label(torch.from_numpy(phi_np).cuda(), (0, 1, 1))
    lab.sync_status()
    assert int(ncl.item()) == want[3]
    np.testing.assert_array_equal(labels.cpu().numpy(), want[0])
    np.testing.assert_array_equal(sizes[:want[3]].cpu().numpy(), want[1])
    np.testing.assert_array_equal(hist.cpu().numpy(), want[2])
    lab.close()
