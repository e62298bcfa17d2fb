"""Where the sizes of a call go: flatten collects them per 32-byte sector of the caller's
buffer, carried from tile to tile along x, so the buffer's place in a sector, the place
where the capacity cuts it and rows of many tiles are checked against the oracle."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_1405_1931_gb300 import fields, hk

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(200, 17, 9), (1023, 16, 5), (64, 33, 48), (516, 5, 3)])
@pytest.mark.parametrize("p", [0.12, 0.3116, 0.5])
def test_sizes_at_every_place_of_a_sector(dims, p):
    nx, ny, nz = dims
    phi_np = fields.iid_field(nx, ny, nz, seed=5, occupancy=p)
    want = oracle.label(phi_np, (1, 0, 1))
    n, full = want[3], (phi_np.size + 1) // 2
    lab = hk.Labeller(0)
    lab.set_small_path(False)
    phi = torch.from_numpy(phi_np).cuda()
    labels, sizes, hist, ncl, _ = lab.alloc_outputs(phi.shape, phi.device, full + 16)
    for off in range(4):
        for cap in (full, n, n - 1, n - 2, n - 3, n // 2, 1):
            sizes.fill_(-7)
            rc = hk.hk_label(lab.ctx, phi.data_ptr(), nx, ny, nz, (1, 0, 1), labels.data_ptr(),
                             sizes.data_ptr() + 8 * off, cap, hist.data_ptr(), ncl.data_ptr(),
                             ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
            lab.sync_status()
            assert rc == (hk.HK_OK if cap >= n else hk.HK_ERR_CAPACITY)
            got = sizes.cpu().numpy()
            k = min(n, cap)
            np.testing.assert_array_equal(got[off:off + k], want[1][:k], err_msg=f"offset {off}, cap {cap}")
            assert (got[:off] == -7).all() and (got[off + k:] == -7).all(), f"offset {off}, cap {cap}"
            np.testing.assert_array_equal(hist.cpu().numpy(), want[2])
            assert int(ncl.item()) == n
    np.testing.assert_array_equal(labels.cpu().numpy(), want[0])
    lab.close()
