"""Output buffers that are not 16-byte aligned beside aligned fields with rows of whole 16-byte
blocks: labels then leave one site a lane after the TMA occupancy pass, alone and in a batch with
aligned lattices, and interior states a byte a lane.  Nothing beside the buffers is written."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_1405_1931_gb300 import fields, hk

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

STREAM = lambda: ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)


@pytest.mark.parametrize("offset", [1, 2, 3])
@pytest.mark.parametrize("dims", [(64, 64, 96), (100, 37, 50), (4, 300, 40), (516, 20, 7)])
def test_labels_at_every_offset(dims, offset):
    nx, ny, nz = dims
    phi_np = fields.iid_field(nx, ny, nz, seed=6, occupancy=0.3116)
    want = oracle.label(phi_np, (1, 1, 0))
    phi = torch.from_numpy(phi_np).cuda()
    assert phi.data_ptr() % 16 == 0
    n = phi.numel()
    lab = hk.Labeller(0)
    lab.set_small_path(False)
    _, sizes, hist, ncl, cap = lab.alloc_outputs(phi.shape, phi.device)
    for batched in (False, True):
        buf = torch.full((n + 8,), -7, dtype=torch.int32, device="cuda")
        out = buf[offset:offset + n].view(nz, ny, nx)
        if batched:
            other = lab.alloc_outputs(phi.shape, phi.device)
            lab.label_batched([(phi, (1, 1, 0), other), (phi, (1, 1, 0), (out, sizes, hist, ncl, cap))])
            np.testing.assert_array_equal(other[0].cpu().numpy(), want[0])
        else:
            lab.label(phi, (1, 1, 0), out=(out, sizes, hist, ncl, cap))
        lab.sync_status()
        got = buf.cpu().numpy()
        np.testing.assert_array_equal(got[offset:offset + n].reshape(nz, ny, nx), want[0])
        assert (got[:offset] == -7).all() and (got[offset + n:] == -7).all()
        np.testing.assert_array_equal(sizes[:want[3]].cpu().numpy(), want[1])
        assert int(ncl.item()) == want[3]
    lab.close()


@pytest.mark.parametrize("offset", [1, 2, 4, 8])
@pytest.mark.parametrize("dims", [(64, 33, 20), (16, 16, 16), (112, 9, 40)])
def test_states_at_every_offset(dims, offset):
    nx, ny, nz = dims
    rng = np.random.default_rng(nx)
    index = rng.choice(np.array([-1.0, -0.5, -0.25, 0.0, 0.25, np.nan], np.float32), size=(nz, ny, nx),
                       p=[0.8, 0.02, 0.08, 0.01, 0.08, 0.01])
    want = oracle.interior_state(index, (0, 1, 1))
    n = index.size
    buf = torch.full((n + 32,), 7, dtype=torch.int8, device="cuda")
    lab = hk.Labeller(0)
    d = torch.from_numpy(index).cuda()
    rc = hk.hk_interior_state(lab.ctx, d.data_ptr(), nx, ny, nz, (0, 1, 1), buf.data_ptr() + offset, STREAM())
    assert rc == hk.HK_OK
    lab.sync_status()
    got = buf.cpu().numpy()
    np.testing.assert_array_equal(got[offset:offset + n].reshape(nz, ny, nx), want)
    assert (got[:offset] == 7).all() and (got[offset + n:] == 7).all()
    lab.close()
