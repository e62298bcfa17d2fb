"""Periodic edges inside a tile, whose run pairs are shared out over its threads: axes that fit in
one tile with stripes across x (a chain of links between the two edges in every column), the
site checkerboard and random sites, every tile shape, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1405_1931_gb300 import fields, hk

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def field(kind, dims):
    nx, ny, nz = dims
    if kind == "random":
        return fields.iid_field(nx, ny, nz, seed=2, occupancy=0.45)
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    s = {"stripes1": x, "stripes2": x // 2, "checkerboard": x + y + z}[kind]
    phi = np.where(s % 2 == 0, 1.0, -1.0).astype(np.float32)
    if kind != "checkerboard":
        phi[np.random.default_rng(1).random(phi.shape) < 0.05] *= -1.0
    return phi


@pytest.mark.parametrize("kind", ["stripes1", "stripes2", "checkerboard", "random"])
@pytest.mark.parametrize("dims", [(70, 16, 40), (70, 40, 16), (64, 8, 8), (33, 32, 5), (96, 2, 50), (32, 7, 7), (9, 16, 16)])
def test_axes_of_one_tile(dims, kind):
    phi = field(kind, dims)
    lab = hk.Labeller(0)
    lab.set_small_path(False)
    for tile in ((8, 8), (16, 8), (16, 16), (32, 8)):
        lab.set_tile(*tile)
        for per in ((1, 1, 1), (0, 1, 0), (0, 0, 1)):
            want = oracle.label(phi, per)
            labels, sizes, hist, ncl = lab.label(torch.from_numpy(phi).cuda(), per)
            lab.sync_status()
            assert int(ncl.item()) == want[3], (tile, per)
            np.testing.assert_array_equal(labels.cpu().numpy(), want[0])
            np.testing.assert_array_equal(sizes[:want[3]].cpu().numpy(), want[1])
            np.testing.assert_array_equal(hist.cpu().numpy(), want[2])
    lab.close()
