"""The one-launch kernels on fields whose links make the longest chains -- stripes across x, one
run on top of the other through the whole lattice, joined at their far ends by the periodic
edges -- and on thin lattices of one or two columns, against the oracle."""
import itertools

import numpy as np
import pytest

import oracle
from paper_1405_1931_gb300 import hk

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def stripes(shape, axis, width):
    nx, ny, nz = shape
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    return np.where(((x, y, z)[axis] // width) % 2 == 0, 1.0, -1.0).astype(np.float32)


def check(lab, phi, per, what):
    want = oracle.label(phi, per)
    labels, sizes, hist, ncl = lab.label(torch.from_numpy(phi).cuda(), per)
    lab.sync_status()
    assert int(ncl.item()) == want[3], what
    np.testing.assert_array_equal(labels.cpu().numpy(), want[0], err_msg=what)
    np.testing.assert_array_equal(sizes[:want[3]].cpu().numpy(), want[1], err_msg=what)
    np.testing.assert_array_equal(hist.cpu().numpy(), want[2], err_msg=what)


SHAPES = [(32, 32, 32), (31, 33, 29), (40, 40, 40), (64, 64, 64), (33, 40, 40), (2, 64, 128), (1, 1, 2048), (1, 1, 16384),
          (5, 1000, 3), (16, 2, 1000), (9, 24, 24), (64, 24, 2)]


@pytest.mark.parametrize("path", [2, 3])
@pytest.mark.parametrize("shape", SHAPES)
def test_stripes(shape, path):
    lab = hk.Labeller(0)
    lab.set_small_path(path)
    for axis, width in [(0, 1), (0, 3), (1, 1), (2, 2)]:
        for per in itertools.product((0, 1), repeat=3):
            check(lab, stripes(shape, axis, width), per, f"{shape} stripes {axis} {width} {per}")
    phi = stripes(shape, 0, 1)                      # the stripes cut here and there
    phi[np.random.default_rng(4).random(phi.shape) < 0.02] *= -1.0
    check(lab, phi, (1, 1, 1), f"{shape} cut stripes")
    lab.close()
