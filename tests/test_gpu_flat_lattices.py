"""Lattices of so many tiles that the default slices of the piece table would run out of 31-bit
ids: flat and thin ones, whose tiles lie mostly outside them, get slices of their own bound.
Labels, sizes, histogram and interior state against the oracle; small shapes of the same kind,
with the default slices, go through the other GPU tests."""
import numpy as np
import pytest

import oracle
from paper_1405_1931_gb300 import hk

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.slow]

# 16 x 16 tiles of 1280 ids each: more than 1,677,721 tiles
SHAPES = [((1, 27_000_000, 1), 0.95), ((1, 1, 27_000_000), 0.97), ((53_760_000, 1, 1), 0.99),
          ((53_760_001, 1, 1), 0.98), ((2, 26_900_000, 2), 0.8), ((1, 20800, 20800), 0.58)]


@pytest.fixture(scope="module")
def lab():
    lab = hk.Labeller(0)
    yield lab
    lab.close()


@pytest.mark.parametrize("dims,p", SHAPES)
def test_labels(lab, dims, p):
    nx, ny, nz = dims
    assert -(-nx // 32) * -(-ny // 16) * -(-nz // 16) * 1280 >= 2 ** 31
    phi = torch.empty((nz, ny, nx), dtype=torch.float32, device="cuda")
    assert hk.hk_gen_iid(phi.data_ptr(), nx, ny, nz, 3, p, 0) == 0
    per = (1, 1, 1) if nx % 2 else (0, 1, 0)
    labels, sizes, hist, ncl = lab.label(phi, per)
    lab.sync_status()
    want = oracle.label(phi.cpu().numpy(), per)
    assert int(ncl.item()) == want[3]
    assert np.array_equal(labels.cpu().numpy(), want[0])
    assert np.array_equal(sizes[:want[3]].cpu().numpy(), want[1])
    assert np.array_equal(hist.cpu().numpy(), want[2])


@pytest.mark.parametrize("dims", [(1, 27_000_000, 1), (53_760_000, 1, 1)])
def test_interior_state(lab, dims):
    nx, ny, nz = dims
    index = torch.rand((nz, ny, nx), device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    index = torch.where(index < 0.97, -1.0, (index - 0.985) * 10.0).contiguous()   # near sites of either sign
    state = lab.interior_state(index, (1, 1, 1))
    lab.sync_status()
    assert np.array_equal(state.cpu().numpy(), oracle.interior_state(index.cpu().numpy(), (1, 1, 1)))
