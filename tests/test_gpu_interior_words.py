"""Votes counted on row words: index fields whose near sites sit on every edge a word can
have -- across tiles, across periodic edges (of axes of one tile, of two sites, of one),
ragged ends -- and dense ones that the second tile pass takes, for every tile shape."""
import numpy as np
import pytest

import oracle
from paper_1405_1931_gb300 import hk

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

VALUES = np.array([-1.0, -0.5, -0.25, -0.0, 0.0, 0.25, 0.5, np.nan, np.inf, -np.inf], dtype=np.float32)
FAR_MOSTLY = [0.62, 0.06, 0.1, 0.01, 0.01, 0.1, 0.06, 0.01, 0.02, 0.01]


def field(shape, kind):
    rng = np.random.default_rng(sum(shape) + len(kind))
    if kind == "mixed":
        return rng.choice(VALUES, size=shape, p=FAR_MOSTLY).astype(np.float32)
    z, y, x = np.indices(shape)
    near = rng.choice(np.array([-0.25, 0.25], np.float32), size=shape)
    return np.where((x + y + z) % 2 == 0, np.float32(-1.0), near).astype(np.float32)   # 16 runs a row


@pytest.mark.parametrize("kind", ["mixed", "checkerboard"])
@pytest.mark.parametrize("shape", [(17, 33, 65), (16, 16, 32), (2, 2, 2), (1, 1, 3), (33, 1, 64), (16, 40, 48), (9, 2, 95)])
def test_tags_and_states(shape, kind):
    I = field(shape, kind)
    d = torch.from_numpy(I).cuda()
    lab = hk.Labeller(0)
    for tile in ((8, 8), (16, 8), (16, 16), (32, 8)):
        lab.set_tile(*tile)
        for per in ((1, 1, 1), (0, 0, 0), (1, 0, 1), (0, 1, 0)):
            what = f"{shape} {kind} tile {tile} per {per}"
            want = oracle.interior(I, per)
            labels, sizes, hist, ncl, inside = lab.label_interior(d, per)
            n = int(ncl.item())
            np.testing.assert_array_equal(labels.cpu().numpy(), want[0], err_msg=what)
            np.testing.assert_array_equal(sizes[:n].cpu().numpy(), want[1], err_msg=what)
            np.testing.assert_array_equal(inside[:n].cpu().numpy(), want[4][:n], err_msg=what)
            state = torch.full(shape, 7, dtype=torch.int8, device="cuda")
            lab.interior_state(d, per, out=state)
            np.testing.assert_array_equal(state.cpu().numpy(), oracle.interior_state(I, per), err_msg=what)
            lab.sync_status()
    lab.close()


def test_tags_stop_at_the_capacity():
    I = field((17, 33, 65), "mixed")
    want = oracle.interior(I, (1, 1, 0))
    n = want[3]
    lab = hk.Labeller(0)
    for cap in (1, n // 2, n - 1, n):
        d = torch.from_numpy(I).cuda()
        labels, sizes, hist, ncl, _ = lab.alloc_outputs(d.shape, d.device, cap)
        inside = torch.full((n + 4,), 7, dtype=torch.int8, device="cuda")
        rc = hk.hk_label_interior(lab.ctx, d.data_ptr(), 65, 33, 17, (1, 1, 0), labels.data_ptr(), sizes.data_ptr(), cap,
                                  hist.data_ptr(), ncl.data_ptr(), inside.data_ptr(), hk._stream_handle(None))
        assert rc == (hk.HK_OK if cap >= n else hk.HK_ERR_CAPACITY)
        got = inside.cpu().numpy()
        np.testing.assert_array_equal(got[:cap], want[4][:cap])
        assert (got[cap:] == 7).all()
    lab.close()
