"""The shapes on either side of the rule that picks one CTA for a lattice (at most 128 rows of at
most 12 sites, or one row of at most 2048) against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1405_1931_gb300 import fields, hk

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def check(lab, phi, per, what):
    want = oracle.label(phi, per)
    labels, sizes, hist, ncl = lab.label(torch.from_numpy(phi).cuda(), per)
    lab.sync_status()
    assert int(ncl.item()) == want[3], what
    np.testing.assert_array_equal(labels.cpu().numpy(), want[0], err_msg=what)
    np.testing.assert_array_equal(sizes[:want[3]].cpu().numpy(), want[1], err_msg=what)
    np.testing.assert_array_equal(hist.cpu().numpy(), want[2], err_msg=what)


@pytest.mark.parametrize("shape", [(12, 8, 16), (13, 8, 16), (12, 129, 1), (12, 1, 128), (1, 1, 129), (2048, 1, 1), (2049, 1, 1),
                                   (8, 2, 65)])
def test_either_side_of_the_one_cta_rule(shape):
    lab = hk.Labeller(0)
    for p in (0.3, 0.7, 1.0):
        check(lab, fields.iid_field(*shape, seed=1, occupancy=p), (1, 1, 1), f"{shape} {p}")
    lab.close()
