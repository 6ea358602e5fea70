"""Levels whose node spectra exceed L2 on columns below 2^8 points, where the
forward column pass prefetches its tiles, the last ones ragged (143 and 144
nodes), against an FP64 plan.

Tolerance: 2 levels x 2 transforms and the entry and exit, each rounding about
log2 N = 17 times at 6e-8, 6e-6."""
import numpy as np
import pytest

from paper_1101_0086_gb300.workloads import dm_map, wdm_field

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split,nodes", [(4, 142), (7, 142), (7, 143)])
def test_level_beyond_l2_on_short_columns(split, nodes):
    import torch
    from paper_1101_0086_gb300 import build as B
    from paper_1101_0086_gb300 import mpa
    B.build()
    n = 1 << 17
    T = 100.0 * n / 128
    a = torch.from_numpy(wdm_field(n, T, 4, 50.0, n // 128, 30.0, 2.0, "qpsk", seed=split)).cuda()
    plan = mpa.Plan(dm_map(1), n, T, 5.0, nodes, 2)
    plan.set_split(split)
    x = plan.propagate(a.to(torch.complex64), 45.0, 50.0)
    y = mpa.Plan(dm_map(1), n, T, 5.0, nodes, 2, precision="fp64").propagate(a, 45.0, 50.0)
    assert plan.status_code() == 0
    x, y = x.cpu().numpy().astype(np.complex128), y.cpu().numpy()
    assert np.linalg.norm(x - y) < 6e-6 * np.linalg.norm(y)
