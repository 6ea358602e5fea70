"""FP64 batches on the on-chip node transform around the number of frequencies
(2^15) from which the scan applies the phases: one interval above it, the next,
with the longer links only, below.  Every link against the oracle.

Tolerance: 2 intervals x 2 levels x 2 transforms round 8 x 13 times at 1.1e-16,
1.2e-14; the oracle's own phases of up to 1e3 rad carry 1e-13: 1e-11."""
import numpy as np
import pytest

import oracle
from paper_1101_0086_gb300.workloads import FiberMap, Segment, dm_map, wdm_field

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    from paper_1101_0086_gb300 import build as B
    from paper_1101_0086_gb300 import mpa
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    B.build()
    return mpa


@pytest.mark.parametrize("logn,long_links,short_links", [(13, 3, 2), (11, 9, 9)])
def test_fp64_onchip_batch_phases(M, logn, long_links, short_links):
    import torch
    n, nodes = 1 << logn, 21
    T = 100.0 * n / 64
    other = FiberMap((Segment(1.25, 40.0, 0.1, 1.1), Segment(3.75, -15.0, -0.2, 1.4, 0.02)), 0.02, 5.0, 2)
    links, refs = [], []
    for i in range(long_links + short_links):
        fib, z = (dm_map(1) if i % 2 else other), (10.0 if i < long_links else 5.0)
        a = wdm_field(n, T, 2, 50.0, n // 64, 30.0, 2.0, "qpsk", seed=i)
        links.append((fib, T, z, torch.from_numpy(a).cuda()))
        refs.append(oracle.mpa(a, fib, T, 0.0, z, 5.0, nodes, 2))
    assert n * (long_links + short_links) >= 1 << 15 > n * long_links
    start = [k[3].clone() for k in links]
    b = M.Batch(links, 5.0, nodes, 2, precision="fp64")
    b.autotune()
    for k, s in zip(links, start):
        k[3].copy_(s)
    M.profile(True)
    b.propagate(use_graph=False)
    assert b.status_code() == 0
    kinds = {k for k, v in M.profile_read().items() if v[1]}
    M.profile(False)
    assert "kn_mpa" in kinds, "the tuned batch runs on chip"
    for k, r in zip(links, refs):
        assert oracle.rel_l2(k[3].cpu().numpy(), r) < 1e-11
