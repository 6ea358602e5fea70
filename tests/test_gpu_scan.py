"""The trapezoid scan of Eq. (6) on the GPU at node counts around the edges of
its runs and panels (8 warps x up to 16 nodes in FP32, 8 in FP64), one and
several links, against the oracle.

Tolerances: two intervals x n_iter levels x two transforms, each rounding
about log2 N times at 2^-24 relative; with the largest case (3 levels,
N = 2^11) 2 x 3 x 2 x 11 x 6e-8 = 8e-6 for FP32, and the same count at 2^-53,
1.5e-14, for FP64, where the oracle's own phases of up to 1e3 rad carry
1e-13: 1e-11."""
import numpy as np
import pytest

import oracle
from paper_1101_0086_gb300.workloads import dm_map, wdm_field

pytestmark = pytest.mark.gpu
TOL = {"fp32": 8e-6, "fp64": 1e-11}


@pytest.fixture(scope="module")
def M():
    import torch
    from paper_1101_0086_gb300 import build as B
    from paper_1101_0086_gb300 import mpa
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    B.build()
    return mpa


def _case(M, n, prec, nodes, n_iter):
    import torch
    fib = dm_map(1)
    T = 100.0 * n / 64
    a = wdm_field(n, T, 2, 50.0, n // 64, 30.0, 2.0, "qpsk", seed=nodes)
    f = torch.from_numpy(a).to(torch.complex64 if prec == "fp32" else torch.complex128).cuda()
    ref = oracle.mpa(f.cpu().numpy().astype(np.complex128), fib, T, 40.0, 50.0, 5.0, nodes, n_iter)
    return fib, T, f, ref


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("n,nodes,n_iter", [(256, 1, 1), (256, 2, 2), (256, 7, 3), (256, 8, 2), (256, 9, 2),
                                            (512, 64, 2), (512, 65, 2), (256, 127, 3), (256, 128, 2), (256, 129, 2),
                                            (2048, 143, 3), (256, 257, 2)])
def test_scan_node_runs(M, prec, n, nodes, n_iter):
    fib, T, f, ref = _case(M, n, prec, nodes, n_iter)
    plan = M.Plan(fib, n, T, 5.0, nodes, n_iter, precision=prec)
    plan.propagate(f, 40.0, 50.0)
    assert plan.status_code() == 0
    assert oracle.rel_l2(f.cpu().numpy().astype(np.complex128), ref) < TOL[prec]


@pytest.mark.parametrize("nodes", [9, 130])
def test_scan_of_several_links(M, nodes):
    import torch
    fib, T = dm_map(2), 800.0
    fields = [wdm_field(512, T, 2, 50.0, 8, 30.0, 2.0, "qpsk", seed=s) for s in range(3)]
    bufs = [torch.from_numpy(a).to(torch.complex64).cuda() for a in fields]
    refs = [oracle.mpa(b.cpu().numpy().astype(np.complex128), fib, T, 0.0, z, 5.0, nodes, 2)
            for b, z in zip(bufs, (10.0, 5.0, 10.0))]
    b = M.Batch([(fib, T, z, x) for x, z in zip(bufs, (10.0, 5.0, 10.0))], 5.0, nodes, 2)
    b.set_persistent(False)
    b.propagate(use_graph=False)
    assert b.status_code() == 0
    for x, r in zip(bufs, refs):
        assert oracle.rel_l2(x.cpu().numpy().astype(np.complex128), r) < TOL["fp32"]
