"""The trapezoid scan of Eq. (6) on the GPU at node counts around the edges of
its runs and panels (8 warps x up to 16 nodes in FP32, 8 in FP64), one and
several links, and the form that applies the phases itself (from 2^14
frequencies in FP32, 2^15 in FP64), on maps whose segments change at the
first node, at the last, between nodes and around its blocks of 128 nodes,
against the oracle.

Tolerances: two intervals x n_iter levels x two transforms, each rounding
about log2 N times at 2^-24 relative; with the largest cases (3 levels,
N = 2^11; 2 levels, N = 2^14) 2 x 3 x 2 x 11 x 6e-8 = 8e-6 for FP32, and the
same count at 2^-53, 1.5e-14, for FP64, where the oracle's own phases of up
to 1e3 rad carry 1e-13: 1e-11."""
import numpy as np
import pytest

import oracle
from paper_1101_0086_gb300.workloads import FiberMap, Segment, dm_map, wdm_field

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


def _uneven_map():
    # 5-km periods: a short first piece (inside the first step of coarse grids),
    # pieces that end on and between nodes, a short last piece, one gain piece
    segs = (Segment(0.01, -21.7, 0.1, 1.3), Segment(1.25, 40.0, 0.1, 1.1), Segment(1.24, 40.0, -0.2, 1.1, 0.02),
            Segment(2.49, -15.0, 0.1, 1.4), Segment(0.01, 190.0, 0.0, 1.2))
    return FiberMap(segs, 0.02, 5.0, 2)


def _propagate_against_oracle(M, n, prec, fib, nodes, n_iter, split):
    import torch
    T = 100.0 * n / 128
    a = wdm_field(n, T, 4, 50.0, n // 128, 30.0, 2.0, "qpsk", seed=nodes)
    f = torch.from_numpy(a).to(torch.complex64 if prec == "fp32" else torch.complex128).cuda()
    ref = oracle.mpa(f.cpu().numpy().astype(np.complex128), fib, T, 0.0, 10.0, 5.0, nodes, n_iter)
    plan = M.Plan(fib, n, T, 5.0, nodes, n_iter, precision=prec)
    plan.set_split(split)
    plan.propagate(f, 0.0, 10.0)
    assert plan.status_code() == 0
    assert oracle.rel_l2(f.cpu().numpy().astype(np.complex128), ref) < TOL[prec]


@pytest.mark.parametrize("split", [0, 7])
@pytest.mark.parametrize("nodes", [1, 2, 4, 127, 128, 129, 257])
def test_scan_with_phases(M, nodes, split):
    _propagate_against_oracle(M, 1 << 14, "fp32", _uneven_map(), nodes, 2, split)


@pytest.mark.parametrize("logn,split", [(15, 0), (16, 8), (17, 8)])
def test_scan_with_phases_cluster_and_tile_layout(M, logn, split):
    _propagate_against_oracle(M, 1 << logn, "fp32", _uneven_map(), 20, 2, split)


@pytest.mark.parametrize("nodes", [1, 8, 19])
def test_scan_with_phases_fp64(M, nodes):
    _propagate_against_oracle(M, 1 << 15, "fp64", _uneven_map(), nodes, 2, 7)


def test_scan_with_phases_of_links_with_different_maps(M):
    import torch
    n, T, nodes = 1 << 13, 6400.0, 40
    maps = [_uneven_map(), dm_map(1), _uneven_map()]
    bufs = [torch.from_numpy(wdm_field(n, T, 4, 50.0, 64, 30.0, 2.0, "qpsk", seed=s)).to(torch.complex64).cuda()
            for s in range(3)]
    refs = [oracle.mpa(b.cpu().numpy().astype(np.complex128), m, T, 0.0, 10.0, 5.0, nodes, 2)
            for b, m in zip(bufs, maps)]
    b = M.Batch([(m, T, 10.0, x) for m, x in zip(maps, bufs)], 5.0, nodes, 2)
    b.set_persistent(False)
    b.propagate(use_graph=False)
    assert b.status_code() == 0
    for x, r in zip(bufs, refs):
        assert oracle.rel_l2(x.cpu().numpy().astype(np.complex128), r) < TOL["fp32"]


@pytest.mark.parametrize("logn,nodes", [(8, 3), (9, 1), (10, 142), (11, 7), (11, 1300), (12, 5), (12, 620)])
def test_onchip_tiles_of_few_and_many_nodes(M, logn, nodes):
    """On-chip node transforms on their fine tiles (fewer than 304 large tiles
    of nodes) and on the large ones, the last tile partly filled."""
    _propagate_against_oracle(M, 1 << logn, "fp32", dm_map(1), nodes, 2, 0)
