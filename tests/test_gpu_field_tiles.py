"""Transforms and split-steps of single fields on their fine and medium tiles,
and FP64 node transforms, with full twiddle tables
(lengths up to 2048, phases from the table from 256 on) at every length of
rows and columns, against the oracle.

Tolerances: a transform rounds about log2 N <= 20 times at 1.1e-16, twice a
step: 8 steps 3.5e-14, a few times that for the partial sums' growth: 2e-13.
The oracle's phases of up to 5e3 rad carry 6e-13 at the band edge, far from
the field's band: 1e-12 with the linear steps."""
import numpy as np
import pytest

import oracle
from paper_1101_0086_gb300.workloads import dm_map, random_field, wdm_field

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    from paper_1101_0086_gb300 import build as B
    from paper_1101_0086_gb300 import mpa
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    B.build()
    return mpa


@pytest.mark.parametrize("logn", [8, 9, 11, 13, 15, 17, 18, 20, 21])
def test_fp64_transform_pair(M, logn):
    import torch
    a = random_field(1 << logn, logn)
    d = torch.from_numpy(a).cuda()
    M.fft(d, +1)
    assert oracle.rel_l2(d.cpu().numpy(), oracle.fft(a, +1)) < 2e-13
    M.fft(d, -1)
    assert oracle.rel_l2(d.cpu().numpy(), a) < 2e-13


@pytest.mark.parametrize("logn", [9, 12, 14, 16, 18, 20])
def test_fp64_split_step(M, logn):
    import torch
    n, spp = 1 << logn, 64 if logn < 14 else 128
    T = 100.0 * n / spp
    a = wdm_field(n, T, 4, 50.0, n // spp, 30.0, 2.0, "qpsk", seed=logn)
    d = torch.from_numpy(a).cuda()
    M.ss_propagate(d, dm_map(1), T, 0.05, 44.8, 45.2)
    assert oracle.rel_l2(d.cpu().numpy(), oracle.ss(a, dm_map(1), T, 44.8, 45.2, 0.05)) < 1e-12


@pytest.mark.parametrize("logn,split", [(12, 0), (13, 0), (12, 4), (14, 5), (14, 9), (16, 8), (18, 7), (18, 11)])
def test_fp64_interval(M, logn, split):
    import torch
    n = 1 << logn
    T = 100.0 * n / 128
    a = wdm_field(n, T, 4, 50.0, n // 128, 30.0, 2.0, "qpsk", seed=logn)
    plan = M.Plan(dm_map(1), n, T, 5.0, 6, 2, precision="fp64")
    plan.set_split(split)
    d = torch.from_numpy(a).cuda()
    plan.propagate(d, 45.0, 50.0)
    assert plan.status_code() == 0
    assert oracle.rel_l2(d.cpu().numpy(), oracle.mpa(a, dm_map(1), T, 45.0, 50.0, 5.0, 6, 2)) < 1e-12


@pytest.mark.parametrize("logn", [8, 10, 13, 16, 18, 19, 20, 22, 23])
def test_fp32_transform_pair(M, logn):
    """Fine and medium tiles in FP32: 22 roundings at 6e-8 and their partial
    sums' growth, 4e-6."""
    import torch
    a = random_field(1 << logn, logn).astype(np.complex64)
    d = torch.from_numpy(a).cuda()
    M.fft(d, +1)
    assert oracle.rel_l2(d.cpu().numpy(), oracle.fft(a.astype(np.complex128), +1)) < 4e-6
    M.fft(d, -1)
    assert oracle.rel_l2(d.cpu().numpy(), a) < 4e-6


@pytest.mark.parametrize("logn", [9, 14, 18, 19, 21])
def test_fp32_split_step(M, logn):
    """Eight steps of two transforms: 16 x 22 roundings at 6e-8, 2e-5."""
    import torch
    n, spp = 1 << logn, 64 if logn < 14 else 128
    T = 100.0 * n / spp
    a = wdm_field(n, T, 4, 50.0, n // spp, 30.0, 2.0, "qpsk", seed=logn).astype(np.complex64)
    d = torch.from_numpy(a).cuda()
    M.ss_propagate(d, dm_map(1), T, 0.05, 44.8, 45.2)
    ref = oracle.ss(a.astype(np.complex128), dm_map(1), T, 44.8, 45.2, 0.05)
    assert oracle.rel_l2(d.cpu().numpy(), ref) < 2e-5


@pytest.mark.parametrize("what", ["ss", "link14", "link18"])
def test_captured_passes_replay(M, what):
    """Kernels that start early (launch_pdl) under stream capture: a replay
    gives the direct call's result, bit for bit."""
    import torch
    logn = {"ss": 13, "link14": 14, "link18": 18}[what]
    n = 1 << logn
    T = 100.0 * n / 128
    a = torch.from_numpy(wdm_field(n, T, 4, 50.0, n // 128, 30.0, 2.0, "qpsk", seed=1)).to(torch.complex64).cuda()
    ws = torch.empty(M.ss_workspace_bytes(n, "fp32"), dtype=torch.uint8, device="cuda")
    plan = M.Plan(dm_map(1), n, T, 5.0, 12, 2)

    def run(x):
        if what == "ss":
            M.ss_propagate(x, dm_map(1), T, 0.05, 44.8, 45.2, workspace=ws)
        else:
            plan.propagate(x, 40.0, 50.0)

    want = a.clone()
    run(want)
    x = a.clone()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        run(x)
    for _ in range(2):
        x.copy_(a)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(torch.view_as_real(x), torch.view_as_real(want))
