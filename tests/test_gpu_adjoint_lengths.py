"""FP32 gradients at the column lengths of the reverse passes that other sizes
do not reach.  The recompute and reverse passes take columns of 2^8 points up
to 2^20 samples (rows of 2^10 at 2^18, 2^11 at 2^19) and of 2^(log2 N - 12)
beyond: 512 at 2^21, 1024 at 2^22, 2048 at 2^23 (the last two on tiles of 16
elements a thread).  Element by element against the oracle adjoint, on one
interval across the segment boundary at 45 km.

Tolerances as for every FP32 gradient: 1e-4 for the field, 1e-3 for each
parameter gradient relative to the largest."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_1101_0086_gb300.workloads import FiberMap, dm_map, wdm_field

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    from paper_1101_0086_gb300 import build as B
    from paper_1101_0086_gb300 import mpa
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    B.build()
    return mpa


@pytest.mark.parametrize("logn,nodes,n_iter", [(18, 4, 2), (19, 4, 2), (21, 2, 2), (22, 2, 2), (23, 2, 1)])
def test_fp32_adjoint_column_lengths(M, logn, nodes, n_iter):
    import torch
    n = 1 << logn
    T = 100.0 * n / 1024
    fib = dm_map(1)
    a = wdm_field(n, T, 16, 50.0, n // 1024, 30.0, 2.0, "qpsk", seed=logn)
    z0, z1, L = 44.5, 45.5, 0.5
    linear = FiberMap(tuple(dataclasses.replace(s, sigma_per_W_km=0.0) for s in fib.segments), fib.gamma_per_km,
                      fib.z_a_km, fib.n_periods)
    # the gradient of |out - target|^2, the target close to the dispersed input
    target = 0.8 * np.exp(0.3j) * oracle.ss(a, linear, T, z0, z1, z1 - z0)
    g_out = 2 * (oracle.mpa(a, fib, T, z0, z1, L, nodes, n_iter) - target)
    ref = oracle.mpa_adjoint(a, g_out, fib, T, z0, z1, L, nodes, n_iter)
    plan = M.Plan(fib, n, T, L, nodes, n_iter)

    def dev(x):
        return torch.from_numpy(x.astype(np.complex64)).cuda()

    gi, gs, gb = plan.adjoint(dev(g_out), z0, z1, field_in=dev(a))
    assert oracle.rel_l2(gi.cpu().numpy().astype(np.complex128), ref.field) < 1e-4
    for got, want in ((gs, ref.sigma), (gb, ref.beta2)):
        assert np.count_nonzero(want) == 2
        assert np.max(np.abs(got - want)) < 1e-3 * np.max(np.abs(want))
