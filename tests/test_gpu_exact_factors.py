"""FP32 split steps on the fine and medium tiles, whose radix-4
to radix-16 passes apply more factors than radix-32 ones, against FP64 runs
of the same library on the same samples.

Tolerances: 40 steps are 80 transforms.  Data roundings average out: about
sqrt(80) x sqrt(2 x 20) x 0.5 x 6e-8 = 1.7e-6.  Errors of the factors recur at
every step and add up: with factors good to half a unit in the last place
(0.25 x 6e-8 rms) and one product in half of them, two factors and a four-step
product of three roundings an element and transform, about 80 x 1e-7 = 8e-6,
less where they cancel: 1.1e-5 together at 2^18 and 2^20 samples (factors that
are products of two table entries each give 1.3e-5 and 1.5e-5).  At 2^10, 32
points each way: one factor of each, direct from the table: 80 x 3.5e-8 =
2.8e-6 and 0.9e-6 of the data, 3.7e-6 (4.3e-6 with products)."""
import numpy as np
import pytest

from paper_1101_0086_gb300.workloads import dm_map, wdm_field

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    from paper_1101_0086_gb300 import build as B
    from paper_1101_0086_gb300 import mpa
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    B.build()
    return mpa


def _rel(a, b):
    return float(np.linalg.norm(a.astype(np.complex128) - b) / np.linalg.norm(b))


@pytest.mark.parametrize("logn,tol", [(10, 3.7e-6), (18, 1.1e-5), (20, 1.1e-5)])
def test_split_step_factors(M, logn, tol):
    import torch
    n, spp = 1 << logn, 128
    T = 100.0 * n / spp
    errors = []
    for seed in range(3):
        a = torch.from_numpy(wdm_field(n, T, 4, 50.0, n // spp, 30.0, 2.0, "qpsk", seed=seed)).cuda()
        x = M.ss_propagate(a.to(torch.complex64), dm_map(1), T, 0.05, 44.0, 46.0)
        y = M.ss_propagate(a, dm_map(1), T, 0.05, 44.0, 46.0)
        errors.append(_rel(x.cpu().numpy(), y.cpu().numpy()))
    assert np.mean(errors) < tol
