"""Transforms around a propagation beyond 2^22 samples, where the field is
transposed around a row pass: they run at the plan's split, as its levels do.
Without the Kerr term only these transforms depend on the split."""
import numpy as np
import pytest

from paper_1101_0086_gb300.workloads import FiberMap, Segment, random_field

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    from paper_1101_0086_gb300 import build as B
    from paper_1101_0086_gb300 import mpa
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    B.build()
    return mpa


def test_transforms_beyond_two_to_22_follow_the_plan(M):
    """Splits 2^10 and 2^11 round in another order (a linear link of 2^23
    samples); both are within the 46 roundings of a transform pair at 6e-8,
    3e-6, of FP64."""
    import torch
    n = 1 << 23
    fib, T = FiberMap((Segment(5.0, -21.7, 0.1, 0.0),), 0.0, 5.0, 1), 100.0 * n / 1024
    a = torch.from_numpy(random_field(n, 3)).cuda()
    p64 = M.Plan(fib, n, T, 5.0, 1, 1, precision="fp64")
    ref = p64.propagate(a.clone(), 0.0, 5.0).cpu().numpy()
    plan = M.Plan(fib, n, T, 5.0, 1, 1)
    out = {}
    for split in (10, 11):
        plan.set_split(split)
        out[split] = plan.propagate(a.to(torch.complex64), 0.0, 5.0).cpu().numpy()
        assert np.linalg.norm(out[split] - ref) / np.linalg.norm(ref) < 3e-6
    assert not np.array_equal(out[10], out[11])
