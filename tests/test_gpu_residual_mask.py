"""The norm that decides whether an energy takes another Newton sweep is the same number in every batch: its residual
is summed by clusters of 8, 4, 2 or 1 CTAs as the batch grows, always over the same slices in the same order."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_2606_25595_gb300 import build
    build.build()
    import paper_2606_25595_gb300 as q
    q.load()
    return q


@pytest.mark.parametrize("b", [45, 128, 200])  # 2025 values: one CTA, one round; 16384: any cluster; the last slices short
def test_sweep_decision_does_not_depend_on_the_batch(q, b):
    dev = W.random_device(b, 1, 1, seed=b, eta=1e-3)

    def solve(ne, tol2):
        plan = q.Plan(q.make_desc(1, b, "emu64", ne, 2, has_scattering=True, outputs=["GR_diag"], refine_tol=float(np.sqrt(np.float64(tol2)))))
        res = q.solve_device(dev, "emu64", energies=np.full(ne, 0.3), outputs=["GR_diag"], plan=plan)["GR_diag"]
        plan.close()
        return res

    once, twice = solve(1, 1.0)[0], solve(1, 2.0 ** -120)[0]
    assert not np.array_equal(once, twice)
    # the squared norm itself, by bisection over the float32 tolerances: the least one that stops after one sweep
    lo, hi = np.float32(2.0 ** -120).view(np.int32).item(), np.float32(1.0).view(np.int32).item()
    while hi - lo > 1:
        mid = (lo + hi) // 2
        if np.array_equal(solve(1, np.int32(mid).view(np.float32))[0], once):
            hi = mid
        else:
            lo = mid
    for ne in (30, 60, 200):  # clusters of 4, 2 and 1
        for bits, want in ((hi, once), (lo, twice)):
            got = solve(ne, np.int32(bits).view(np.float32))
            assert all(np.array_equal(g, want) for g in got), (ne, bits - hi)
