"""Products of a slice's stage that share a launch against the same products launched one by one (a plan with
GEMM profiling on): which launch computes a tile does not change how it is computed, so every output is equal bit
for bit.  The shapes cover the last column tile's widths, one and two row tiles, and sizes below the tensor cores'."""
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


@pytest.mark.parametrize("prec,b,bits", [("emu64", 24, 0), ("emu64", 97, 0), ("emu64", 130, 0), ("emu64", 49, 40),
                                         ("fp32", 96, 0), ("fp32", 129, 0), ("bf16x3", 65, 0), ("fp64", 33, 0),
                                         ("fp64", 130, 0)])
@pytest.mark.parametrize("bt", [False, True])
def test_grouped_products_equal_single_launches(q, prec, b, bits, bt):
    dev = W.random_device(b, 4, 3, seed=b, scattering=True, offdiag_sigma=bt, eta=1e-3)
    names = [k for k in q.OUT if k not in ("continuity", "contact", "transmission")]
    desc = q.make_desc(4, b, prec, 2, 2, has_scattering=True, energy_dependent_sigma=dev["SigR"].shape[0] > 1,
                       outputs=names, offdiag_sigma=bt, storage_bits=bits)
    got = []
    for profiling in (False, True):
        plan = q.Plan(desc)
        plan.set_profiling(profiling)
        n0 = q.load().qtx_kernel_launches()
        got.append(q.solve_device(dev, prec, outputs=names, max_energies_in_flight=2, plan=plan, storage_bits=bits))
        got[-1]["launches"] = q.load().qtx_kernel_launches() - n0
    one, many = got[1], got[0]
    assert (many["status"] == 0).all()
    for k, v in one.items():
        if k != "launches":
            assert np.array_equal(v, many[k]), k
    assert many["launches"] <= one["launches"]
