"""FP32 devices with contacts above 64 orbitals (eliminated by a complex128 recursion in the plan's scratch)
against the FP64 plan, with many energies in flight beside few slices, so that the scratch is most of what lies
between the recursion's blocks and the areas behind them."""
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


# halves that are leaves (65, 100, 128) and one that recurses again (140); the last chunk is short
@pytest.mark.parametrize("b,nb,ne,ec", [(65, 2, 24, 24), (100, 4, 12, 12), (128, 2, 20, 16), (140, 3, 12, 12)])
def test_fp32_wide_contacts_equal_fp64(q, b, nb, ne, ec):
    rng = np.random.default_rng(b)
    dev = W.random_device(b, nb, ne, seed=b, scattering=False, eta=1e-2)
    cg = lambda: (rng.standard_normal((b, b)) + 1j * rng.standard_normal((b, b))) / np.sqrt(2 * b)  # noqa: E731
    h = lambda: (lambda x: (x + x.conj().T) / 2)(cg())  # noqa: E731
    dev["leads"] = dict(H00_L=h(), H01_L=0.5 * cg(), H00_R=h(), H01_R=0.5 * cg())
    dev["mu_L"], dev["mu_R"] = 0.1, -0.1
    names = ["GR_diag", "GL_diag", "density", "contact"]
    ref = q.solve_device(dev, "fp64", outputs=names, max_energies_in_flight=ec)
    got = q.solve_device(dev, "fp32", outputs=names, max_energies_in_flight=ec)
    assert not ref["status"].any() and not got["status"].any()
    # per energy; complex64 sweeps: 2^-24 times the slices' conditioning (eta = 1e-2: below 1e3), the contact
    # current as a difference of traces of the density's size
    for e in range(ne):
        for k in ("GR_diag", "GL_diag", "density"):
            assert np.linalg.norm(got[k][e] - ref[k][e]) <= 1e-4 * np.linalg.norm(ref[k][e]), (k, e)
        assert np.abs(got["contact"][e] - ref["contact"][e]).max() <= 1e-4 * np.abs(ref["density"][e]).max() * b, e
