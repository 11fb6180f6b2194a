"""The bond current of an emulated-FP64 solve with an overlap matrix is reduced in FP64: against the sum, in
extended precision, over the returned G^<_{i,i+1} blocks themselves."""
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


# b = 3: 18 products, so that their rounding does not average out (H - E S rounded to a df32 pair, about 2^-49 of a
# term, would be 2^-51 of the terms' absolute sum); 33: tiles in pairs, with remainders
@pytest.mark.parametrize("b,bar", [(3, 2.0 ** -53), (33, 2.0 ** -56)])
def test_emulated_current_with_overlap_is_reduced_in_fp64(q, b, bar):
    nb, ne = 3, 64
    dev = W.random_device(b, nb, ne, seed=b, eta=1e-3)
    rng = np.random.default_rng(b)
    cg = lambda *s: (rng.standard_normal(s) + 1j * rng.standard_normal(s)) / np.sqrt(2 * b)  # noqa: E731
    x = 0.05 * cg(nb, b, b)
    dev["S_diag"] = np.eye(b) + x + np.conj(np.swapaxes(x, 1, 2))
    dev["S_upper"] = 0.05 * cg(nb - 1, b, b)
    res = q.solve_device(dev, "emu64", outputs=["GL_upper", "current"])
    E = np.array(dev["energies"])[:, None, None, None]
    h = dev["H_upper"][None].astype(np.clongdouble) - E * dev["S_upper"][None]
    u = res["GL_upper"].astype(np.clongdouble)
    terms = np.concatenate([(h.real * u.real).reshape(ne, nb - 1, -1), (h.imag * u.imag).reshape(ne, nb - 1, -1)], 2)
    err = np.abs(res["current"] + 2 * terms.sum(2)) / (2 * np.abs(terms).sum(2))
    # a rounding's root mean square is 2^-54.8 of its value: with b = 3 that of a term's difference and product and of
    # a few partial sums below the terms' absolute sum add up to less than 2^-53; with 33, 2178 terms average out
    assert np.sqrt((err ** 2).mean()) <= bar, np.log2(np.sqrt((err ** 2).mean()))
