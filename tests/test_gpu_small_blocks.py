"""FP64 devices of small blocks (one CTA per energy) against the launched sweeps: the same plan with the
continuity output takes the launched path.  Both are FP64, so they agree to rounding times the
conditioning of the slices (the contacts' decimation: kappa up to 1e4 here)."""
import numpy as np
import pytest

import oracle as O
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


def _device(b, nb, ne, S, leads, scattering, per_energy, seed=0):
    rng = np.random.default_rng(seed + 31 * b + nb)
    dev = W.random_device(b, nb, ne, seed=seed, scattering=scattering, eta=1e-4)
    cg = lambda *s: (rng.standard_normal(s) + 1j * rng.standard_normal(s)) / np.sqrt(2 * b)  # noqa: E731
    if S:
        x = 0.05 * cg(nb, b, b)
        dev["S_diag"] = np.eye(b) + x + np.conj(np.swapaxes(x, 1, 2))
        dev["S_upper"] = 0.05 * cg(nb - 1, b, b)
    if per_energy and scattering:
        f = (1.0 + 0.3 * np.arange(ne))[:, None, None, None]
        dev["SigR"], dev["SigL"] = f * dev["SigR"], f * dev["SigL"]
    if leads:
        h = lambda: (lambda x: x + x.conj().T)(cg(b, b))  # noqa: E731
        dev["leads"] = dict(H00_L=h(), H01_L=0.7 * np.eye(b) + 0.2 * cg(b, b), H00_R=h(), H01_R=0.6 * np.eye(b) + 0.2 * cg(b, b))
        dev["mu_L"], dev["mu_R"] = 0.1, -0.1
    return dev


# one block row (1), odd sizes, both paddings and their edges (16, 17, 32); a single slice
SHAPES = [(1, 3, 2), (5, 1, 3), (15, 4, 3), (16, 5, 2), (17, 2, 3), (32, 3, 2)]


@pytest.mark.parametrize("b,nb,ne", SHAPES)
@pytest.mark.parametrize("S,leads,scattering,per_energy", [(0, 1, 0, 0), (0, 0, 1, 0), (1, 1, 1, 1), (1, 0, 1, 0)])
def test_small_blocks_equal_launched_path(q, b, nb, ne, S, leads, scattering, per_energy):
    dev = _device(b, nb, ne, S, leads, scattering, per_energy)
    names = [k for k in q.OUT if k != "continuity"]
    got = q.solve_device(dev, "fp64", outputs=names, max_energies_in_flight=2)
    ref = q.solve_device(dev, "fp64", outputs=list(q.OUT), max_energies_in_flight=2)
    assert (got["status"] == 0).all() and (ref["status"] == 0).all()
    for k, v in ref.items():
        if k in ("status", "continuity") or v.size == 0:
            continue
        scale = np.linalg.norm(v)
        if k.startswith("GG"):  # nearly cancels for occupied states
            scale += np.linalg.norm(ref["GR_diag"])
        if k in ("current", "contact", "current_int", "transmission"):
            scale = max(scale, np.linalg.norm(ref["density"]) * 1e-2)  # a difference of traces of that size
        assert np.linalg.norm(got[k] - v) <= 2e-10 * max(scale, 1e-30), (k, np.linalg.norm(got[k] - v) / scale)


def test_small_blocks_against_oracle_and_singular_energy(q):
    dev = _device(12, 4, 3, 1, 0, 1, 0)
    ref = O.solve(dev)
    E = np.array(dev["energies"])
    res = q.solve_device(dev, "fp64")
    for k in ("GR_diag", "GR_upper", "GR_lower", "GL_diag", "GL_upper", "GG_diag", "GG_upper", "current", "density"):
        assert np.linalg.norm(res[k] - ref[k]) <= 1e-10 * np.linalg.norm(ref[k]), k
    bad = E.copy()
    bad[1] = np.nan
    r2 = q.solve_device(dev, "fp64", energies=bad, weights=np.ones(3))
    assert r2["status"].tolist() == [0, 4, 0]
    for e in (0, 2):
        assert np.array_equal(r2["GL_diag"][e], res["GL_diag"][e])


def test_decimation_of_ill_conditioned_leads(q):
    """Leads at a band edge (kappa far beyond FP32's reach: the eliminated inverses) and a zero coupling."""
    import torch
    n = 9
    H00 = np.diag(np.full(n - 1, -1.0), 1) + np.diag(np.full(n - 1, -1.0), -1) + 0j
    H01 = -np.eye(n) + 0j
    E = np.array([2.0 * np.cos(np.pi / (n + 1)) + 2.0 - 1e-9, 0.3, 1.1])
    got, st = q.lead_self_energy(torch.tensor(H00).cuda(), torch.tensor(H01).cuda(), torch.tensor(E).cuda(), 1e-9)
    assert (st.cpu().numpy() == 0).all()
    # closed form per mode: (z' - sqrt(z' - 2) sqrt(z' + 2)) / 2
    ev, U = np.linalg.eigh(H00)
    for e in range(3):
        z = E[e] + 1e-9j - ev
        ref = (U * ((z - np.sqrt(z - 2) * np.sqrt(z + 2)) / 2)) @ U.conj().T
        assert np.linalg.norm(got[e].cpu().numpy() - ref) / np.linalg.norm(ref) < (1e-4 if e == 0 else 1e-9)
    zero, st = q.lead_self_energy(torch.tensor(H00).cuda(), torch.zeros_like(torch.tensor(H01)).cuda(),
                                  torch.tensor(E[1:]).cuda(), 1e-6)
    assert (st.cpu().numpy() == 0).all() and (zero == 0).all()
