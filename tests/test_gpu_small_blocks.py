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


# the FP64 elimination in clusters of 8, 4, 2 and 1 CTAs (as the batch grows): columns split unevenly, one or two
# rows a lane; every split rounds alike, so a block's inverse does not depend on the batch it is in
@pytest.mark.parametrize("n", [1, 9, 17, 31, 32])
def test_fp64_leaf_inverse_is_the_same_in_every_cluster_size(q, n):
    import torch
    rng = np.random.default_rng(n)
    A = rng.standard_normal((200, n, n)) + 1j * rng.standard_normal((200, n, n))
    dev = torch.tensor(A).cuda()
    full, st = q.zinv_batched(dev.clone(), precision="fp64")
    assert not st.any()
    X = full.cpu().numpy()
    for e in range(0, 200, 40):  # Gauss-Jordan with partial pivoting: a few n eps kappa
        ref = np.linalg.inv(A[e])
        assert np.abs(X[e] - ref).max() <= 16 * n * 2.0**-53 * np.linalg.cond(A[e]) * np.abs(ref).max()
    for batch in (1, 30, 70):
        part, _ = q.zinv_batched(dev[:batch].clone(), precision="fp64")
        assert torch.equal(part, full[:batch])


# launched contacts (blocks above 32): their eliminations over 8 to 1 CTAs, and a device's two contacts together
@pytest.mark.parametrize("n", [33, 50, 64])
def test_launched_contacts_are_the_same_in_every_cluster_size(q, n):
    import torch
    rng = np.random.default_rng(n)
    H00 = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    H00 = torch.tensor((H00 + H00.conj().T) / 4).cuda()
    H01 = torch.tensor((rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))) / 8).cuda()
    E = torch.linspace(-1, 1, 160, dtype=torch.float64).cuda()
    full, st = q.lead_self_energy(H00, H01, E, 1e-2, max_iter=30)
    assert not st.any() and torch.isfinite(torch.view_as_real(full)).all()
    for ne in (1, 12, 40):
        part, _ = q.lead_self_energy(H00, H01, E[:ne].clone(), 1e-2, max_iter=30)
        assert torch.equal(part, full[:ne])


def test_two_launched_contacts_in_uneven_chunks(q):
    dev = _device(40, 2, 5, 0, 1, 0, 0)
    ref = O.solve(dev)
    res = q.solve_device(dev, "fp64", max_energies_in_flight=2)  # chunks of 2, 2 and 1 energies
    for k in ("GR_diag", "GL_diag", "current"):  # 2^-53 times the decimation's conditioning (kappa to 1e4, squared)
        assert np.linalg.norm(res[k] - ref[k]) <= 1e-8 * np.linalg.norm(ref[k]), k
    bad = np.array(dev["energies"])
    bad[1] = np.nan
    r2 = q.solve_device(dev, "fp64", energies=bad, weights=np.ones(5), max_energies_in_flight=2)
    assert r2["status"].tolist() == [0, 4, 0, 0, 0]
    for e in (0, 2, 3, 4):
        assert np.array_equal(r2["GL_diag"][e], res["GL_diag"][e])


def test_fp64_elimination_reciprocal(q):
    """1 x 1 inverses: Smith's quotients, each rounded to nearest, over both orders of the parts, signs, exponents
    inside and outside the range of the FP32-seeded divisions, tiny parts and zeros."""
    import torch
    from fractions import Fraction as F
    rng = np.random.default_rng(3)
    m = rng.uniform(1, 2, (4000, 2)) * rng.choice([-1, 1], (4000, 2))
    ex = np.concatenate([rng.integers(-3, 4, (2000, 2)), rng.integers(-90, 90, (1000, 2)), rng.integers(-480, 480, (1000, 1)) + rng.integers(-70, 70, (1000, 2))])
    z = np.ldexp(m, ex)
    z[:6] = [[1, 0], [0, 1], [3, -0.0], [1, 1], [-1.5, 1.5], [1 + 2.0**-52, 1 - 2.0**-53]]
    got, st = q.zinv_batched(torch.tensor(z[:, 0] + 1j * z[:, 1]).reshape(-1, 1, 1).cuda(), precision="fp64")
    assert not st.any()
    got = got.cpu().numpy().ravel()
    for (re, im), w in zip(z, got):
        tall = abs(re) >= abs(im)
        p, d0 = (im, re) if tall else (re, im)
        r = float(F(p) / F(d0))
        d = float(F(p) * F(r) + F(d0))  # one rounding, as a fused multiply-add
        one, other = float(1 / F(d)), float(F(r) / F(d))
        ref = complex(one, -other) if tall else complex(other, -one)
        if (re, im) == (z[5, 0], z[5, 1]):  # 1/d within 2^-106 of the middle of two numbers: either may come
            assert abs(w.real - ref.real) <= 2.0**-53 and abs(w.imag - ref.imag) <= 2.0**-53
        else:
            assert w == ref, (re, im, w, ref)


# both contacts in one launch (8), and in the same launches one kernel at a time (40)
@pytest.mark.parametrize("b", [8, 40])
def test_of_two_failing_contacts_the_left_code_stands(q, b):
    dev = _device(b, 2, 6, 0, 1, 0, 0)
    dev["energies"] = np.full(6, 0.25)
    z = 0.25 + 1j * dev["eta"]
    sing, slow = (z * np.eye(b), 0.5 * np.eye(b) + 0j), (dev["leads"]["H00_R"], dev["leads"]["H01_R"])
    for left, right, code in ((sing, slow, 4), (slow, sing, 5)):  # z - H00 = 0; one sweep is not enough
        dev["leads"] = dict(H00_L=left[0], H01_L=left[1], H00_R=right[0], H01_R=right[1])
        plan = q.Plan(q.make_desc(2, b, "fp64", 6, has_scattering=False, leads=True, decim_max_iter=1, outputs=["density"]))
        for _ in range(5):
            assert q.solve_device(dev, "fp64", outputs=["density"], plan=plan)["status"].tolist() == [code] * 6
        plan.close()


def test_profile_of_small_blocks(q):
    """One kernel launch a chunk; 6 products a slice (2 of the first), 6 an interface, 7 with G_{i,i+1}; 2 more with
    contacts."""
    b, nb, ne = 7, 4, 5
    for leads, outs, n in ((0, ["GR_diag"], 20 + 18), (1, ["GR_diag", "GR_upper"], 20 + 21 + 2)):
        dev = _device(b, nb, ne, 0, leads, 1 - leads, 0)
        plan = q.Plan(q.make_desc(nb, b, "fp64", 2, has_scattering=not leads, leads=bool(leads), outputs=outs))
        plan.set_profiling(True)
        q.solve_device(dev, "fp64", outputs=outs, plan=plan)
        prof = plan.gemm_profile()
        assert prof["launches"] == 3 and prof["ms"] > 0  # chunks of 2, 2 and 1 energies
        assert prof["useful_flops"] == 8 * b ** 3 * n * ne and prof["pipe_flops"] == 45 * prof["useful_flops"]
        plan.close()


# one value of Sigma^< of one energy infinite: G^< = (g Sigma^<) g^H takes infinities and NaN where the launched path's
# DFMA products do (same order of the sums), and the padded rows and the other energies nothing
@pytest.mark.parametrize("b", [3, 16, 21, 32])
def test_small_blocks_propagate_infinities(q, b):
    dev = _device(b, 1, 3, 0, 0, 1, 1)
    names = ["GR_diag", "GL_diag", "GG_diag", "density"]
    clean = q.solve_device(dev, "fp64", outputs=names)
    dev["SigL"][1, 0, 1, 2] = np.inf
    got = q.solve_device(dev, "fp64", outputs=names)
    ref = q.solve_device(dev, "fp64", outputs=names + ["continuity"])
    parts = lambda x: np.stack([x.real, x.imag])  # noqa: E731
    for k in names:
        x, y = parts(got[k][1]), parts(ref[k][1])
        assert np.array_equal(np.isnan(x), np.isnan(y)) and np.array_equal(x[np.isinf(x)], y[np.isinf(y)]), k
        assert np.array_equal(got[k][[0, 2]], clean[k][[0, 2]])
    assert np.isinf(parts(got["GL_diag"][1])).any()
