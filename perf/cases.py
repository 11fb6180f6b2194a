"""Measured cases: the work a user of this library has it do, through its public entry points.

* ``strip``    ballistic strip between two contacts (the strip workload's recipe): FP64, every output.
* ``lead``     contact self-energies alone (``lead_self_energy``).
* ``device``   one solve of a dense random block-tridiagonal device on a kept plan, in each precision,
               with the options used in earnest (block-tridiagonal per-energy self-energies, FPX storage
               between the sweeps, overlap matrices with contacts wider than one CTA's decimation).
* ``uneven``   several devices of different block sizes in one group solve.
* ``wsystem``  the screened-Coulomb system: assembly and solve.
* ``zgemm``, ``zinv``  the sweep's products and block inverses on their own.
* ``fpx``      the storage codec, encode and decode.

Sizes follow the repository's workloads (b = 16 strips of 32 slices and 64 energies, b = 64 ... 512
devices), its tests' odd sizes, and energy counts a card holds beside its other work.
"""
import math

import numpy as np
import torch

import paper_2606_25595_gb300 as q

ETA = 1e-6
BLOCKS = ("GR_diag", "GR_upper", "GR_lower", "GL_diag", "GL_upper", "GG_diag", "GG_upper")


# ------------------------------------------------------------------------------------------ cases
def listed():
    return [
        # the smallest solve in use (the smoke test's strip): launches and latency are all of it
        dict(name="strip_4e", kind="strip", b=16, nb=8, ne=4, prec="fp64"),
        # the strip workload as configured: 64 energies, contacts at both ends, every output
        dict(name="strip_64e", kind="strip", b=16, nb=32, ne=64, prec="fp64"),
        # a wide strip with an overlap matrix: contacts beyond 32 orbitals, S at every block
        dict(name="contacts_b48", kind="device", b=48, nb=6, ne=12, prec="fp64", out="obs", S=True, leads=True),
        # the plain FP64 path on a dense device, a few energies (reference runs, hard energies)
        dict(name="fp64_b128", kind="device", b=128, nb=12, ne=8, prec="fp64", out="diag"),
        # complex64 solve of one of the uneven batch's wide devices
        dict(name="fp32_b384", kind="device", b=384, nb=8, ne=32, prec="fp32", out="diag"),
        # the benchmark's mode and block size, with fewer slices and energies in flight
        dict(name="emu64_b256", kind="device", b=256, nb=16, ne=96, prec="emu64", out="diag", tol=2.0 ** -12),
        # a scGW iteration's solve: block-tridiagonal per-energy self-energies, every block returned,
        # a block size that fills no tile
        dict(name="bt_emu64_b120", kind="device", b=120, nb=10, ne=24, prec="emu64", out="all", bt=True),
        # more energies per GB: left-connected blocks in 40-bit storage between the sweeps
        dict(name="fpx40_b192", kind="device", b=192, nb=16, ne=32, prec="emu64", out="diag", tol=2.0 ** -12, bits=40),
        # uneven batch: devices of different block sizes solved together
        dict(name="uneven_fp32", kind="uneven", bs="64,96,128,256", nbs="12,9,8,6", ne=24, prec="fp32"),
        # screened-Coulomb system, W^R, W^< and W^> per energy
        dict(name="wsystem_b96", kind="wsystem", b=96, nb=6, ne=16, prec="emu64"),
        # the product on its own at ragged sizes, right operand conjugate-transposed, C0 added
        dict(name="zgemm_emu64", kind="zgemm", m=250, n=256, k=300, batch=32, prec="emu64", opa="N", opb="C", beta=True),
        # the codec on one large array of blocks
        dict(name="fpx_24", kind="fpx", bits=24, count=60_000_004),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["strip", "lead", "fp64", "contacts", "fp32", "emu64", "emu64", "bt", "fpxstore", "uneven",
                       "wsystem", "zgemm", "zinv", "fpx"])
    if kind == "strip":
        return dict(kind="strip", b=rng.randint(5, 32), nb=_log(rng, 3, 40), ne=_log(rng, 2, 96), prec="fp64")
    if kind == "lead":
        return dict(kind="lead", b=_log(rng, 8, 80), ne=_log(rng, 4, 48))
    if kind == "contacts":
        return dict(kind="device", b=rng.randint(33, 72), nb=rng.randint(3, 9), ne=_log(rng, 3, 20), prec="fp64",
                    out="obs", S=rng.random() < 0.5, leads=True)
    if kind == "fp64":
        b = _log(rng, 24, 160)
        return dict(kind="device", b=b, nb=_log(rng, 4, 20), ne=_log(rng, 2, 24), prec="fp64",
                    out=rng.choice(["diag", "all"]))
    if kind == "fp32":
        return dict(kind="device", b=_log(rng, 64, 400), nb=_log(rng, 4, 16), ne=_log(rng, 4, 40), prec="fp32",
                    out=rng.choice(["diag", "all"]))
    if kind == "emu64":
        return dict(kind="device", b=_log(rng, 64, 288), nb=_log(rng, 4, 16), ne=_log(rng, 4, 80), prec="emu64",
                    out=rng.choice(["diag", "diag", "all"]), tol=2.0 ** -12)
    if kind == "bt":
        return dict(kind="device", b=_log(rng, 48, 200), nb=rng.randint(3, 12), ne=_log(rng, 4, 24), prec="emu64",
                    out="all", bt=True)
    if kind == "fpxstore":
        return dict(kind="device", b=_log(rng, 64, 256), nb=rng.randint(4, 16), ne=_log(rng, 4, 40), prec="emu64",
                    out="diag", tol=2.0 ** -12, bits=rng.choice([40, 48, 56]))
    if kind == "uneven":
        n = rng.randint(2, 4)
        return dict(kind="uneven", bs=",".join(str(_log(rng, 64, 256)) for _ in range(n)),
                    nbs=",".join(str(rng.randint(4, 12)) for _ in range(n)), ne=_log(rng, 4, 32),
                    prec=rng.choice(["fp32", "emu64"]))
    if kind == "wsystem":
        return dict(kind="wsystem", b=_log(rng, 48, 128), nb=rng.randint(2, 6), ne=_log(rng, 4, 16), prec="emu64")
    if kind == "zgemm":
        return dict(kind="zgemm", m=_log(rng, 32, 320), n=_log(rng, 32, 320), k=_log(rng, 32, 320),
                    batch=_log(rng, 2, 48), prec=rng.choice(["emu64", "emu64", "fp64", "fp32", "bf16x3"]),
                    opa=rng.choice("NC"), opb=rng.choice("NC"), beta=rng.random() < 0.5)
    if kind == "zinv":
        return dict(kind="zinv", b=_log(rng, 16, 256), batch=_log(rng, 4, 64),
                    prec=rng.choice(["emu64", "fp64", "fp32"]))
    return dict(kind="fpx", bits=rng.choice([56, 48, 40, 32, 24, 16]), count=2 * _log(rng, 50_000, 30_000_000) + rng.randint(0, 1))


# ----------------------------------------------------------------------------------------- inputs
class _Draw:
    """Seeded complex Gaussians on the GPU."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(int(seed) * 7919 + 17)

    def real(self, *shape):
        return torch.randn(shape, dtype=torch.float64, device="cuda", generator=self.g)

    def uniform(self, lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(shape, dtype=torch.float64, device="cuda", generator=self.g)

    def cx(self, var, *shape):
        s = math.sqrt(var / 2.0)
        return torch.complex(self.real(*shape) * s, self.real(*shape) * s)


def _H(x):
    return x.conj().transpose(-1, -2)


def _chain(w):
    h = torch.zeros(w, w, dtype=torch.complex128, device="cuda")
    i = torch.arange(w - 1, device="cuda")
    h[i, i + 1] = -1.0
    h[i + 1, i] = -1.0
    return h


def _grid(lo, hi, n):
    return torch.linspace(lo, hi, n, dtype=torch.float64, device="cuda") if n > 1 else \
        torch.full((1,), 0.5 * (lo + hi), dtype=torch.float64, device="cuda")


def _strip(case, seed):
    """Disordered square-lattice strip between two clean leads (the strip workload's recipe); with S a
    small Hermitian overlap on every block.  The grid keeps off the rational mode thresholds (such as
    E = 1, 2) where the lead's surface Green's function has a branch point."""
    d, b, nb = _Draw(seed), case["b"], case["nb"]
    eye = torch.eye(b, dtype=torch.complex128, device="cuda")
    dev = dict(b=b, nb=nb, E=_grid(-3.4637, 3.5219, case["ne"]), mu=(0.1, -0.1))
    dev["H_diag"] = _chain(b) + torch.diag_embed(d.uniform(-0.25, 0.25, nb, b)).to(torch.complex128)
    dev["H_upper"] = (-eye).expand(nb - 1, b, b).contiguous()
    dev["leads"] = (_chain(b), -eye.clone())
    if case.get("S"):
        x = d.cx(1.0 / b, nb, b, b) * 0.02
        dev["S_diag"] = (eye + x + _H(x)).contiguous()
        dev["S_upper"] = d.cx(1.0 / b, max(nb - 1, 0), b, b) * 0.02
    return dev


def _random_device(case, seed):
    """Dense random device (the benchmark's recipe): H of unit bandwidth, Sigma^< = i s F F^H,
    Sigma^> = -i s G G^H (block-diagonal, or block-tridiagonal and scaled per energy with ``bt``)."""
    d, b, nb, ne, s = _Draw(seed), case["b"], case["nb"], case["ne"], 1e-2
    dev = dict(b=b, nb=nb, E=_grid(-2.0, 2.0, ne), mu=(0.0, 0.0))
    x = d.cx(1.0 / b, nb, b, b)
    dev["H_diag"] = ((x + _H(x)) / math.sqrt(2.0) + torch.diag_embed(d.uniform(-1.0, 1.0, nb, b))).contiguous()
    dev["H_upper"] = d.cx(0.3 / b, nb - 1, b, b)
    fa, fb = d.cx(1.0 / b, nb, b, b), d.cx(1.0 / b, nb, b, b)
    sl, sg = 1j * s * (fa @ _H(fa)), -1j * s * (fb @ _H(fb))
    if case.get("bt"):
        ca, cb = d.cx(1.0 / b, nb - 1, b, b), d.cx(1.0 / b, nb - 1, b, b)
        sl[1:] += 1j * s * (ca @ _H(ca))
        sg[1:] += -1j * s * (cb @ _H(cb))
        slu, sgu = 1j * s * (fa[:-1] @ _H(ca)), -1j * s * (fb[:-1] @ _H(cb))
        sru = (sgu - slu) / 2
        f = (1.0 + 0.1 * torch.arange(ne, dtype=torch.float64, device="cuda") / ne)[:, None, None, None]
        dev["SigL_upper"], dev["SigR_upper"] = (f * slu).contiguous(), (f * sru).contiguous()
        dev["SigR_lower"] = (-_H(f * sru)).contiguous()
        sl, sg = f * sl, f * sg
    dev["SigL"], dev["SigR"] = sl.contiguous(), ((sg - sl) / 2).contiguous()
    return dev


def _device(case, seed):
    return _strip(case, seed) if case.get("leads") or case["kind"] == "strip" else _random_device(case, seed)


def _wanted(case):
    out = case.get("out", "all")
    if out == "diag":  # the benchmark's outputs
        return ("GR_diag", "GL_diag", "current", "density", "integrals")
    if out == "obs":
        return ("GR_diag", "GL_diag", "current", "density", "contact", "transmission", "integrals")
    return BLOCKS + ("current", "density", "integrals") + (("contact", "transmission") if case["kind"] == "strip" else ())


def _solve_state(case, dev, prec):
    """A user's program around one plan: the plan, the resident inputs and the output buffers."""
    b, nb, ne, want = dev["b"], dev["nb"], dev["E"].numel(), _wanted(case)
    bt = "SigL_upper" in dev
    plan = q.Plan(q.make_desc(nb, b, prec, ne, has_S="S_diag" in dev, has_scattering="SigL" in dev,
                              energy_dependent_sigma=bt, leads="leads" in dev, outputs=want, offdiag_sigma=bt,
                              storage_bits=case.get("bits", 0), refine_tol=case.get("tol", 0.0)))
    inp = q.Inputs()
    for field, key in (("H_diag", "H_diag"), ("H_upper", "H_upper"), ("S_diag", "S_diag"), ("S_upper", "S_upper"),
                       ("SigR_diag", "SigR"), ("SigL_diag", "SigL"), ("SigR_upper", "SigR_upper"),
                       ("SigR_lower", "SigR_lower"), ("SigL_upper", "SigL_upper"), ("energies", "E")):
        if key in dev:
            setattr(inp, field, dev[key].data_ptr())
    if "leads" in dev:
        inp.lead_H00_L = inp.lead_H00_R = dev["leads"][0].data_ptr()
        inp.lead_H01_L = inp.lead_H01_R = dev["leads"][1].data_ptr()
    inp.eta, inp.mu_L, inp.mu_R, inp.kT = ETA, dev["mu"][0], dev["mu"][1], 0.025
    inp.n_energies = ne
    out, bufs = q.Outputs(), {}
    f64 = dict(dtype=torch.float64, device="cuda")
    for name in want:
        if name == "integrals":
            bufs["current_int"], bufs["density_int"] = torch.zeros(nb - 1, **f64), torch.zeros(nb, **f64)
        elif name in BLOCKS:
            bufs[name] = torch.empty((ne, nb if "diag" in name else nb - 1, b, b), dtype=torch.complex128, device="cuda")
        else:
            bufs[name] = torch.empty(dict(current=(ne, nb - 1), density=(ne, nb), contact=(ne, 2), transmission=(ne,))[name], **f64)
    bufs["status_per_energy"] = torch.zeros(ne, dtype=torch.int32, device="cuda")
    for name, t in bufs.items():
        setattr(out, name, t.data_ptr())
    return dict(plan=plan, inp=inp, out=out, bufs=bufs, dev=dev)


def _uneven(case, seed):
    bs, nbs = [int(x) for x in case["bs"].split(",")], [int(x) for x in case["nbs"].split(",")]
    subs = [dict(kind="device", b=b, nb=nb, ne=case["ne"], prec=case["prec"], out="diag") for b, nb in zip(bs, nbs)]
    return subs, [_random_device(c, seed * 8 + k) for k, c in enumerate(subs)]


def _w_inputs(case, seed):
    """Screened-Coulomb inputs (the W workload's recipe): Hermitian BT V, anti-Hermitian BT P^<, P^>."""
    d, b, nb, ne = _Draw(seed), case["b"], case["nb"], case["ne"]
    eye = torch.eye(b, dtype=torch.complex128, device="cuda")
    x = d.cx(1.0, nb, b, b)
    w = dict(V_diag=eye + (x + _H(x)) / (2 * math.sqrt(b)), V_upper=d.cx(1.0, nb - 1, b, b) / (2 * math.sqrt(b)))
    f = (1.0 + 0.5 * torch.arange(ne, dtype=torch.float64, device="cuda") / ne)[:, None, None, None]
    for key, sgn in (("PL", 4j), ("PG", -4j)):
        dd, lo = d.cx(1.0 / b, nb, b, b), d.cx(1.0 / b, nb - 1, b, b)
        d0 = dd @ _H(dd)
        d0[1:] += lo @ _H(lo)
        w[key + "_diag"], w[key + "_upper"] = sgn * f * d0, sgn * f * (dd[:-1] @ _H(lo))
    w["PR_diag"], w["PR_upper"] = (w["PG_diag"] - w["PL_diag"]) / 2, (w["PG_upper"] - w["PL_upper"]) / 2
    w["PR_lower"] = -_H(w["PR_upper"])
    return w


def _zgemm_operands(case, seed):
    d, m, n, k, bt = _Draw(seed), case["m"], case["n"], case["k"], case["batch"]
    A = d.cx(1.0, bt, m, k) if case["opa"] == "N" else d.cx(1.0, bt, k, m)
    B = d.cx(1.0 / k, bt, k, n) if case["opb"] == "N" else d.cx(1.0 / k, bt, n, k)
    return A, B, d.cx(1.0, bt, m, n) if case["beta"] else None


def _lead(case, seed):
    d, n = _Draw(seed), case["b"]
    x = d.cx(1.0 / n, n, n) * 0.1
    H00 = (_chain(n) + x + _H(x)).contiguous()
    H01 = (-torch.eye(n, dtype=torch.complex128, device="cuda") + 0.1 * d.cx(1.0 / n, n, n)).contiguous()
    return H00, H01, _grid(-3.0, 3.0, case["ne"])


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("strip", "device"):
        return dict(kind=kind, **_solve_state(case, _device(case, seed), case["prec"]))
    if kind == "uneven":
        subs, devs = _uneven(case, seed)
        items = [_solve_state(c, dev, case["prec"]) for c, dev in zip(subs, devs)]
        return dict(kind=kind, items=items, group=q.Group([it["plan"] for it in items]))
    if kind == "wsystem":
        w = {k: v.cpu().numpy() for k, v in _w_inputs(case, seed).items()}
        w.update(n_blocks=case["nb"], block_size=case["b"], n_energies=case["ne"])
        return dict(kind=kind, ws=q.WSystem(w, case["prec"], case["ne"]))
    if kind == "zgemm":
        A, B, C0 = _zgemm_operands(case, seed)
        return dict(kind=kind, A=A, B=B, C0=C0, case=case)
    if kind == "zinv":
        d, n = _Draw(seed), case["b"]
        A = d.cx(1.0 / n, case["batch"], n, n) + (2.0 + 0.5j) * torch.eye(n, dtype=torch.complex128, device="cuda")
        return dict(kind=kind, A=A, prec=case["prec"])
    if kind == "lead":
        H00, H01, E = _lead(case, seed)
        return dict(kind=kind, H00=H00, H01=H01, E=E)
    d = _Draw(seed)  # values over the decades that Green's functions span
    x = d.real(case["count"]) * torch.exp(d.uniform(-25.0, 5.0, case["count"]))
    return dict(kind=kind, x=x, bits=case["bits"])


def run(state):
    kind = state["kind"]
    stream = torch.cuda.current_stream().cuda_stream
    if kind in ("strip", "device"):
        state["plan"].solve(state["inp"], state["out"], stream)
        return state["bufs"]
    if kind == "uneven":
        items = state["items"]
        state["group"].solve([it["inp"] for it in items], [it["out"] for it in items], stream)
        return [it["bufs"] for it in items]
    if kind == "wsystem":
        state["ws"].run()
        return state["ws"].res
    if kind == "zgemm":
        c = state["case"]
        return q.zgemm_batched(state["A"], state["B"], c["prec"], c["opa"], c["opb"], alpha=-0.5,
                               beta=1.0 if c["beta"] else 0.0, C0=state["C0"])
    if kind == "zinv":
        return q.zinv_batched(state["A"].clone(), state["prec"])
    if kind == "lead":
        return q.lead_self_energy(state["H00"], state["H01"], state["E"], ETA)
    codes = q.fpx_compress(state["x"], state["bits"])
    return codes, q.fpx_decompress(codes, state["bits"], state["x"].numel())


# ------------------------------------------------------------------------------------------- work
def _solve_work(b, nb, ne, prec, want, bt=False, leads=False, S=False):
    # per slice: inverse, 6 products forward, 6 backward (7 with G_{i,i+1}), 3 more cross terms with bt
    prods = 13 + (1 if "GR_upper" in want else 0) + (3 if bt else 0)
    n_blk = sum(nb if "diag" in w else nb - 1 for w in want if w in BLOCKS)
    sets = ne if bt else 1
    inputs = (2 * nb - 1) * (2 if S else 1) + (0 if leads else 2 * nb * sets) + (3 * (nb - 1) * sets if bt else 0)
    # contacts: about 20 decimation sweeps of one inverse and six products, at both ends
    flops = 8.0 * b ** 3 * ne * (prods * nb + (2 * 20 * 7 if leads else 0))
    return 16.0 * b * b * (ne * n_blk + inputs), flops


def work(case):
    kind = case["kind"]
    if kind in ("strip", "device"):
        leads = kind == "strip" or bool(case.get("leads"))
        by, fl = _solve_work(case["b"], case["nb"], case["ne"], case["prec"], _wanted(case), bool(case.get("bt")), leads, bool(case.get("S")))
        return dict(bytes=by, flops=fl)
    if kind == "uneven":
        subs = [_solve_work(int(b), int(nb), case["ne"], case["prec"], _wanted(dict(kind="device", out="diag")))
                for b, nb in zip(case["bs"].split(","), case["nbs"].split(","))]
        return dict(bytes=sum(s[0] for s in subs), flops=sum(s[1] for s in subs))
    if kind == "wsystem":
        b, nb, ne = case["b"], case["nb"], case["ne"]
        # assembly: 7 + 2 (13 + 6) block products per inner slice; solve: BT sweeps, two right-hand sides
        return dict(bytes=16.0 * b * b * ne * nb * (7 + 7 + 7), flops=8.0 * b ** 3 * ne * nb * (45 + 8 + 2 * 11))
    if kind == "zgemm":
        m, n, k, bt = case["m"], case["n"], case["k"], case["batch"]
        return dict(bytes=16.0 * bt * (m * k + k * n + m * n * (2 if case["beta"] else 1)), flops=8.0 * bt * m * n * k)
    if kind == "zinv":
        return dict(bytes=32.0 * case["batch"] * case["b"] ** 2, flops=8.0 * case["batch"] * case["b"] ** 3)
    if kind == "lead":
        return dict(bytes=16.0 * case["b"] ** 2 * (case["ne"] + 2), flops=8.0 * case["b"] ** 3 * case["ne"] * 20 * 7)
    return dict(bytes=case["count"] * (16.0 + 2 * case["bits"] / 8.0), flops=0)


def tolerance(case):
    """About four times the largest error against ``exact`` over the declared ranges."""
    kind, prec = case["kind"], case.get("prec")
    if kind == "fpx":
        return "exact"
    # FP64 with contacts: the decimation inverts blocks of condition 3e4 and more at eta = 1e-6
    # (measured up to 4e-9 on the strips, 2e-8 for wide leads)
    if kind == "strip":
        return {"rel": 2e-8}
    if kind == "lead" or case.get("leads"):
        return {"rel": 8e-8}
    # measured 3.4e-16 (fp64), 1.8e-7 (fp32), 9.9e-12 (emu64), 2.5e-4 (bf16x3)
    if kind == "zgemm":
        return {"rel": dict(fp64=2e-15, fp32=1e-6, emu64=4e-11, bf16x3=1e-3)[prec]}
    # measured 5e-16 (fp64, n = 18), 1.4e-6 (fp32), 9e-11 (emu64)
    if kind == "zinv":
        return {"rel": dict(fp64=2e-14, fp32=1e-5, emu64=4e-10)[prec]}
    # solves: the current is a small difference of large traces and carries the largest error
    # (measured 1.2e-11 in fp64, 4.5e-3 in fp32, 1.1e-7 in emu64)
    return {"rel": dict(fp64=1e-10, fp32=2e-2, emu64=5e-7)[prec]}


# ------------------------------------------------------------- the same in plain torch, 64 bits
def _exact_lead(H00, H01, E):
    n = H00.shape[0]
    z = (E + 1j * ETA)[:, None, None] * torch.eye(n, dtype=torch.complex128, device="cuda")
    al, be = H01.expand(len(E), n, n), _H(H01).expand(len(E), n, n)
    ep = es = H00.expand(len(E), n, n)
    for _ in range(100):
        g = torch.linalg.inv(z - ep)
        ag, bg = al @ g, be @ g
        d = ag @ be
        es, ep = es + d, ep + d + bg @ al
        al, be = ag @ al, bg @ be
        if max(al.abs().max().item(), be.abs().max().item()) < 1e-16:
            break
    return H01 @ torch.linalg.inv(z - es) @ _H(H01)


def _exact_sweeps(A, U, V, SL, L=None):
    """Selected inverse and lesser blocks of a block-tridiagonal system: A(i), U(i), V(i) and the
    right-hand side SL(i) (upper blocks L(i)) as batched blocks.  Returns per-slice lists."""
    nb = len(A)
    g, gl = [], []
    for i in range(nb):
        a, s = A[i], SL[i]
        if i:
            a = a - V[i - 1] @ g[i - 1] @ U[i - 1]
            s = s + V[i - 1] @ gl[i - 1] @ _H(V[i - 1])
            if L is not None:
                y = V[i - 1] @ g[i - 1] @ L[i - 1]
                s = s - y + _H(y)
        g.append(torch.linalg.inv(a))
        gl.append(g[i] @ s @ _H(g[i]))
    R = dict(GR_diag=[None] * nb, GR_upper=[None] * (nb - 1), GR_lower=[None] * (nb - 1),
             GL_diag=[None] * nb, GL_upper=[None] * (nb - 1))
    R["GR_diag"][-1], R["GL_diag"][-1] = g[-1], gl[-1]
    for i in range(nb - 2, -1, -1):
        Gn, GLn = R["GR_diag"][i + 1], R["GL_diag"][i + 1]
        p, z = g[i] @ U[i], V[i] @ g[i]
        qq = V[i] @ gl[i]
        if L is not None:
            qq = qq + _H(g[i] @ L[i])
        R["GR_upper"][i], R["GR_lower"][i] = -p @ Gn, -Gn @ z
        R["GR_diag"][i] = g[i] + p @ Gn @ z
        x2 = Gn @ qq
        k = p @ x2
        R["GL_diag"][i] = gl[i] + p @ GLn @ _H(p) + k - _H(k)
        R["GL_upper"][i] = -p @ GLn + _H(x2)
    return R


def _exact_solve(case, dev):
    nb, b, E, ne = dev["nb"], dev["b"], dev["E"], dev["E"].numel()
    eye = torch.eye(b, dtype=torch.complex128, device="cuda")
    z = (E + 1j * ETA)[:, None, None]
    S = dev["S_diag"] if "S_diag" in dev else eye.expand(nb, b, b)
    per = lambda k, i: dev[k][:, i] if dev[k].dim() == 4 else dev[k][i]  # noqa: E731
    A = [z * S[i] - dev["H_diag"][i] - (per("SigR", i) if "SigR" in dev else 0) for i in range(nb)]
    SL = [per("SigL", i).expand(ne, b, b) if "SigL" in dev else torch.zeros(ne, b, b, dtype=torch.complex128, device="cuda")
          for i in range(nb)]
    Su = dev.get("S_upper")
    hu = [(z * Su[i] if Su is not None else 0) - dev["H_upper"][i].expand(ne, b, b) for i in range(nb - 1)]
    hl = [(z * _H(Su[i]) if Su is not None else 0) - _H(dev["H_upper"][i]).expand(ne, b, b) for i in range(nb - 1)]
    U = [hu[i] - (per("SigR_upper", i) if "SigR_upper" in dev else 0) for i in range(nb - 1)]
    V = [hl[i] - (per("SigR_lower", i) if "SigR_lower" in dev else 0) for i in range(nb - 1)]
    con = []
    if "leads" in dev:
        sr = _exact_lead(*dev["leads"], E)
        for i, mu in ((0, dev["mu"][0]), (nb - 1, dev["mu"][1])):
            gam = 1j * (sr - _H(sr))
            f = torch.sigmoid(-(E - mu) / 0.025)[:, None, None]
            con.append((i, gam, 1j * f * gam, -1j * (1 - f) * gam))
            A[i] = A[i] - sr
            SL[i] = SL[i] + con[-1][2]
    L = [per("SigL_upper", i) for i in range(nb - 1)] if "SigL_upper" in dev else None
    R = _exact_sweeps(A, U, V, SL, L)
    res = {k: torch.stack(R[k], 1) for k in R}
    gd = [R["GL_diag"][i] + R["GR_diag"][i] - _H(R["GR_diag"][i]) for i in range(nb)]
    tr = lambda x, y: (x * y.transpose(-1, -2)).sum((-1, -2))  # noqa: E731
    cur = torch.stack([-2 * ((dev["H_upper"][i] - (E[:, None, None] * Su[i] if Su is not None else 0)) * R["GL_upper"][i].conj()).sum((-1, -2)).real
                       for i in range(nb - 1)], 1)
    den = torch.stack([torch.diagonal(R["GL_diag"][i], dim1=-2, dim2=-1).sum(-1).imag for i in range(nb)], 1)
    res.update(GG_diag=torch.stack(gd, 1), current=cur, density=den,
               GG_upper=torch.stack([R["GL_upper"][i] + R["GR_upper"][i] - _H(R["GR_lower"][i]) for i in range(nb - 1)], 1))
    w = torch.zeros_like(E)
    if ne > 1:
        d = E[1:] - E[:-1]
        w[:-1] += d / 2
        w[1:] += d / 2
    res["current_int"], res["density_int"] = (w[:, None] * cur).sum(0), (w[:, None] * den).sum(0) / (2 * math.pi)
    if con:
        res["contact"] = torch.stack([(tr(sl, gd[i]) - tr(sg, R["GL_diag"][i])).real for i, _, sl, sg in con], 1)
        gam, G0 = con[0][1], R["GR_diag"][0]
        res["transmission"] = tr(gam, 1j * (G0 - _H(G0))).real - tr(gam @ G0, gam @ _H(G0)).real
    names = [n for n in _wanted(case) if n != "integrals"] + (["current_int", "density_int"] if "integrals" in _wanted(case) else [])
    out = {n: res[n].contiguous() for n in names}
    out["status_per_energy"] = None
    return out


def _exact_w(case, seed):
    w, nb, b = _w_inputs(case, seed), case["nb"], case["b"]
    full = lambda i, j, d, u, lo: d[..., i, :, :] if i == j else (u[..., i, :, :] if j == i + 1 else lo[..., j, :, :])  # noqa: E731
    V = lambda i, j: full(i, j, w["V_diag"], w["V_upper"], _H(w["V_upper"]))  # noqa: E731
    ok = lambda i, j: abs(i - j) <= 1 and 0 <= j < nb  # noqa: E731
    out, sys = {}, {}

    def row(P, i, j):  # (V P)_ij
        return sum(V(i, k) @ P(k, j) for k in range(max(0, i - 1), min(nb, i + 2)) if ok(k, j))

    PR = lambda i, j: full(i, j, w["PR_diag"], w["PR_upper"], w["PR_lower"])  # noqa: E731
    eye = torch.eye(b, dtype=torch.complex128, device="cuda")
    out["M_diag"] = torch.stack([eye - row(PR, i, i) for i in range(nb)], 1)
    out["M_upper"] = torch.stack([-row(PR, i, i + 1) for i in range(nb - 1)], 1)
    out["M_lower"] = torch.stack([-row(PR, i + 1, i) for i in range(nb - 1)], 1)
    for key in ("L", "G"):
        d, u = w["P%s_diag" % key], w["P%s_upper" % key]
        P = lambda i, j, d=d, u=u: full(i, j, d, u, -_H(u))  # noqa: E731
        B = lambda i, j, P=P: sum(row(P, i, l) @ _H(V(j, l)) for l in range(max(0, j - 1), min(nb, j + 2)) if abs(i - l) <= 2)  # noqa: E731,E741
        out["B%s_diag" % key] = torch.stack([B(i, i) for i in range(nb)], 1)
        out["B%s_upper" % key] = torch.stack([B(i, i + 1) for i in range(nb - 1)], 1)
        blk = lambda k: [out[k][:, i] for i in range(out[k].shape[1])]  # noqa: E731
        R = _exact_sweeps(blk("M_diag"), blk("M_upper"), blk("M_lower"), blk("B%s_diag" % key), blk("B%s_upper" % key))
        for name in ("diag", "upper"):
            sys["X%s_%s" % (key, name)] = torch.stack(R["GL_" + name], 1)
        for name in ("diag", "upper", "lower"):
            sys["XR_" + name] = torch.stack(R["GR_" + name], 1)
    out.update(sys)
    out["status"] = None
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("strip", "device"):
        return _exact_solve(case, _device(case, seed))
    if kind == "uneven":
        subs, devs = _uneven(case, seed)
        return [_exact_solve(c, d) for c, d in zip(subs, devs)]
    if kind == "wsystem":
        return _exact_w(case, seed)
    if kind == "zgemm":
        A, B, C0 = _zgemm_operands(case, seed)
        C = -0.5 * ((A if case["opa"] == "N" else _H(A)) @ (B if case["opb"] == "N" else _H(B)))
        return C + C0 if C0 is not None else C
    if kind == "zinv":
        return [torch.linalg.inv(prepare(case, seed)["A"]), None]
    if kind == "lead":
        return [_exact_lead(*_lead(case, seed)), None]
    # round to X - 9 stored significand bits, ties to even (the values are normal FP32 numbers)
    u = prepare(case, seed)["x"].view(torch.int64)
    sh = 52 - (case["bits"] - 9)
    r = ((u + ((1 << (sh - 1)) - 1) + ((u >> sh) & 1)) >> sh) << sh
    return [None, r.view(torch.float64)]
