"""Performance cases: what a user of the library has it do, through its public
entry points, from the smallest call to gigabytes of pair elements.

Most cases are one build of the blocks A and B (Eqs. emat, vrrofM, wrrm,
wrabar) from pair elements that are on the device: through a plan made once
(how a program that sweeps momentum transfers or repeats a build calls the
library) or through the one-call FP64 build.  The others are the steps before
and after it: the static screening W of one q, eps_M on a frequency grid by
the Lanczos recursion, and the lowest excitons.

Band windows, plane-wave counts and k grids are those of this repository's
configurations and of the published workloads its baseline lists (2 x 2 to
20 x 20 bands, 59 to 500 plane waves); k grids are cut where a problem would
not fit the card several times over.
"""
import math

import numpy as np
import torch

import paper_1904_05575_gb300 as bse

HARTREE_EV = 27.211386245988
A_LAT = 10.26                       # Si lattice constant (bohr), FCC cell
OMEGA_CELL = A_LAT ** 3 / 4
STEPS = 640                         # Lanczos steps that eps_M on the grid below takes, about


def listed():
    return [
        # the smallest problem: a 2 x 2 x 2 grid with 2 x 2 bands, as in a first
        # convergence check or a server that answers many small requests
        _build("first_check", grid=2, nv=2, nc=2, ng=59),
        # optical limit of a small unit cell: 4 x 4 bands on 4 x 4 x 4 k points
        _build("optical_limit", grid=4, nv=4, nc=4, ng=181, autotune=True),
        # several momentum transfers with uneven band windows in one plan
        _build("uneven_windows", grid=6, windows="2x2,3x5,4x6", ng=113, autotune=True,
               hermitian=True),
        # 4 occupied x 12 unoccupied bands: the window of the LiF and Si spectra
        _build("valence_window", grid=4, nv=4, nc=12, ng=181),
        # molecular crystal: 20 x 20 bands, 500 plane waves, Hermitian plan
        _build("molecular", grid=3, nv=20, nc=20, ng=500, autotune=True, hermitian=True),
        # 12 x 12 bands (a molecule in a cell), Tamm-Dancoff, pair elements kept
        # in single precision to halve their memory
        _build("molecular_tda_c64", grid=4, nv=12, nc=12, ng=300, coupling=False, dtype="c64"),
        # core levels: 2 x 20 bands, a slab of k rows of a problem whose pair
        # elements are too many to hold at once
        _build("core_slab", grid=5, nv=2, nc=20, ng=300, slab=32, autotune=True),
        # the plain FP64 build in one call: checks and reference results
        _build("fp64_call", grid=3, nv=4, nc=4, ng=181, call=True, precision="fp64"),
        # eps_M on a grid of 2,000 frequencies from A and B, FP64 products
        {"name": "eps_grid", "kind": "eps", "n": 1024, "precision": "fp64"},
        # the same for a larger problem, products on the tensor cores
        {"name": "eps_grid_large", "kind": "eps", "n": 4860, "precision": "bf16x6"},
        # the lowest excitons (bound states below the onset)
        {"name": "lowest_excitons", "kind": "excitons", "n": 2560, "nev": 8,
         "precision": "bf16x6"},
        # static RPA screening of one q from the transitions of a whole grid
        {"name": "screening", "kind": "screening", "grid": 4, "nv": 20, "nc": 20, "ng": 500,
         "precision": "bf16x6"},
    ]


def draw(rng):
    fam = rng.choice(["small", "optical", "uneven", "window", "molecular", "c64", "core", "fp64",
                      "eps", "eps_large", "excitons", "screening"])
    if fam == "small":
        return _build(None, grid=rng.randint(1, 3), nv=rng.randint(1, 3), nc=rng.randint(1, 3),
                      ng=_log(rng, 15, 113))
    if fam == "optical":
        b = rng.choice([2, 4])
        return _build(None, grid=rng.randint(3, 4), nv=b, nc=b, ng=rng.randint(65, 192),
                      autotune=True, hermitian=rng.random() < 0.5)
    if fam == "uneven":
        w = ["%dx%d" % (rng.randint(2, 4), rng.randint(2, 6)) for _ in range(rng.randint(1, 3))]
        return _build(None, grid=rng.randint(3, 5), windows=",".join(w), ng=rng.randint(59, 137),
                      autotune=True, hermitian=rng.random() < 0.5)
    if fam == "window":
        return _build(None, grid=rng.randint(2, 4), nv=rng.randint(3, 6), nc=rng.randint(8, 13),
                      ng=rng.randint(89, 220), hermitian=rng.random() < 0.5)
    if fam == "molecular":
        return _build(None, grid=rng.randint(2, 3), nv=rng.randint(8, 20), nc=rng.randint(8, 18),
                      ng=_log(rng, 113, 480), autotune=True, hermitian=True)
    if fam == "c64":
        return _build(None, grid=rng.randint(2, 4), nv=rng.randint(8, 12), nc=rng.randint(8, 12),
                      ng=_log(rng, 89, 300), coupling=rng.random() < 0.5, dtype="c64")
    if fam == "core":
        g = rng.randint(3, 5)
        return _build(None, grid=g, nv=rng.randint(1, 2), nc=rng.randint(8, 20),
                      ng=_log(rng, 113, 300), slab=rng.randint(g, 5 * g), autotune=True)
    if fam == "fp64":
        return _build(None, grid=rng.randint(2, 3), nv=rng.randint(2, 4), nc=rng.randint(2, 4),
                      ng=_log(rng, 59, 181), call=True, precision="fp64")
    if fam == "eps":
        return {"kind": "eps", "n": _log(rng, 100, 2000), "precision": "fp64"}
    if fam == "eps_large":
        return {"kind": "eps", "n": _log(rng, 2000, 4800), "precision": "bf16x6"}
    if fam == "excitons":
        return {"kind": "excitons", "n": _log(rng, 400, 2500), "nev": rng.randint(4, 8),
                "precision": rng.choice(["fp64", "bf16x6"])}
    return {"kind": "screening", "grid": rng.randint(2, 4), "nv": rng.randint(4, 20),
            "nc": rng.randint(4, 20), "ng": _log(rng, 59, 480),
            "precision": rng.choice(["fp64", "bf16x6", "bf16x6"])}


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _build(name, grid, ng, nv=0, nc=0, windows="", autotune=False, hermitian=False, coupling=True,
           dtype="c128", slab=0, call=False, precision="bf16x6"):
    c = {"kind": "build", "grid": grid, "windows": windows or "%dx%d" % (nv, nc), "ng": ng,
         "autotune": autotune, "hermitian": hermitian, "coupling": coupling, "dtype": dtype,
         "slab": min(slab, grid ** 3), "call": call, "precision": precision}
    return c if name is None else dict(c, name=name)


def _windows(case):
    return [tuple(int(x) for x in w.split("x")) for w in case["windows"].split(",")]


def _precision(case):
    return {"fp64": bse.BSE_PREC_FP64, "bf16x6": bse.BSE_PREC_BF16X6}[case["precision"]]


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed, *more):
    g = torch.Generator(device="cuda")
    for m in more:
        seed = (seed * 1000003 + m) % (1 << 40)
    g.manual_seed(seed)
    return g


def _cn(g, *shape):
    """Complex normal numbers; what they are multiplied with fills all 64 bits."""
    return torch.randn(shape, dtype=torch.complex64, device="cuda", generator=g).to(torch.complex128)


def _g2(ng):
    """|G|^2 of the first ng reciprocal-lattice vectors of the FCC cell."""
    b = 2.0 * np.pi / A_LAT * np.array([[-1, 1, 1], [1, -1, 1], [1, 1, -1]], float)
    r = np.arange(-9, 10)
    cart = np.stack(np.meshgrid(r, r, r, indexing="ij"), -1).reshape(-1, 3) @ b
    order = np.argsort((cart ** 2).sum(1), kind="stable")[:ng]
    return cart[order]


def _maps(n):
    r = np.arange(n)
    k = np.stack(np.meshgrid(r, r, r, indexing="ij"), -1).reshape(-1, 3)
    idx = lambda c: ((c[..., 0] % n) * n + c[..., 1] % n) * n + c[..., 2] % n  # noqa: E731
    return (idx(k[:, None] - k[None]).astype(np.int32), idx(-k[:, None] - k[None]).astype(np.int32),
            idx(-k))


def _pairs(g, rows, nk, nb, damp, herm):
    """Pair elements [rows, nk, nb, nb, ng]; Hermitian in (k b) <-> (k' b') for whole problems."""
    x = _cn(g, rows, nk, nb, nb, damp.numel())
    if herm:
        x += x.permute(1, 0, 3, 2, 4).conj()
        x *= damp * math.sqrt(0.5)
    else:
        x *= damp
    return x


def _problem(case, i, seed):
    """One momentum transfer's arrays, as bse.upload_problem takes them."""
    nv, nc = _windows(case)[i]
    n, ng = case["grid"], case["ng"]
    nk = n ** 3
    g = _gen(seed, i)
    gvec = _g2(ng)
    core = nv <= 2 and nc >= 8
    damp = torch.as_tensor(1.0 / (1.0 + (0.05 if core else 1.0) * (gvec ** 2).sum(1)), device="cuda")
    lo = -400.5 if core else -3.0
    rand = lambda *s: torch.rand(s, dtype=torch.float64, device="cuda", generator=g)  # noqa: E731
    rows = case["slab"] or nk
    qm, qp, neg = _maps(n)
    w = _cn(g, nk, ng, ng)
    w = 0.5 * (w + w.transpose(1, 2).conj())
    w = 0.5 * (w + w[torch.as_tensor(neg, device="cuda")].conj())
    gv = torch.as_tensor(gvec, device="cuda")
    w /= 1.0 + torch.cdist(gv, gv)
    w.diagonal(dim1=1, dim2=2).copy_(1.0 + w.abs().sum(2))
    w *= 0.002 if nv * nc >= 64 else 0.25
    gq2 = ((gvec + np.array([0.1 * i, 0.0, 0.0])) ** 2).sum(1)
    v_bar = np.zeros(ng)
    v_bar[1:] = 4.0 * np.pi / gq2[1:]
    return dict(nk=nk, nv=nv, nc=nc, ng=ng, omega_cell=OMEGA_CELL, e_v=lo + rand(nk, nv) * (1.0 if core else 3.0),
                e_c=1.0 + 3.0 * rand(nk, nc), m_x=_cn(g, nk, nv, nc, ng) * damp,
                m_vv=_pairs(g, rows, nk, nv, damp, rows == nk), m_cc=_pairs(g, rows, nk, nc, damp, rows == nk),
                n_vc=_cn(g, nk, nk, nv, nc, ng) * damp, w=w, q_minus=torch.as_tensor(qm),
                q_plus=torch.as_tensor(qp), v_bar=torch.as_tensor(v_bar))


def _upload(case, i, seed):
    return bse.upload_problem(_problem(case, i, seed),
                              complex_dtype=torch.complex64 if case["dtype"] == "c64" else None)


def _two_particle(n, seed):
    """A, B (tensors whose row r is column r of the matrix) of a full problem:
    transition energies, a collective exchange part and a random direct part,
    A - B and A + B positive definite; rho; the frequency grid."""
    g = _gen(seed, 7)
    e = 1.0 + 6.0 * torch.rand(n, dtype=torch.float64, device="cuda", generator=g)
    m = _cn(g, n, 16)
    v = (m @ m.transpose(0, 1).conj()) * (0.5 / n)
    out = []
    for sigma in (0.15, 0.08):
        x = _cn(g, n, n)
        x = (x + x.transpose(0, 1).conj()) * (sigma / math.sqrt(2.0 * n)) + v
        x.diagonal().imag.zero_()
        out.append(x)
    out[0].diagonal().real.add_(e)
    rho = m[:, 0] + 0.3 * _cn(g, n)
    return out[0].contiguous(), out[1].contiguous(), rho.contiguous(), torch.linspace(
        0.0, 10.0, 2000, dtype=torch.float64, device="cuda")


def _screening(case, seed):
    nk, nv, nc, ng = case["grid"] ** 3, case["nv"], case["nc"], case["ng"]
    g = _gen(seed, 9)
    gvec = _g2(ng)
    damp = torch.as_tensor(1.0 / (1.0 + (gvec ** 2).sum(1)), device="cuda")
    rand = lambda *s: torch.rand(s, dtype=torch.float64, device="cuda", generator=g)  # noqa: E731
    v = torch.as_tensor(4.0 * np.pi / ((gvec + np.array([0.05, 0.02, 0.0])) ** 2).sum(1), device="cuda")
    return -3.0 * rand(nk, nv), 1.0 + 3.0 * rand(nk, nc), _cn(g, nk, nv, nc, ng) * damp * 0.3, v


# ---------------------------------------------------------------------------
# a pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    prec = _precision(case)
    if case["kind"] == "build":
        ds = [_upload(case, i, seed) for i in range(len(_windows(case)))]
        sts = [bse.make_problem_struct(d, coupling=case["coupling"], k_count=case["slab"]) for d in ds]
        plan = None
        if not case["call"]:
            plan = bse.Plan(sts, precision=prec, autotune=case["autotune"], hermitian=case["hermitian"])
        return dict(case=case, prec=prec, problems=sts, data=ds, plan=plan)
    if case["kind"] == "screening":
        e_v, e_c, m, v = _screening(case, seed)
        w = torch.empty((case["ng"], case["ng"]), dtype=torch.complex128, device="cuda")
        return dict(case=case, prec=prec, args=(e_v, e_c, m, v), w=w)
    n = case["n"]
    a, b, rho, omega = _two_particle(n, seed)
    return dict(case=case, prec=prec, n=n, A=a, B=b, rho=rho, omega=omega,
                eps=torch.empty(omega.numel(), dtype=torch.complex128, device="cuda"),
                E=torch.empty(case.get("nev", 1), dtype=torch.float64, device="cuda"))


VC, DELTA = 64 * OMEGA_CELL, 0.05


def run(state):
    case, prec = state["case"], state["prec"]
    if case["kind"] == "build":
        if state["plan"] is not None:
            state["plan"].execute()
        else:
            bse.bse_build_kernel(state["problems"], prec)
        return [[d["A"], d["B"]] if case["coupling"] else [d["A"]] for d in state["data"]]
    if case["kind"] == "screening":
        bse.bse_rpa_screening(*state["args"], OMEGA_CELL, state["w"], precision=prec)
        return state["w"]
    n, a, b = state["n"], state["A"], state["B"]
    if case["kind"] == "eps":
        bse.bse_spectrum_lanczos(n, a, b, state["rho"], 4.0 * math.pi, VC, state["omega"], DELTA,
                                 state["eps"], tol=1e-8, matvec_precision=prec)
        return state["eps"]
    bse.bse_lowest_excitons(n, a, b, case["nev"], state["E"], tol_ev=1e-5, max_iter=200,
                            matvec_precision=prec)
    return state["E"]


def work(case):
    if case["kind"] == "build":
        nk, ng, el = case["grid"] ** 3, case["ng"], 8 if case["dtype"] == "c64" else 16
        rows, half = case["slab"] or nk, case["hermitian"]
        pairs = nk * (nk + 1) // 2 if half else rows * nk      # blocks of the direct terms
        b = f = 0
        for nv, nc in _windows(case):
            n, cpl = nk * nv * nc, 1 if case["coupling"] else 0
            b += el * ng * (n + pairs * (nv * nv + nc * nc) + cpl * nk * nk * nv * nc + nk * ng)
            b += 16 * (1 + cpl) * rows * nv * nc * n
            f += 8 * ng * (n * (n + 1) // 2 if rows == nk else rows * nv * nc * n)
            f += 8 * pairs * ng * (min(nv, nc) ** 2 * ng + (nv * nc) ** 2)
            f += 8 * cpl * pairs * ng * (nv * nc * ng + (nv * nc) ** 2)
        return {"bytes": b, "flops": f}
    if case["kind"] == "screening":
        t, ng = case["grid"] ** 3 * case["nv"] * case["nc"], case["ng"]
        return {"bytes": 16 * ng * (t + ng), "flops": 4 * t * ng * ng + 8 * ng ** 3}
    n = case["n"]
    if case["kind"] == "eps":
        return {"bytes": 32 * n * n, "flops": 16 * n * n * STEPS}
    return {"bytes": 32 * n * n, "flops": 16 * n * n * 10 * case["nev"]}


# ---------------------------------------------------------------------------
# the same results in plain 64-bit torch
# ---------------------------------------------------------------------------
def exact(case, seed):
    if case["kind"] == "build":
        return [_exact_build(case, i, seed) for i in range(len(_windows(case)))]
    if case["kind"] == "screening":
        e_v, e_c, m, v = _screening(case, seed)
        nk, nv, nc, ng = m.shape
        t = (m / torch.sqrt(e_c[:, None, :] - e_v[:, :, None])[..., None]).reshape(-1, ng)
        x = t.transpose(0, 1).conj() @ t
        kap = HARTREE_EV / (nk * OMEGA_CELL)
        eps = torch.eye(ng, dtype=torch.complex128, device="cuda") + 2.0 * kap * x * v[None, :]
        return v[:, None] * torch.linalg.inv(eps)
    n = case["n"]
    if n > 5000:
        return None
    at, bt, rho, omega = _two_particle(n, seed)
    a, b = at.transpose(0, 1), bt.transpose(0, 1)
    low = torch.linalg.cholesky(a - b)
    s = low.transpose(0, 1).conj() @ (a + b) @ low
    s = 0.5 * (s + s.transpose(0, 1).conj())
    if case["kind"] == "excitons":
        return torch.sqrt(torch.linalg.eigvalsh(s)[:case["nev"]])
    e2, z = torch.linalg.eigh(s)
    u = z.transpose(0, 1).conj() @ (low.transpose(0, 1).conj() @ rho.conj())
    z2 = torch.complex(omega, torch.full_like(omega, DELTA)) ** 2
    terms = (u.abs() ** 2)[None, :] / (z2[:, None] - e2[None, :])
    return 1.0 - 4.0 * math.pi * HARTREE_EV * (2.0 / VC) * terms.sum(1)


def _exact_build(case, i, seed):
    d = _problem(case, i, seed)
    if case["dtype"] == "c64":
        for k in ("m_x", "m_vv", "m_cc", "n_vc", "w"):
            d[k] = d[k].to(torch.complex64).to(torch.complex128)
    nk, nv, nc, ng = d["nk"], d["nv"], d["nc"], d["ng"]
    n, rows = nk * nv * nc, case["slab"] or nk
    kap = HARTREE_EV / (nk * OMEGA_CELL)
    qm, qp = d["q_minus"].cuda().long(), d["q_plus"].cuda().long()
    # at[k' v' c' k v c]: row r of the tensor is column r of the matrix
    mx = d["m_x"].reshape(n, ng)
    at = torch.zeros((nk, nv, nc, nk, nv, nc), dtype=torch.complex128, device="cuda")
    r = rows * nv * nc
    at.view(n, n)[:, :r] = 2.0 * kap * (mx @ (mx[:r].conj() * d["v_bar"].cuda()).transpose(0, 1))
    bt = at.clone() if case["coupling"] else None
    w = d["w"]
    for k in range(rows):
        u = d["m_vv"][k].reshape(nk, nv * nv, ng).conj() @ w[qm[k]]
        p = u @ d["m_cc"][k].reshape(nk, nc * nc, ng).transpose(1, 2)
        p = p.reshape(nk, nv, nv, nc, nc)                       # k' v v' c c'
        at[:, :, :, k] -= kap * p.permute(0, 2, 4, 1, 3)        # k' v' c' v c
        if bt is not None:
            u = d["n_vc"][:, k].reshape(nk, nv * nc, ng).conj() @ w[qp[k]]
            p = u @ d["n_vc"][k].reshape(nk, nv * nc, ng).transpose(1, 2)
            p = p.reshape(nk, nv, nc, nv, nc)                   # k' v' c v c'
            bt[:, :, :, k] -= kap * p.permute(0, 1, 4, 3, 2)    # k' v' c' v c
    e = (d["e_c"][:, None, :] - d["e_v"][:, :, None]).reshape(-1)[:r]
    at.view(n, n)[:, :r].diagonal().add_(e)
    return [at.view(n, n)] + ([bt.view(n, n)] if bt is not None else [])
