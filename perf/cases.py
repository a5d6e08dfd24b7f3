"""Performance cases: what programs that use this package have it compute.

Each case is one call (or the forward and backward of one training step) through
the public entry points, on synthetic inputs of the forms this repository's
configurations, tests and benchmark use: gapped random spectra (dense Haar-like
eigenvectors), gapped tight-binding rods (4 orbitals per site, sites sorted along
the rod), and gapless spectra at finite temperature. Every input is made on the
GPU from the case and a seed alone. `exact` gives the same outputs from FP64
eigendecompositions.
"""
import math

import torch

import paper_2409_17033_gb300 as sp2

NORB = 4          # orbitals per site
RCUT, DECAY, DENSITY, WIDTH = 6.0, 1.5, 0.1, 6.0
MAX_EXACT_N = 4200    # above this an FP64 eigendecomposition takes too long


def listed():
    return [
        # The FP64 reference calculation of a small molecule: idempotency 1e-10, the
        # smallest whole call, where launches and latency count.
        dict(name="density_fp64_n128", op="density", inp="spectrum", n=128, mode="fp64"),
        # A full-precision susceptibility of one dense observable at an odd size: the
        # reference every mixed-precision result is judged by (forward + adjoint).
        dict(name="chi_fp64_n1001", op="chi", inp="spectrum", n=1001, mode="fp64", batch=1,
             diag=False, direction="backward"),
        # The binding's default arithmetic on a small ragged system: one density
        # matrix per geometry of a molecular-dynamics run.
        dict(name="density_bf16x2_n300", op="density", inp="rod", n=300, mode="bf16x2"),
        # Primal responses to a batch of site potentials on a ragged mid-size system.
        dict(name="response_fp16x2_n1000_k16", op="response", inp="rod", n=1000, mode="fp16x2",
             batch=16, diag=True),
        # One training step through torch.autograd: D(H), a loss Tr[G D], dloss/dH.
        dict(name="autograd_fp16x2_n2048", op="autograd", inp="rod", n=2048, mode="fp16x2"),
        # The plain single-precision form users compare the mixed modes with
        # (forward susceptibility of one observable).
        dict(name="chi_fwd_fp32_n1500", op="chi", inp="rod", n=1500, mode="fp32", batch=1,
             diag=True, direction="forward"),
        # The dual form of four diagonal observables at N = 4096 (then any number of
        # perturbations costs one contraction each).
        dict(name="chi_bwd_fp16x2_n4096_l4", op="chi", inp="rod", n=4096, mode="fp16x2", batch=4,
             diag=True, direction="backward"),
        # The flagship solve: density and adjoint susceptibility at N = 16384, X_n kept
        # every 4 steps.
        dict(name="solve_fp16x2_n16384", op="chi", inp="rod", n=16384, mode="fp16x2", batch=1,
             diag=True, direction="backward"),
        # Finite-temperature density and canonical responses of a gapless system.
        dict(name="fermi_fp16x2_n2048_k4", op="fermi", inp="metal", n=2048, mode="fp16x2",
             batch=4),
        # Self-consistent site-charge response of 16 external fields, FP64, linear mixing.
        dict(name="scf_fp64_n256_f16", op="scf", inp="rod", n=256, mode="fp64", batch=16),
        # Thresholded block-sparse density of a long rod.
        dict(name="sparse_fp16x2_n8192", op="sparse", inp="rod", n=8192, mode="fp16x2"),
        # Contractions of 4 susceptibilities with 64 dense perturbations.
        dict(name="contract_fp32_n4096_l4_k64", op="contract", n=4096, rows=4, batch=64,
             mode="fp32"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges."""
    kind = rng.randrange(12)
    split = rng.choice(["bf16x2", "fp16x2", "bf16x3"])
    if kind == 0:
        return dict(op="density", inp="spectrum", n=_logint(rng, 64, 700), mode="fp64")
    if kind == 1:
        return dict(op="chi", inp="spectrum", n=_logint(rng, 200, 1400), mode="fp64", batch=1,
                    diag=False, direction=rng.choice(["forward", "backward"]))
    if kind == 2:
        return dict(op="density", inp="rod", n=4 * _logint(rng, 24, 400), mode=split)
    if kind == 3:
        return dict(op="response", inp="rod", n=4 * _logint(rng, 64, 400), mode=split,
                    batch=rng.randint(1, 16), diag=rng.random() < 0.5)
    if kind == 4:
        return dict(op="autograd", inp="rod", n=4 * _logint(rng, 128, 800), mode=split)
    if kind == 5:
        return dict(op="chi", inp="rod", n=4 * _logint(rng, 100, 500), mode="fp32", batch=1,
                    diag=True, direction=rng.choice(["forward", "backward"]))
    if kind == 6:
        return dict(op="chi", inp="rod", n=4 * _logint(rng, 300, 1024), mode="fp16x2",
                    batch=rng.randint(1, 4), diag=True, direction="backward")
    if kind == 7:
        return dict(op="chi", inp="rod", n=4 * _logint(rng, 1024, 3000),
                    mode=rng.choice(["fp16x2", "bf16x3"]), batch=1, diag=True,
                    direction="backward")
    if kind == 8:
        return dict(op="fermi", inp="metal", n=_logint(rng, 300, 2048), mode="fp16x2",
                    batch=rng.randint(1, 4))
    if kind == 9:
        return dict(op="scf", inp="rod", n=4 * _logint(rng, 24, 80), mode="fp64",
                    batch=rng.randint(2, 16))
    if kind == 10:
        return dict(op="sparse", inp="rod", n=4 * _logint(rng, 1000, 2600), mode="fp16x2")
    return dict(op="contract", n=_logint(rng, 700, 4096), rows=rng.randint(1, 4),
                batch=_logint(rng, 4, 64), mode=rng.choice(["fp32", "fp64"]))


# ------------------------------------------------------------------ inputs (FP64, on the GPU)
def _gen(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * (int(seed) + 1) + salt)
    return g


def _u(g, lo, hi, *shape):
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo


def _spectrum(g, n, e):
    q, r = torch.linalg.qr(torch.randn(n, n, generator=g, device="cuda", dtype=torch.float64))
    q = q * torch.sign(torch.diagonal(r))
    h = (q * e) @ q.T
    return 0.5 * (h + h.T)


def _sym(g, n, batch, dtype):
    """`batch` symmetric matrices with entries of variance 1/n."""
    out = torch.empty(batch, n, n, device="cuda", dtype=dtype)
    for b in range(batch):
        a = torch.randn(n, n, generator=g, device="cuda", dtype=dtype) / math.sqrt(n)
        u = torch.triu(a)
        out[b] = u + torch.triu(u, 1).T
    return out


def _rod(g, n):
    """Gapped tight-binding rod: H (n x n, FP64) and the site coordinates."""
    ns = n // NORB
    box = torch.tensor([ns / (DENSITY * WIDTH * WIDTH), WIDTH, WIDTH], device="cuda",
                       dtype=torch.float64)
    pos = _u(g, 0.0, 1.0, ns, 3) * box
    pos = pos[torch.argsort(pos[:, 0])]
    r2 = torch.zeros(ns, ns, device="cuda", dtype=torch.float64)
    for k in range(3):
        d = pos[:, None, k] - pos[None, :, k]
        d -= box[k] * torch.round(d / box[k])
        r2 += d * d
    r = torch.sqrt(r2)
    t = torch.where(r < RCUT, -torch.exp(-r / DECAY), torch.zeros_like(r))
    t.fill_diagonal_(0.0)
    h = t.repeat_interleave(NORB, 0).repeat_interleave(NORB, 1)
    onsite = _u(g, -0.3, 0.3, n) + 2.0 * (1.0 - 2.0 * (torch.arange(n, device="cuda") % 2))
    h.diagonal().add_(onsite)
    return h, pos, r


def _hamiltonian(case, seed):
    """(H in FP64 rounded to the case's input type, number of occupied states, extras)."""
    n = case["n"]
    g = _gen(seed)
    if case["inp"] == "rod":
        h, pos, r = _rod(g, n)
        return h.to(_dtype(case)), n // 2, (pos, r)
    if case["inp"] == "spectrum":
        nocc = n // 2
        e = torch.cat([_u(g, -1.0, -0.2, nocc), _u(g, 0.2, 1.0, n - nocc)])
    else:
        nocc, e = n // 2, _u(g, -1.0, 1.0, n)
    return _spectrum(g, n, e).to(_dtype(case)), nocc, None


def _dtype(case):
    return torch.float64 if case["mode"] == "fp64" else torch.float32


def _operators(case, seed, extra):
    """The batch of observables or perturbations, (batch, n, n) or diagonals (batch, n)."""
    n, batch, dt = case["n"], case.get("batch", 1), _dtype(case)
    g = _gen(seed, 17)
    if not case.get("diag", False):
        return _sym(g, n, batch, dt)
    if case["op"] == "response":   # site potentials, shared by a site's orbitals
        return _u(g, -1.0, 1.0, batch, n // NORB).repeat_interleave(NORB, 1).to(dt).contiguous()
    pos = extra[0]                 # x, y, z of each orbital's site, then one site's population
    c = (pos - pos.mean(0)).T.repeat_interleave(NORB, 1)
    pop = torch.zeros(1, n, device="cuda", dtype=torch.float64)
    pop[0, :NORB] = 1.0
    return torch.cat([c, pop])[:batch].to(dt).contiguous()


KT, MU = 0.02, 0.0
ALPHA, TOL = 0.7, 1e-6


def _scf_inputs(case, seed, r):
    """Site-site kernel 1/sqrt(r^2+1) and the external site fields, FP64."""
    g = _gen(seed, 29)
    kern = 1.0 / torch.sqrt(r * r + 1.0)
    v = 0.1 * torch.randn(case["batch"], case["n"] // NORB, generator=g, device="cuda",
                          dtype=torch.float64)
    return kern.contiguous(), v


def prepare(case, seed):
    s = dict(case=case)
    if case["op"] == "contract":
        g = _gen(seed)
        n, dt = case["n"], _dtype(case)
        s["P"] = torch.randn(case["rows"], n, n, generator=g, device="cuda", dtype=dt)
        s["Q"] = torch.randn(case["batch"], n, n, generator=g, device="cuda", dtype=dt)
        s["handle"] = sp2.Handle()
        return s
    h, s["nocc"], extra = _hamiltonian(case, seed)
    s["H"] = h.contiguous()
    s["handle"] = sp2.Handle()
    s["tol"] = 1e-10 if case["mode"] == "fp64" else 0.0
    if case["op"] in ("chi", "response", "autograd", "fermi"):
        s["B"] = _operators(case, seed, extra)
    if case["op"] == "scf":
        s["K"], s["V"] = _scf_inputs(case, seed, extra[1])
    return s


def run(s):
    case, h, mode, hd = s["case"], s.get("H"), s["case"]["mode"], s["handle"]
    op = case["op"]
    if op == "contract":
        return sp2.response_contract(s["P"], s["Q"], handle=hd)
    if op == "density":
        d, _ = sp2.sp2_density(h, s["nocc"], mode=mode, idem_tol=s["tol"], handle=hd)
        return d
    if op == "sparse":
        d, _ = sp2.sp2_density(h, s["nocc"], mode=mode, block_tau=1e-5, handle=hd)
        return d
    if op == "chi":
        chi, d, _ = sp2.sp2_susceptibility(h, s["nocc"], s["B"], direction=case["direction"],
                                           diag_only=case["diag"], mode=mode, want_density=True,
                                           idem_tol=s["tol"], handle=hd)
        return chi, d
    if op == "response":
        d1, d, _ = sp2.sp2_response(h, s["nocc"], s["B"], diag_only=case["diag"], mode=mode,
                                    want_density=True, handle=hd)
        return d1, d
    if op == "autograd":
        x = h.detach().requires_grad_(True)
        d = sp2.sp2_density_autograd(x, s["nocc"], mode=mode, handle=hd)
        loss = (s["B"][0] * d).sum()
        (grad,) = torch.autograd.grad(loss, x)
        return d.detach(), grad
    if op == "fermi":
        d1, d, _ = sp2.sp2_fermi(h, MU, KT, s["B"], mode=mode, handle=hd)
        return d1, d
    q, _, _, _ = sp2.sp2_scf_response(h, s["nocc"], NORB, s["K"], s["V"], mixer="linear",
                                      alpha=ALPHA, tol=TOL, mode=mode, handle=hd)
    return q


# ------------------------------------------------------------------ necessary work
def work(case):
    """Inputs read and outputs written once; the products of the recursion (the upper
    triangle of each square, the whole of each response product), three tensor-core
    products per split product (six with three planes)."""
    n, op, b = float(case["n"]), case["op"], float(case.get("batch", 1))
    el = 8.0 if case["mode"] == "fp64" else 4.0
    if op == "contract":
        r = float(case["rows"])
        return dict(bytes=(r + b) * n * n * el + 8.0 * r * b, flops=2.0 * r * b * n * n)
    terms = {"fp64": 1.0, "fp32": 1.0, "bf16x3": 6.0}.get(case["mode"], 3.0)
    m = 24.0                                 # SP2 steps of these gaps
    square, prod = n ** 3 * terms, 2.0 * n ** 3 * terms
    bvals = b * n * (1.0 if case.get("diag") else n)
    if op == "sparse":                       # the blocks near the diagonal
        return dict(bytes=2.0 * n * n * el, flops=m * n * terms * 2.0 * (6 * 256.0) ** 2)
    if op == "density":
        return dict(bytes=2.0 * n * n * el, flops=m * square)
    if op == "scf":
        f = 12.0 * (m * square + b * m * prod)
        return dict(bytes=(n * n + (n / NORB) ** 2 + 2.0 * b * n / NORB) * 8.0, flops=f)
    if op == "fermi":                        # 20 doublings; 2 + 4 products each, 5 per response
        return dict(bytes=(2.0 * n * n + 2.0 * bvals) * el, flops=20.0 * (6.0 + 5.0 * b) * prod)
    out = b * n * n + n * n
    return dict(bytes=(n * n + bvals + out) * el, flops=m * square + b * m * prod)


# ------------------------------------------------------------------ exact results
def _rotate(v, w):
    return v @ w @ v.T


def exact(case, seed):
    op, n = case["op"], case["n"]
    if op == "contract":
        s = prepare(case, seed)
        p = s["P"].reshape(case["rows"], -1).double()
        return torch.stack([p @ q.reshape(-1).double() for q in s["Q"]], 1)
    if n > MAX_EXACT_N:
        return None
    h, nocc, extra = _hamiltonian(case, seed)
    e, v = torch.linalg.eigh(h.double())
    if op == "fermi":
        x = (e - MU) / KT
        f = torch.sigmoid(-x)
        # divided differences of f, from sinh to keep near pairs accurate:
        # (f_i - f_j) / (e_i - e_j) = -sinh(u) / (u kT) / (4 cosh(x_i/2) cosh(x_j/2)), u = (x_i-x_j)/2
        u = 0.5 * (x[:, None] - x[None, :])
        small = u.abs() < 1e-4
        us = torch.where(small, torch.ones_like(u), u)
        # sinh(u) / (cosh(x_i/2) cosh(x_j/2)) = tanh(x_i/2) - tanh(x_j/2)
        t = torch.tanh(0.5 * x)
        c = 1.0 / torch.cosh(0.5 * x)
        dd = torch.where(small, (1.0 + u * u / 6.0) * c[:, None] * c[None, :],
                         (t[:, None] - t[None, :]) / us) * (-0.25 / KT)
        ri = torch.diagonal(dd)                      # response to the identity, diagonal in V
        b = _operators(case, seed, extra).double()
        outs = []
        for k in range(b.shape[0]):
            w = dd * (v.T @ b[k] @ v)
            w = w - torch.diag(ri * (torch.diagonal(w).sum() / ri.sum()))
            outs.append(_rotate(v, w))
        return torch.stack(outs), (v * f) @ v.T
    vo = v[:, :nocc]
    dm = vo @ vo.T
    if op in ("density", "sparse"):
        return dm
    vv = v[:, nocc:]
    den = 1.0 / (e[:nocc, None] - e[None, nocc:])     # (f_i - f_a) / (e_i - e_a)
    if op == "scf":
        kern, vext = _scf_inputs(case, seed, extra[1])
        ns = n // NORB
        # site susceptibility: charges of the response to a unit potential on each site
        chi = torch.empty(ns, ns, device="cuda", dtype=torch.float64)
        for a in range(ns):
            rows = slice(a * NORB, (a + 1) * NORB)
            w = den * (vo[rows].T @ vv[rows])
            chi[:, a] = 2.0 * ((vo @ w) * vv).sum(1).reshape(ns, NORB).sum(1)
        q = torch.zeros_like(vext)
        norm0 = None
        for _ in range(100):
            qo = (vext + q @ kern.T) @ chi.T
            r = qo - q
            norm0 = qo.norm() if norm0 is None else norm0
            if (r.norm() / norm0).item() <= TOL:
                break
            q = q + ALPHA * r
        return q
    b = _operators(case, seed, extra).double()
    outs = []
    for k in range(b.shape[0]):
        bo = vo.T * b[k] if case.get("diag") else vo.T @ b[k]
        y = (vo @ (den * (bo @ vv))) @ vv.T
        outs.append(y + y.T)
    chi = torch.stack(outs)
    return (dm, chi[0]) if op == "autograd" else (chi, dm)
