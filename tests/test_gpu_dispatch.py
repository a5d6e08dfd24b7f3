"""The forms a call's sizes choose between: CUDA-core product tiles, narrow tensor-core
tiles, contraction kernels, and batches of finite-temperature responses, each at the
sizes where it can go wrong."""
import ctypes as C

import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp2():
    import __graft_entry__ as g
    g.build()
    import paper_2409_17033_gb300 as p
    return p


def _sym(n, rng, scale=1.0):
    g = rng.standard_normal((n, n)) * scale
    return g + g.T


# A K-long sum of products in arithmetic of unit roundoff u is off by at most
# (K + 2) u |a| . |b| <= (K + 2) u ||a|| ||b||; the response adds two such sums, and the
# update's own roundings of 4 u of its terms.
@pytest.mark.parametrize("mode,n", [("fp64", 2), ("fp64", 64), ("fp64", 129), ("fp64", 190),
                                    ("fp64", 200), ("fp32", 2), ("fp32", 127), ("fp32", 300),
                                    ("fp32", 700), ("fp32", 1026), ("fp32", 1500)])
@pytest.mark.parametrize("diag", [False, True])
def test_cuda_core_products(sp2, mode, n, diag):
    rng = np.random.default_rng(n)
    dt = np.float64 if mode == "fp64" else np.float32
    u = 2.0 ** -53 if mode == "fp64" else 2.0 ** -24
    h = _sym(n, rng).astype(dt)
    b = np.stack([rng.standard_normal(n) if diag else _sym(n, rng) for _ in range(2)]).astype(dt)
    for sig in (1, -1):
        # bounds (-1, 0): X_1 = -H, Y_1 = -B; one step
        d1, d, _ = sp2.sp2_response(torch.from_numpy(h).cuda(), max(n // 2, 1),
                                    torch.from_numpy(b).cuda(), diag_only=diag, mode=mode,
                                    sigma=[sig], bounds=(-1.0, 0.0), want_density=True,
                                    handle=sp2.Handle(), allow_noconv=True)
        d1, d = d1.cpu().numpy(), d.cpu().numpy()
        x = -h.astype(np.float64)
        nx = np.linalg.norm(x, axis=1)
        c = x @ x
        ref = c if sig > 0 else 2.0 * x - c
        tol = (2 * n + 6) * u * (nx[:, None] * nx[None, :] + np.abs(x))
        assert np.array_equal(d, d.T) and np.all(np.abs(d - ref) <= tol)
        for k in range(2):
            y = -b[k].astype(np.float64)
            y = np.diag(y) if diag else y
            ny = np.linalg.norm(y, axis=1)
            s = y @ x + x @ y
            ref = s if sig > 0 else 2.0 * y - s
            cross = ny[:, None] * nx[None, :]
            tol = (2 * n + 6) * u * (cross + cross.T + np.abs(y))
            assert np.array_equal(d1[k], d1[k].T) and np.all(np.abs(d1[k] - ref) <= tol)


@pytest.mark.parametrize("mode", ["bf16x2", "fp16x2", "bf16x3"])
@pytest.mark.parametrize("n", [96, 256, 300, 770, 1030])
def test_narrow_tiles_keep_the_bits(sp2, mode, n):
    """Tiles of a CTA pair as narrow as the size makes them against 128 x 256 tiles of
    one SM: the same arithmetic per entry, so the same bits. The recursion's branches are
    given, since the traces' sums depend on the tiles in their last bits."""
    p = workloads.random_spectrum(n, nocc=n // 2, k=2, seed=n)
    H = torch.from_numpy(p.H.astype(np.float32)).cuda()
    B = torch.from_numpy(p.H1[:2].astype(np.float32)).cuda()
    out = []
    for pair in (1, 0):
        h = sp2.Handle()
        h.set_option("pair_tiles", pair)
        d1, d, _ = sp2.sp2_response(H, p.nocc, B, mode=mode, sigma=[1, -1, -1, 1, 1],
                                    want_density=True, handle=h, allow_noconv=True)
        out.append((d1.clone(), d.clone()))
    assert torch.equal(out[0][1], out[1][1]) and torch.equal(out[0][0], out[1][0])


# FP32 entries' products are summed exactly up to 2^-40 of their magnitudes (bound
# 1e-12), FP64 ones by a fused multiply-add each over at most N^2 terms.
@pytest.mark.parametrize("L,K,n,shift", [(1, 1, 1, 0), (1, 8, 64, 0), (2, 9, 65, 0), (3, 8, 64, 0),
                                         (3, 7, 130, 0), (5, 17, 101, 0), (4, 16, 96, 1),
                                         (9, 3, 66, 0)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_contraction_forms(sp2, L, K, n, shift, dtype):
    g = torch.Generator().manual_seed(L * 100 + K)
    def make(rows):   # shift: the matrices do not start on a 16-byte boundary
        buf = torch.empty(rows * n * n + shift, dtype=dtype, device="cuda")
        v = buf[shift:].view(rows, n, n)
        v.copy_(torch.randn(rows, n, n, generator=g, dtype=torch.float64))
        return v
    P, Q = make(L), make(K)
    out = sp2.response_contract(P, Q, handle=sp2.Handle()).cpu().numpy()
    p, q = P.double().cpu().numpy().reshape(L, -1), Q.double().cpu().numpy().reshape(K, -1)
    ref = (p.astype(np.longdouble) @ q.astype(np.longdouble).T)
    mag = np.abs(p) @ np.abs(q).T
    tol = (1e-12 if dtype == torch.float32 else (n * n + 40) * 2.0 ** -53) * mag
    assert np.all(np.abs(out - ref).astype(float) <= tol)


def test_contraction_in_a_graph(sp2):
    """The allocation-free contraction captured behind a copy and a kernel, replayed on
    other inputs."""
    from paper_2409_17033_gb300 import _lib
    lib = _lib.load()
    P = torch.randn(3, 96, 96, device="cuda")
    Q = torch.randn(9, 96, 96, device="cuda")
    src = torch.randn_like(Q)
    out = torch.zeros(3, 9, dtype=torch.float64, device="cuda")

    def call(stream):
        return lib.response_contract_noalloc(
            C.c_void_p(P.data_ptr()), 3, C.c_void_p(Q.data_ptr()), 9, 96, 1, 0,
            C.c_void_p(out.data_ptr()), C.c_void_p(stream.cuda_stream))
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        assert call(s) == 0
        P.mul_(1.0)
    s.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        Q.copy_(src)
        assert call(torch.cuda.current_stream()) == 0
        P.mul_(2.0)
        assert call(torch.cuda.current_stream()) == 0
    for _ in range(2):
        src.normal_()
        p0 = P.double()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        ref = torch.einsum("lij,kij->lk", 2.0 * p0, src.double())
        assert torch.allclose(out, ref, rtol=1e-11, atol=1e-9)


@pytest.mark.parametrize("mode,n,k,diag,canonical,limit", [
    ("fp16x2", 96, 1, False, True, 0), ("fp16x2", 300, 5, True, True, 0),
    ("fp16x2", 300, 5, False, True, 160 << 20), ("fp16x2", 301, 3, False, False, 0),
    ("bf16x2", 513, 3, False, True, 0), ("bf16x3", 300, 2, True, False, 0),
    ("fp32", 130, 3, False, True, 0), ("fp64", 100, 4, True, True, 0),
    ("fp64", 300, 3, False, True, 0), ("fp64", 300, 3, False, True, 200 << 20)])
def test_fermi_batches(sp2, mode, n, k, diag, canonical, limit):
    """Responses computed as a batch against one perturbation at a time: the same
    arithmetic per entry (FP64: the same error-free products, or sums in another order,
    whose rounding the doublings carry: 1e-10)."""
    rng = np.random.default_rng(n)
    dt = torch.float64 if mode == "fp64" else torch.float32
    H = torch.from_numpy(_sym(n, rng, 0.3 / np.sqrt(n))).to(dt).cuda()
    b = rng.standard_normal((k, n)) if diag else np.stack([_sym(n, rng) for _ in range(k)])
    b *= 10.0 ** (2 * np.arange(k)).reshape((k,) + (1,) * (b.ndim - 1))
    B = torch.from_numpy(b).to(dt).cuda()
    kw = dict(diag_only=diag, canonical=canonical, mode=mode, n_doublings=12)
    h = sp2.Handle(limit) if limit else sp2.Handle()
    D1, D, _ = sp2.sp2_fermi(H, 0.05, 0.1, B, handle=h, **kw)
    one = sp2.Handle()
    for i in range(k):
        r, d, _ = sp2.sp2_fermi(H, 0.05, 0.1, B[i:i + 1].contiguous(), handle=one, **kw)
        assert torch.equal(D, d)
        assert (torch.equal(D1[i], D1[i].T) if mode != "fp64" else True)
        if mode == "fp64":
            assert (D1[i] - r[0]).norm() <= 1e-10 * r[0].norm()
        else:
            assert torch.equal(D1[i], r[0])


@pytest.mark.parametrize("n,batch,diag", [(200, 1, False), (256, 2, True), (257, 1, False),
                                          (300, 4, True), (600, 2, False)])
def test_fp64_step_in_one_launch(sp2, n, batch, diag):
    """Both products of a step in one launch against the same products apart (a square
    without responses): the same integers, so the same bits from np = 512 on, where both
    sides use them; and against the recursion in FP64 sums."""
    p = workloads.random_spectrum(n, nocc=n // 2, k=batch, seed=n)
    H = torch.from_numpy(np.ascontiguousarray(p.H)).cuda()
    b = np.stack([np.diag(p.H1[i]) if diag else p.H1[i] for i in range(batch)])
    B = torch.from_numpy(np.ascontiguousarray(b)).cuda()
    kw = dict(mode="fp64", sigma=[1, -1, -1, 1], allow_noconv=True)
    d1, d, _ = sp2.sp2_response(H, p.nocc, B, diag_only=diag, want_density=True,
                                handle=sp2.Handle(), **kw)
    dens, _ = sp2.sp2_density(H, p.nocc, handle=sp2.Handle(), **kw)
    if n > 256:
        assert torch.equal(d, dens)
    # the recursion's four steps in FP64 sums
    _, info = sp2.sp2_density(H, p.nocc, handle=sp2.Handle(), **kw)
    x = info["alpha"] * np.eye(n) + info["beta"] * p.H
    ys = [info["beta"] * (np.diag(v) if diag else v) for v in b]
    for s in (1, -1, -1, 1):
        ys = [(y @ x + x @ y) if s > 0 else 2.0 * y - (y @ x + x @ y) for y in ys]
        x = x @ x if s > 0 else 2.0 * x - x @ x
    # each step rounds sums of n products of entries' row and column norms (at most 1
    # for X, ||Y||_F for Y) and doubles what came before
    u = 64.0 * (n + 4) * 2.0 ** -53
    assert np.abs(d.cpu().numpy() - x).max() <= u
    for k in range(batch):
        y0 = np.linalg.norm(info["beta"] * b[k])
        assert np.abs(d1[k].cpu().numpy() - ys[k]).max() <= u * 16.0 * y0


@pytest.mark.parametrize("n", [33, 128, 129, 190])
def test_fp64_floor_candidate(sp2, n):
    """The recursion run to its precision floor returns the kept candidate (X_n kept by
    the square's last block up to np = 128, by a copy kernel above)."""
    p = workloads.random_spectrum(n, nocc=n // 2, k=1, seed=n)
    H = torch.from_numpy(np.ascontiguousarray(p.H)).cuda()
    D, info = sp2.sp2_density(H, p.nocc, mode="fp64", handle=sp2.Handle())
    e, v = np.linalg.eigh(p.H)
    ref = v[:, :p.nocc] @ v[:, :p.nocc].T
    D = D.cpu().numpy()
    # N-long FP64 sums through some 30 steps, each at most doubling an error off the gap
    assert info["converged"] and np.linalg.norm(D - ref) <= 1e-10 * np.sqrt(n)
    assert np.linalg.norm(D @ D - D) <= 1e-11 * np.sqrt(n)


@pytest.mark.parametrize("mode", ["fp32", "bf16x2", "bf16x3", "fp16x2"])
@pytest.mark.parametrize("n", [60, 64, 300, 301])
def test_dense_incoming_gradient(sp2, mode, n):
    """The adjoint takes the symmetric part of a dense gradient, rounded once from its
    exact value: the same result as from that part itself."""
    p = workloads.random_spectrum(n, nocc=n // 2, k=1, seed=n)
    H = torch.from_numpy(p.H.astype(np.float32)).cuda()
    g = torch.Generator().manual_seed(n)
    W = torch.randn(n, n, generator=g).cuda()
    half = 0.5 * (W.double() + W.double().T)
    out = []
    for w in (W, half.float()):
        x = H.clone().requires_grad_(True)
        d = sp2.sp2_density_autograd(x, p.nocc, mode=mode, handle=sp2.Handle())
        (grad,) = torch.autograd.grad((w * d).sum(), x)
        out.append(grad)
    assert torch.equal(out[0], out[1]) and out[0].abs().max() > 0


@pytest.mark.parametrize("L,K,n,shift", [(1, 1, 45, 0), (2, 2, 33, 0), (5, 3, 77, 0), (7, 5, 131, 0),
                                         (1, 6, 65, 1), (6, 7, 32, 1), (3, 15, 91, 0), (8, 4, 37, 0),
                                         (1, 23, 701, 0), (5, 12, 701, 0), (3, 17, 702, 1)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_contraction_remainders(sp2, L, K, n, shift, dtype):
    """Every count of perturbations and rows that a block can be left with, of matrices on
    16-byte boundaries and not, N^2 of every remainder: bounds as in test_contraction_forms."""
    test_contraction_forms(sp2, L, K, n, shift, dtype)


@pytest.mark.parametrize("L", [1, 3])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_offset_contractions_cost_what_aligned_ones_do(sp2, L, dtype):
    """The same bytes and operations, with single-entry copies in place of 16-byte ones
    (4 or 2 times their number, beside 16 arithmetic operations or more per entry): less
    than twice the time. The best of several runs of each, in turn."""
    n, K = 2000, 40
    h = sp2.Handle()
    def make(rows, shift):
        buf = torch.randn(rows * n * n + 1, dtype=dtype, device="cuda")
        return buf[shift:shift + rows * n * n].view(rows, n, n)
    forms = [(make(L, s), make(K, s)) for s in (0, 1)]
    best = [float("inf")] * 2
    for _ in range(6):
        for i, (P, Q) in enumerate(forms):
            t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            sp2.response_contract(P, Q, handle=h)
            t0.record()
            for _ in range(4):
                sp2.response_contract(P, Q, handle=h)
            t1.record()
            t1.synchronize()
            best[i] = min(best[i], t0.elapsed_time(t1))
    assert best[1] <= 2.0 * best[0]
