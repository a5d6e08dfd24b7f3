"""FP64 products by digits on the tensor cores (csrc/gemm_dig.cu): one square and one
response step against extended precision on sampled rows, at the sizes and values
where the digit arithmetic can go wrong.

Tolerance. With u_i = 2^ex_i <= 2 ||a_i|| (1 + 2^-6), an entry of a K-long product
drops digit pairs of weight s >= 8, at most 7 K 2^14 2^48 (and a hundredth of that
for s > 8) of 2^126 u_i u_j, and rounds each factor entry to 2^-64 of u (together
at most 2 sqrt(K) 2^-64 u_i u_j) and the last weight's sums to 2^-63: together below
(6.2 K + 2 sqrt(K) + 28) 2^-63 u_i u_j (the bound of 7 digits of 9 bits, which the
tests keep), plus one FP64 rounding of the result (and of each sum of the response
update)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _bound(k, a, b):
    u = 4.1 * a[:, None] * b[None, :]
    return (6.2 * k + 2.0 * np.sqrt(k) + 28.0) * 2.0 ** -63 * u


def _matrix(kind, n, rng):
    if kind == "normal":
        g = rng.standard_normal((n, n))
        return g + g.T
    if kind == "constant":           # every digit of every entry alike: the largest chunk sums
        return np.full((n, n), 0.1)
    if kind == "graded":             # rows and columns from 2^-100 to 2^100 (||X_2||_F^2 stays finite), some zero
        g = rng.standard_normal((n, n))
        s = np.exp2(rng.integers(-100, 101, n).astype(float))
        s[:: 17] = 0.0
        return s[:, None] * (g + g.T) * s[None, :]
    g = np.diag(rng.uniform(0.5, 1.0, n))   # a dominant diagonal beside small couplings
    c = rng.standard_normal((n, n)) * 1e-9
    return g + c + c.T


@pytest.mark.parametrize("n,kind", [(256, "normal"), (257, "constant"), (300, "graded"),
                                    (511, "diagonal"), (768, "normal"), (1100, "constant"),
                                    (4352, "constant")])
def test_square(n, kind):
    import torch
    from paper_2409_17033_gb300 import Handle, sp2_density
    h = _matrix(kind, n, np.random.default_rng(n))
    H = torch.from_numpy(h).cuda()
    # bounds (-1, 0): X_1 = -H; one square: H^2
    D, _ = sp2_density(H, n // 2, mode="fp64", sigma=[1], bounds=(-1.0, 0.0), handle=Handle(),
                       allow_noconv=True)
    D = D.cpu().numpy()
    assert np.array_equal(D, D.T)
    rows = np.unique(np.linspace(0, n - 1, 6).astype(int))
    hl = h.astype(np.longdouble)
    ref = np.stack([(hl[r][None, :] * hl).sum(1) for r in rows])
    nrm = np.sqrt(np.einsum("ij,ij->i", h, h))
    tol = _bound(n, nrm[rows], nrm) + 2.0 ** -53 * np.abs(ref.astype(float))
    assert np.all(np.abs(D[rows] - ref).astype(float) <= tol)


@pytest.mark.parametrize("n,batch,sig", [(256, 1, 1), (300, 3, -1), (640, 5, 1)])
def test_response(n, batch, sig):
    import torch
    from paper_2409_17033_gb300 import Handle, sp2_response
    rng = np.random.default_rng(n)
    h = _matrix("normal", n, rng)
    b = np.stack([_matrix("normal", n, rng) * 10.0 ** (3 * k) for k in range(batch)])
    D1, _, _ = sp2_response(torch.from_numpy(h).cuda(), n // 2, torch.from_numpy(b).cuda(),
                            mode="fp64", sigma=[sig], bounds=(-1.0, 0.0), handle=Handle(),
                            allow_noconv=True)
    D1 = D1.cpu().numpy()
    x, y = -h, -b
    xl = x.astype(np.longdouble)
    nx = np.sqrt(np.einsum("ij,ij->i", x, x))
    rows = np.unique(np.linspace(0, n - 1, 5).astype(int))
    for k in range(batch):
        assert np.array_equal(D1[k], D1[k].T)
        yl = y[k].astype(np.longdouble)
        ny = np.sqrt(np.einsum("ij,ij->i", y[k], y[k]))
        z = np.stack([(yl[r][None, :] * xl).sum(1) for r in rows])        # (Y X)_rj
        zt = np.stack([(yl * xl[r][None, :]).sum(1) for r in rows])       # (Y X)_jr
        s = z + zt
        ref = s if sig > 0 else 2.0 * yl[rows] - s
        tol = _bound(n, ny[rows], nx) + _bound(n, nx[rows], ny)
        tol = tol + 2.0 ** -52 * (np.abs(z) + np.abs(zt) + 2.0 * np.abs(y[k][rows])).astype(float)
        assert np.all(np.abs(D1[k][rows] - ref).astype(float) <= tol)


def test_nonfinite_response():
    """A NaN in a perturbation reaches the rows it reached as an FP64 sum would."""
    import torch
    from paper_2409_17033_gb300 import Handle, sp2_response
    n = 300
    rng = np.random.default_rng(0)
    h = _matrix("normal", n, rng)
    b = np.stack([_matrix("normal", n, rng)] * 2)
    b[1, 7, 7] = np.nan
    D1, _, _ = sp2_response(torch.from_numpy(h).cuda(), n // 2, torch.from_numpy(b).cuda(),
                            mode="fp64", sigma=[1], bounds=(-1.0, 0.0), handle=Handle(),
                            allow_noconv=True)
    nan = np.isnan(D1.cpu().numpy())
    want = np.zeros((n, n), bool)
    want[7] = want[:, 7] = True
    assert not nan[0].any() and np.array_equal(nan[1], want)


def test_workspace_limit():
    """A limit that leaves no room for the digits falls back to the CUDA cores."""
    import torch
    from paper_2409_17033_gb300 import Handle, sp2_density
    n = 512
    h = _matrix("normal", n, np.random.default_rng(1))
    h /= np.abs(h).sum(1).max()
    H = torch.from_numpy(h).cuda()
    D, info = sp2_density(H, n // 2, mode="fp64", max_iter=60, handle=Handle(), allow_noconv=True)
    el = 8 * n * n
    D2, info2 = sp2_density(H, n // 2, mode="fp64", max_iter=60, handle=Handle(3 * el + (1 << 20)),
                            allow_noconv=True)
    assert info["M"] > 5 and (D - D2).norm() <= 1e-9 * D.norm()


def test_fermi_products():
    """C = A X (finite-temperature recursion) against the eigendecomposition."""
    import torch
    from paper_2409_17033_gb300 import Handle, sp2_fermi
    n, kt = 300, 0.1
    rng = np.random.default_rng(3)
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    e = rng.uniform(-1.0, 1.0, n)
    h = (q * e) @ q.T
    h = 0.5 * (h + h.T)
    _, D, _ = sp2_fermi(torch.from_numpy(h).cuda(), 0.0, kt, mode="fp64", handle=Handle())
    e, q = np.linalg.eigh(h)
    ref = (q / (1.0 + np.exp(e / kt))) @ q.T
    assert np.linalg.norm(D.cpu().numpy() - ref) <= 1e-10 * np.linalg.norm(ref)
