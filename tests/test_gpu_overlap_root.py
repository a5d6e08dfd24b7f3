"""The inverse square root of an overlap matrix in FP64 (Loewdin factor), to the accuracy of
its converged iteration for every input: the density in the atomic-orbital representation
against the eigendecomposition."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _spectrum(n, seed):
    rng = np.random.default_rng(seed)
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    e = np.concatenate([rng.uniform(-1, -.2, n // 2), rng.uniform(.2, 1, n - n // 2)])
    h = (q * e) @ q.T
    return 0.5 * (h + h.T)


@pytest.mark.parametrize("n,seed", [(60, 1), (256, 2), (300, 0), (520, 0), (520, 10), (700, 0), (700, 10),
                                    (1100, 0)])
def test_converged_root(n, seed):
    """Z S Z = I to some N 2^-53 of rounding, through three products with cond(S) = 1.5; an
    iteration stopped one step early leaves 1e-11 and more (quadratic convergence from
    residuals of 1e-5 on)."""
    import __graft_entry__ as g
    g.build()
    import paper_2409_17033_gb300 as sp2
    h, s, a = _spectrum(n, seed), np.eye(n) + 0.2 * _spectrum(n, seed + 5), _spectrum(n, seed + 1)
    H, S, A = (torch.from_numpy(x).cuda() for x in (h, s, a))
    D, _, _, Z, _ = sp2.sp2_nonorth_susceptibility(H, S, n // 2, A, mode="fp64", want_z=True,
                                                   idem_tol=1e-10, handle=sp2.Handle())
    z = Z.cpu().numpy()
    assert np.linalg.norm(z @ s @ z - np.eye(n)) <= 8.0 * n * 2.0 ** -53 * np.sqrt(n)
    es, vs = np.linalg.eigh(s)
    zr = (vs / np.sqrt(es)) @ vs.T
    e, v = np.linalg.eigh(zr @ h @ zr)
    vo = zr @ v[:, :n // 2]
    ref = vo @ vo.T
    assert np.linalg.norm(D.cpu().numpy() - ref) <= 1e-12 * np.linalg.norm(ref)
