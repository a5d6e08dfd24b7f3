"""FP64 products by digits where the result is known exactly: small integers (every digit
pair that is not zero is formed, so the products must be equal bit for bit), and K axes at
and above 8192, the longest that one 32-bit sum of eight digit pairs spans."""
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")
import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp2():
    import __graft_entry__ as g
    g.build()
    import paper_2409_17033_gb300 as m
    return m


def _integers(n, seed, top=1000):
    h = np.random.default_rng(seed).integers(-top, top + 1, (n, n))
    return np.triu(h) + np.triu(h, 1).T


@pytest.mark.parametrize("n", [257, 300, 511, 768, 1100, 2100, 8192, 8200])
def test_integer_square(sp2, n):
    """Entries of 10 bits stand in the first three digits of a row's scale (2^24 at most):
    pairs of weight 5 at most, sums below 2^53."""
    h = _integers(n, n)
    D, _ = sp2.sp2_density(torch.from_numpy(h.astype(float)).cuda(), n // 2, mode="fp64", sigma=[1],
                           bounds=(-1.0, 0.0), handle=sp2.Handle(), allow_noconv=True)   # X_1 = -H
    rows = np.unique(np.linspace(0, n - 1, 7).astype(int))
    got = D[torch.from_numpy(rows).cuda()].cpu().numpy()
    assert np.array_equal(got, (h[rows] @ h).astype(float))
    assert torch.equal(D, D.T)


@pytest.mark.parametrize("n,batch,sig", [(256, 3, 1), (300, 1, -1), (300, 4, 1), (700, 2, -1), (1100, 5, 1)])
def test_integer_response(sp2, n, batch, sig):
    h = _integers(n, n)
    b = np.stack([_integers(n, n + 1 + k, 10 ** (k % 3 + 1)) for k in range(batch)])
    D1, D, _ = sp2.sp2_response(torch.from_numpy(h.astype(float)).cuda(), n // 2,
                                torch.from_numpy(b.astype(float)).cuda(), mode="fp64", sigma=[sig],
                                bounds=(-1.0, 0.0), want_density=True, handle=sp2.Handle(), allow_noconv=True)
    rows = np.unique(np.linspace(0, n - 1, 7).astype(int))
    x, xr = -h, -h[rows]
    sq = xr @ x
    assert np.array_equal(D.cpu().numpy()[rows], (sq if sig > 0 else 2 * xr - sq).astype(float))
    for k in range(batch):
        y = -b[k]
        s = y[rows] @ x + xr @ y        # symmetric factors: (Y X + X Y)_r
        want = s if sig > 0 else 2 * y[rows] - s
        assert np.array_equal(D1[k].cpu().numpy()[rows], want.astype(float))


@pytest.mark.parametrize("n", [8192, 8193])
@pytest.mark.parametrize("shift", range(8))
def test_largest_sums_of_one_sign(sp2, n, shift):
    """Entries alike of six bytes 0x7f, at every place against the row's scale: where bytes and
    digits meet, six digits of 127, the largest sums of one sign that an FP64 entry gives
    (a sum past 32 bits at the last weight would be an error of 2^-38 u^2). Tolerance: seven
    pairs of weight 8 dropped, K 2^14 each, of 2^64 u^2; half a unit of each factor entry's
    and of the last weight's rounding; one FP64 rounding; u <= 2 (1 + 2^-6) ||row||."""
    v = float(0x7f7f7f7f7f7f) * 2.0 ** (shift - 47)
    H = torch.full((n, n), v, dtype=torch.float64, device="cuda")
    D, _ = sp2.sp2_density(H, n // 2, mode="fp64", sigma=[1], bounds=(-1.0, 0.0), handle=sp2.Handle(),
                           allow_noconv=True)
    exact = Fraction(v) ** 2 * n
    u2 = 4.13 * n * v * v
    tol = (7.0 * n * 2.0 ** 14 * 2.0 ** 48 / 2.0 ** 126 + (2.0 * n ** 0.5 + 28.0) * 2.0 ** -64) * u2
    tol += 2.0 ** -53 * float(exact)
    lo, hi = float(D.min()), float(D.max())
    assert max(abs(float(Fraction(lo) - exact)), abs(float(Fraction(hi) - exact))) <= tol


@pytest.mark.parametrize("n", [33, 64, 128, 129, 190])
def test_kept_candidate_is_the_iterate(sp2, n):
    """Where the stop at the precision floor goes back (more squares than steps of the
    result), the result is the kept X_{M+1}: what the same branches give as fixed steps."""
    for seed in range(12):
        p = workloads.random_spectrum(n, nocc=n // 2, k=1, seed=100 * n + seed)
        H = torch.from_numpy(np.ascontiguousarray(p.H)).cuda()
        D, info = sp2.sp2_density(H, p.nocc, mode="fp64", handle=sp2.Handle())
        m = info["M"]
        if info["n_gemm_launches"] > m:
            break
    else:
        pytest.fail("no recursion went back")
    want, _ = sp2.sp2_density(H, p.nocc, mode="fp64", sigma=list(info["sigma"])[:m], handle=sp2.Handle(),
                              allow_noconv=True)
    assert torch.equal(D, want)


@pytest.mark.parametrize("n,canonical", [(60, True), (200, False), (300, True), (520, True)])
def test_fp64_finite_t_responses_are_symmetric(sp2, n, canonical):
    """The update adds entry pairs in one order for both, in FP64 as in FP32."""
    rng = np.random.default_rng(n)
    h = rng.standard_normal((n, n)) * 0.2 / np.sqrt(n)
    b = rng.standard_normal((3, n, n))
    D1, D, _ = sp2.sp2_fermi(torch.from_numpy(h + h.T).cuda(), 0.05, 0.1,
                             torch.from_numpy(b + b.transpose(0, 2, 1)).cuda(), canonical=canonical,
                             mode="fp64", n_doublings=12, handle=sp2.Handle())
    assert torch.equal(D, D.T)
    for k in range(3):
        assert torch.equal(D1[k], D1[k].T)
