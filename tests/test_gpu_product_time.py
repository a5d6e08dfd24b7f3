"""sp2_info.product_ms of FP64 products by digits: the whole product, digits and sums too."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [0, 1])
def test_products_are_most_of_a_solve(batch):
    """A recursion of 20 given steps launches little else than its products (bounds, X_1, the
    copy of the result, once each), so they take most of its time; k_gemm_dig by itself is
    half of a step at this size."""
    import __graft_entry__ as g
    g.build()
    import paper_2409_17033_gb300 as sp2
    n = 1001
    gen = torch.Generator(device="cuda").manual_seed(0)
    H = torch.randn(n, n, generator=gen, device="cuda", dtype=torch.float64) / n
    H = H + H.T
    kw = dict(mode="fp64", sigma=[1, -1] * 10, time_kernels=True, handle=sp2.Handle(), allow_noconv=True)
    best = 0.0
    for _ in range(4):
        t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        torch.cuda.synchronize()
        t0.record()
        if batch:
            info = sp2.sp2_response(H, n // 2, H[None].contiguous(), **kw)[2]
        else:
            info = sp2.sp2_density(H, n // 2, **kw)[1]
        t1.record()
        t1.synchronize()
        assert info["product_launches_timed"] == 20
        best = max(best, info["product_ms"] / t0.elapsed_time(t1))
    assert 0.7 < best <= 1.0
