"""A call on a stream that other work keeps busy: the end of its recursion is learned from
its own work, not from the stream falling idle."""
import threading
import time

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp2():
    import __graft_entry__ as g
    g.build()
    import paper_2409_17033_gb300 as m
    return m


@pytest.mark.parametrize("mode", ["fp64", "fp16x2"])
@pytest.mark.parametrize("bad", [False, True])
def test_call_returns_beside_other_work(sp2, mode, bad):
    """Another thread keeps the stream busy with kernels of some milliseconds for at most
    eight seconds, two of them enqueued at a time. A solve returns in between, one whose H
    is not finite (no step of it runs) with its error."""
    n = 200
    H = torch.randn(n, n, dtype=torch.float64 if mode == "fp64" else torch.float32, device="cuda")
    H = H + H.T
    sp2.sp2_density(H, n // 2, mode=mode, handle=sp2.Handle(), allow_noconv=True)   # kernels loaded
    if bad:
        H[3, 5] = H[5, 3] = float("nan")
    s = torch.cuda.Stream()
    started, stop = threading.Event(), threading.Event()

    def busy():
        ends = []
        t0 = time.monotonic()
        with torch.cuda.stream(s):
            while not stop.is_set() and time.monotonic() - t0 < 8.0:
                torch.cuda._sleep(10_000_000)
                ends.append(torch.cuda.Event())
                ends[-1].record()
                if len(ends) > 2:
                    ends.pop(0).synchronize()
                    started.set()

    torch.cuda.synchronize()
    t = threading.Thread(target=busy)
    with torch.cuda.stream(s):
        h = sp2.Handle()
        t.start()
        try:
            assert started.wait(5.0)
            if bad:
                with pytest.raises(sp2.SP2Error):
                    sp2.sp2_density(H, n // 2, mode=mode, handle=h, sync=False)
            else:
                sp2.sp2_density(H, n // 2, mode=mode, handle=h, sync=False, allow_noconv=True)
            assert t.is_alive()
        finally:
            stop.set()
            t.join()
    torch.cuda.synchronize()
