"""What a handle asks for: limits that hold a call by its least form, what earlier calls
leave, and the optional buffers (digits of FP64 products, batches of responses)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp2():
    import __graft_entry__ as g
    g.build()
    import paper_2409_17033_gb300 as m
    return m


def _gapped(n, seed=0):
    rng = np.random.default_rng(seed)
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    e = np.concatenate([rng.uniform(-1, -.2, n // 2), rng.uniform(.2, 1, n - n // 2)])
    h = (q * e) @ q.T
    return 0.5 * (h + h.T)


def _inputs(n, mode):
    dt = torch.float64 if mode == "fp64" else torch.float32
    H = torch.from_numpy(_gapped(n)).to(dt).cuda()
    return H, torch.from_numpy(np.stack([_gapped(n, s) for s in (1, 2, 3)])).to(dt).cuda()


def _call(sp2, name, n, mode, H, B, handle):
    """One call; its outputs."""
    kw = dict(mode=mode, idem_tol=1e-10 if mode == "fp64" else 0.0, handle=handle)
    if name == "density":
        return sp2.sp2_density(H, n // 2, **kw)[0]
    if name == "response":
        return sp2.sp2_response(H, n // 2, B, **kw)[0]
    if name == "chi":
        return sp2.sp2_susceptibility(H, n // 2, B[:2], direction="backward", **kw)[0]
    if name == "chi_k1":
        return sp2.sp2_susceptibility(H, n // 2, B[:1], direction="backward", ckpt_k=1, **kw)[0]
    if name == "fermi":
        del kw["idem_tol"]
        return sp2.sp2_fermi(H, 0.0, 0.05, B, n_doublings=12, **kw)[0]
    sp2.sp2_density(H, n // 2, keep_history=True, **kw)
    return sp2.sp2_adjoint(B[0].contiguous(), handle)


# Bytes that each call takes with its matrices at the least padding (64 in FP64), one
# response at a time and no digits: the limit that has to be enough for it.
LEAST = {
    **{("fp64", 128, k): v for k, v in dict(density=398340, response=1971204, chi=2778436,
            chi_k1=5268804, fermi=4986896, adjoint=2385220).items()},
    **{("fp64", 190, k): v for k, v in dict(density=892388, response=4431332, chi=6221604,
            chi_k1=11824932, fermi=11215840, adjoint=5336868).items()},
    **{("fp64", 256, k): v for k, v in dict(density=1583300, response=7874756, chi=11041284,
            chi_k1=22051332, fermi=19935440, adjoint=9468420).items()},
    **{("fp64", 300, k): v for k, v in dict(density=2472196, response=12302596, chi=17238596,
            chi_k1=34441796, fermi=31146608, adjoint=14780996).items()},
    **{("fp64", 520, k): v for k, v in dict(density=8002244, response=39852740, chi=58452996,
            chi_k1=116845572, fermi=100903696, adjoint=50490372).items()},
    **{("fp32", 300, k): v for k, v in dict(density=1783492, response=8861380, chi=13600772,
            chi_k1=28936196, fermi=22428544, adjoint=11831300).items()},
    **{("fp32", 1000, k): v for k, v in dict(density=12623492, response=62955140, chi=96530372,
            chi_k1=209776580, fermi=159428144, adjoint=83947460).items()},
    **{("fp16x2", 300, k): v for k, v in dict(density=5259968, response=24134396, chi=33592360,
            chi_k1=52466708, fermi=79710384, adjoint=28349460).items()},
    **{("fp16x2", 1000, k): v for k, v in dict(density=21012096, response=96509628, chi=138473448,
            chi_k1=213970900, fermi=318812000, adjoint=117501908).items()},
    **{("bf16x3", 300, k): v for k, v in dict(density=6308544, response=28328640, chi=38835200,
            chi_k1=56136704, fermi=99633024, adjoint=32543744).items()},
}


@pytest.mark.parametrize("mode,n,name", sorted(LEAST))
def test_least_limit_is_enough(sp2, mode, n, name):
    """With the same result as without a limit (other products in FP64: digits or sums)."""
    H, B = _inputs(n, mode)
    free = _call(sp2, name, n, mode, H, B, sp2.Handle())
    h = sp2.Handle(LEAST[mode, n, name])
    got = _call(sp2, name, n, mode, H, B, h)
    assert h.workspace_bytes() <= LEAST[mode, n, name]
    if mode == "fp64":
        # some 30 steps of sums whose rounding, relative to the norms, each at most doubles
        assert (got - free).norm() <= 1e-8 * free.norm()
    else:
        assert torch.equal(got, free)


def test_wide_fp64_padding_needs_its_room(sp2):
    """Matrices of N = 300 are padded for the digits without a limit or under one with room
    for them, to 64 otherwise, and a call gives back nothing that another still needs."""
    n = 300
    H, B = _inputs(n, "fp64")
    wide, tight = sp2.Handle(64 << 20), sp2.Handle(16 << 20)
    d1, d2 = (_call(sp2, "density", n, "fp64", H, B, h) for h in (wide, tight))
    assert (d1 - d2).norm() <= 1e-10 * d1.norm()
    assert wide.workspace_bytes() > 16 * 512 * 512 + 3 * 8 * 512 * 512
    assert tight.workspace_bytes() < 4 * 8 * 320 * 320
    # a kept history outlives calls that are short of room
    sp2.sp2_density(H, n // 2, mode="fp64", keep_history=True, handle=tight, idem_tol=1e-10)
    want = sp2.sp2_adjoint(B[0].contiguous(), tight)
    try:
        sp2.sp2_density(_inputs(700, "fp32")[0], 350, mode="fp32", handle=tight)
    except sp2.SP2Error:
        pass
    assert torch.equal(sp2.sp2_adjoint(B[0].contiguous(), tight), want)


@pytest.mark.parametrize("extra", [0, 1, 3, 6, 12])
@pytest.mark.parametrize("name", ["chi", "chi_k1", "adjoint"])
def test_history_that_outgrows_the_room_runs_again(sp2, name, extra):
    """Limits between the least and what digits, the wide padding and the history take: the
    call returns its result under each of them (on the least padding where the number of
    checkpoints shows that the wide one has no room), and so does a second one."""
    n = 300
    H, B = _inputs(n, "fp64")
    want = _call(sp2, name, n, "fp64", H, B, sp2.Handle())
    h = sp2.Handle(LEAST["fp64", n, name] + extra * (8 << 20))
    for _ in range(2):
        got = _call(sp2, name, n, "fp64", H, B, h)
        assert (got - want).norm() <= 1e-8 * want.norm()


def test_short_room_of_one_call_leaves_the_digits_to_others(sp2):
    """A history that ran again on the least padding does not keep a density of the same size,
    which has room, from the wide one and its digits."""
    n = 300
    H, B = _inputs(n, "fp64")
    limit = LEAST["fp64", n, "chi"] + (44 << 20)      # 63.4 MB; chi with its digits takes 67.1
    h = sp2.Handle(limit)
    want = _call(sp2, "chi", n, "fp64", H, B, sp2.Handle())
    for _ in range(2):
        assert (_call(sp2, "chi", n, "fp64", H, B, h) - want).norm() <= 1e-8 * want.norm()
        held = h.workspace_bytes()
        assert held < 2 * LEAST["fp64", n, "chi"]
        _call(sp2, "density", n, "fp64", H, B, h)
        assert h.workspace_bytes() - held > 16 * 512 * 512      # the digits of X alone
        h = sp2.Handle(limit)


def test_batches_leave_room_for_the_next_call(sp2):
    """Finite-T responses by batches take free room under a limit; the density that follows
    finds the room it would have found beside one response at a time."""
    mode = "fp16x2"
    Hs, Bs = _inputs(300, mode)
    Hl, _ = _inputs(1000, mode)
    h = sp2.Handle(LEAST[mode, 300, "fermi"] + LEAST[mode, 1000, "density"])
    want = _call(sp2, "fermi", 300, mode, Hs, Bs, sp2.Handle())
    dens = _call(sp2, "density", 1000, mode, Hl, None, sp2.Handle())
    for _ in range(2):
        assert torch.equal(_call(sp2, "fermi", 300, mode, Hs, Bs, h), want)
        assert torch.equal(_call(sp2, "density", 1000, mode, Hl, None, h), dens)


def test_batch_growth_keeps_the_digits(sp2):
    """FP64 finite-T responses on a GPU that is nearly full: the scratch of a larger batch
    does not fit, and the products keep their digit buffers."""
    n, k, dbl = 2000, 6, 12
    mat = 8 * 2048 * 2048
    g = torch.Generator(device="cuda").manual_seed(0)
    H = torch.randn(n, n, generator=g, device="cuda", dtype=torch.float64)
    H = (H + H.T) * 0.2 / n ** 0.5
    B = torch.randn(k, n, generator=g, device="cuda", dtype=torch.float64)
    kw = dict(diag_only=True, mode="fp64", n_doublings=dbl)
    h = sp2.Handle()
    least = (2 * dbl + 1 + 6 + 6 + 1) * mat + 8 * mat      # history, scratch, R_I; digits and sums
    torch.cuda.empty_cache()
    fill = torch.cuda.mem_get_info()[0] - least - (n * n * 8 * (k + 1)) - 24 * mat
    filler = torch.empty(max(fill, 0), dtype=torch.uint8, device="cuda")
    try:
        D1, _, _ = sp2.sp2_fermi(H, 0.0, 0.1, B, handle=h, **kw)
    finally:
        del filler
        torch.cuda.empty_cache()
    assert h.workspace_bytes() > least - mat
    ref, _, _ = sp2.sp2_fermi(H, 0.0, 0.1, B, handle=sp2.Handle(), **kw)
    assert (D1 - ref).norm() <= 1e-9 * ref.norm()


def test_history_leaves_room_for_the_digits(sp2):
    """From K = 8193 on the sums of a product come in parts along K, two or three here, of 32
    bytes an entry each: the automatic checkpoint interval counts them (by one part it would
    choose the interval 1, and 2 + 9 + 2 matrices beside 16 of digits and sums do not fit)."""
    n = 8300
    mat = 8 * 8448 * 8448
    g = torch.Generator(device="cuda").manual_seed(0)
    H = torch.randn(n, n, generator=g, device="cuda", dtype=torch.float64)
    H = (H + H.T) * 0.002
    b = torch.ones(1, n, device="cuda", dtype=torch.float64)
    h = sp2.Handle(27 * mat + (1 << 30))
    chi, _, info = sp2.sp2_susceptibility(H, n // 2, b, direction="backward", diag_only=True, mode="fp64",
                                          sigma=[1, -1] * 4 + [1], bounds=(-1.0, 1.0), ckpt_k="auto",
                                          handle=h, allow_noconv=True)
    assert info["ckpt_k"] > 1 and bool(torch.isfinite(chi).all())
    assert h.workspace_bytes() > 18 * mat      # without the digits: 9 to 14 of them
