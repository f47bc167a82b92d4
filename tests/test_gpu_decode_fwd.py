"""The inference decode latentam_decode_fwd at the rims of its tiles against float64 PyTorch: ragged
row counts (one row, a partial warp, several tiles per CTA), atoms that do not fill a 64-wide K
chunk, one to four 256-feature column tiles, every tensor-core form.  Bars: the parity bars of the
forms (relative 1e-4 per row for FP32; per-pixel cosine 0.999 for BF16 and 0.995 for FP8), and
rows past the last one untouched."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_2602_12314_gb300 import api as _api
    return _api


@pytest.fixture(scope="module")
def ctx(api):
    c = api.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("precision", ["FP32", "BF16", "FP8"])
@pytest.mark.parametrize("n,d,M,D", [(1, 16, 32, 128), (33, 32, 96, 384), (129, 64, 288, 640),
                                     (300, 32, 64, 256),
                                     (45_003, 32, 160, 1024), (2_000, 32, 1024, 768)])
def test_rows_match_float64(api, ctx, precision, n, d, M, D):
    g = torch.Generator(device="cuda").manual_seed(n + M)
    Q = torch.randn(n, d, generator=g, device="cuda")
    K = torch.randn(M, d, generator=g, device="cuda") / d**0.5
    V = torch.randn(M, D, generator=g, device="cuda") / d**0.5
    prec = getattr(api, precision)
    Fh, stats = api.decode_fwd(ctx, Q, K, V, precision=prec)
    S = Q.double() @ K.double().T / d**0.5
    want = torch.softmax(S, 1) @ V.double()
    got = Fh.double()
    if precision == "FP32":
        err = ((got - want).norm(dim=1) / want.norm(dim=1)).max()
        assert float(err) <= 1e-4
    else:
        cos = torch.nn.functional.cosine_similarity(got, want, dim=1).min()
        assert float(cos) >= (0.999 if precision == "BF16" else 0.995)
    assert torch.isfinite(stats).all()


def test_rows_past_the_last_one_are_not_written(api, ctx):
    import ctypes

    from paper_2602_12314_gb300 import _lib as L
    n, d, M, D = 70, 32, 64, 256
    Q, K, V = (torch.randn(*s, device="cuda") for s in ((n, d), (M, d), (M, D)))
    out = torch.full((128, D), 7.0, device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    L.check(L.load().latentam_decode_fwd(ctx.handle, p(Q), n, d, p(K), p(V), M, D, 0.0, int(api.BF16), p(out), None,
                                         st))
    torch.cuda.synchronize()
    assert bool((out[n:] == 7.0).all()) and bool((out[:n] != 7.0).any(dim=1).all())


@pytest.mark.parametrize("precision,M", [("FP32", 32), ("BF16", 32), ("FP8", 32), ("FP32", 256), ("BF16", 384)])
def test_many_short_tiles_per_cta_leave_no_wait_behind(api, ctx, precision, M):
    """Two dozen of the shortest tiles per CTA (one feature tile, few atoms), launched back to back:
    the warps that send their own output must not run ahead of any other warp's wait.  A wait that
    gives up raises the flag that the next binning reports."""
    from workloads import random_scene
    n, d, D = 24 * 152 * 128 + 77, 16, 128
    g = torch.Generator(device="cuda").manual_seed(M)
    Q = torch.randn(n, d, generator=g, device="cuda")
    K = torch.randn(M, d, generator=g, device="cuda") / d**0.5
    V = torch.randn(M, D, generator=g, device="cuda") / d**0.5
    prec = getattr(api, precision)
    first, _ = api.decode_fwd(ctx, Q, K, V, precision=prec, want_stats=False)
    for _ in range(20):
        again, _ = api.decode_fwd(ctx, Q, K, V, precision=prec, want_stats=False)
    assert torch.equal(first, again)
    s = random_scene(5, n=200, d=16, M=32, D=128, width=48, height=40, log_scale=-2.6)
    api.sort(ctx, api.project(ctx, s.means, s.quats, s.scales, s.opacities, s.camera), s.camera)  # raises if flagged
    want = torch.softmax(Q.double() @ K.double().T / d**0.5, 1) @ V.double()
    if precision == "FP32":
        assert float(((first - want).norm(dim=1) / want.norm(dim=1)).max()) <= 1e-4
    else:
        cos = torch.nn.functional.cosine_similarity(first.double(), want, dim=1).min()
        assert float(cos) >= (0.999 if precision == "BF16" else 0.995)


@pytest.mark.parametrize("precision", ["FP32", "BF16"])
@pytest.mark.parametrize("n,D", [(44_900, 768), (300, 256), (128, 128)])
def test_cta_pairs_with_several_and_odd_row_tiles(api, ctx, precision, n, D):
    """The paired form (M = 512): 351 row tiles are several per CTA and an odd number, three and one
    leave the last pair's odd CTA past the rows; nothing is written there."""
    import ctypes

    from paper_2602_12314_gb300 import _lib as L
    d, M = 32, 512
    g = torch.Generator(device="cuda").manual_seed(n)
    Q = torch.randn(n, d, generator=g, device="cuda")
    K = torch.randn(M, d, generator=g, device="cuda") / d**0.5
    V = torch.randn(M, D, generator=g, device="cuda") / d**0.5
    out = torch.full((n + 256, D), 7.0, device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    L.check(L.load().latentam_decode_fwd(ctx.handle, p(Q), n, d, p(K), p(V), M, D, 0.0,
                                         int(getattr(api, precision)), p(out), None, st))
    want = torch.softmax(Q.double() @ K.double().T / d**0.5, 1) @ V.double()
    assert bool((out[n:] == 7.0).all())
    if precision == "FP32":
        assert float(((out[:n] - want).norm(dim=1) / want.norm(dim=1)).max()) <= 1e-4
    else:
        assert float(torch.nn.functional.cosine_similarity(out[:n].double(), want, dim=1).min()) >= 0.999
