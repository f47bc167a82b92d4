"""The training decode past 512 atoms, three and four column tiles a row (BF16: one tile of target
boxes; single CTAs or CTA pairs, an odd last row tile; dV split into whole waves over the pixels),
against float64 PyTorch with the forms' bars: BF16 gradients by norm 2e-2 and loss parts 5e-3, FP32
1e-3 and 1e-4; row counts that leave partial tiles and give every CTA several."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_2602_12314_gb300 import api as _api
    return _api


@pytest.mark.parametrize("precision,grad_bar,loss_bar", [("BF16", 2e-2, 5e-3), ("FP32", 1e-3, 1e-4)])
@pytest.mark.parametrize("n,d,M,D", [(130, 32, 544, 128), (41_001, 16, 544, 384), (33_000, 32, 800, 640),
                                     (20_011, 64, 1024, 1024),
                                     (300, 16, 1024, 768), (33_001, 32, 768, 512)])
def test_gradients_match_float64(api, n, d, M, D, precision, grad_bar, loss_bar):
    g = torch.Generator(device="cuda").manual_seed(n)
    Q = torch.randn(n, d, generator=g, device="cuda")
    K, V = (torch.randn(M, w, generator=g, device="cuda") / d**0.5 for w in (d, D))
    F = torch.nn.functional.normalize(torch.randn(n, D, generator=g, device="cuda"), dim=1)
    F = F.bfloat16() if precision == "BF16" else F
    mask = (torch.rand(n, generator=g, device="cuda") > 0.1).to(torch.uint8)
    cfg = api.LossConfig(lambda_D=0.0)
    with api.Context(0) as ctx:
        parts, dQ, dK, dV = api.decode_loss_bwd(ctx, Q, K, V, V, F, mask, cfg, precision=getattr(api, precision))
    q, k, v = (x.double().requires_grad_() for x in (Q, K, V))
    Fh = torch.softmax(q @ k.T / d**0.5, 1) @ v
    f, m, nv = F.double(), mask.double(), float(mask.sum())
    cos = (m * (1 - torch.nn.functional.cosine_similarity(Fh, f, dim=1, eps=1e-8))).sum() / nv
    l2 = (m * (Fh - f).square().sum(1)).sum() / (nv * D)
    (cfg.lambda_f * (cfg.lambda_cos * cos + cfg.lambda_2 * l2)).backward()
    for got, want in ((parts[0], cos.detach()), (parts[1], l2.detach())):
        assert abs(float(got) - float(want)) <= loss_bar * abs(float(want))
    for got, want in ((dQ, q.grad), (dK, k.grad), (dV, v.grad)):
        assert float((got.double() - want).norm() / want.norm()) <= grad_bar
