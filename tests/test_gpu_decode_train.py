"""The BF16 training decode past 512 atoms (one tile of target boxes, five operand stages) and at
two to four column tiles, against float64 PyTorch with the BF16 bars: gradients by norm (2e-2), loss
parts 5e-3; row counts that leave partial tiles and give every CTA several."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_2602_12314_gb300 import api as _api
    return _api


@pytest.mark.parametrize("n,d,M,D", [(130, 32, 544, 128), (41_001, 16, 544, 384), (33_000, 32, 800, 640),
                                     (20_011, 64, 1024, 1024)])
def test_bf16_gradients_match_float64(api, n, d, M, D):
    g = torch.Generator(device="cuda").manual_seed(n)
    Q = torch.randn(n, d, generator=g, device="cuda")
    K, V = (torch.randn(M, w, generator=g, device="cuda") / d**0.5 for w in (d, D))
    F = torch.nn.functional.normalize(torch.randn(n, D, generator=g, device="cuda"), dim=1).bfloat16()
    mask = (torch.rand(n, generator=g, device="cuda") > 0.1).to(torch.uint8)
    cfg = api.LossConfig(lambda_D=0.0)
    with api.Context(0) as ctx:
        parts, dQ, dK, dV = api.decode_loss_bwd(ctx, Q, K, V, V, F, mask, cfg, precision=api.BF16)
    q, k, v = (x.double().requires_grad_() for x in (Q, K, V))
    Fh = torch.softmax(q @ k.T / d**0.5, 1) @ v
    f, m, nv = F.double(), mask.double(), float(mask.sum())
    cos = (m * (1 - torch.nn.functional.cosine_similarity(Fh, f, dim=1, eps=1e-8))).sum() / nv
    l2 = (m * (Fh - f).square().sum(1)).sum() / (nv * D)
    (cfg.lambda_f * (cfg.lambda_cos * cos + cfg.lambda_2 * l2)).backward()
    for got, want in ((parts[0], cos), (parts[1], l2)):
        assert abs(float(got) - float(want)) <= 5e-3 * abs(float(want))
    for got, want in ((dQ, q.grad), (dK, k.grad), (dV, v.grad)):
        assert float((got.double() - want).norm() / want.norm()) <= 2e-2
