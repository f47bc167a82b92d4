"""The query render's backward on a full chip: images of many tiles, so that blocks run in several
waves, and tile lists of many batches of splats.  Every channel's sums are taken in the same order
whatever their number, so the gradient of 64 channels must be that of its two halves of 32 and of its
four quarters of 16, up to the order of the atomics between the tiles of a splat (FP32 rounding over
up to some hundred adds: 2e-6 of the norm)."""
import pytest

from workloads import Camera, random_scene

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


@pytest.mark.parametrize("n,width,height,log_scale", [(20_000, 640, 480, -2.0), (200_000, 320, 240, -4.0),
                                                      (3000, 1000, 700, -0.5)])
def test_channels_do_not_depend_on_their_number(api, ctx, n, width, height, log_scale):
    s = random_scene(7, n=n, d=64, M=32, D=128, width=20, height=20, log_scale=log_scale)
    cam = Camera(R=s.camera.R, t=s.camera.t, fx=0.94 * width, fy=0.94 * width, cx=width / 2, cy=height / 2, width=width,
                 height=height, z_near=s.camera.z_near)
    proj = api.project(ctx, s.means, s.quats, s.scales, s.opacities, cam)
    bins = api.sort(ctx, proj, cam)
    Q, _, nc = api.render_fwd(ctx, proj, cam, bins, torch.as_tensor(s.f, device="cuda"))
    dQ = torch.randn(Q.shape, generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    whole = api.render_bwd(ctx, proj, cam, bins, nc, dQ)
    assert bool(torch.isfinite(whole).all()) and float(whole.norm()) > 0
    for d in (32, 16):
        parts = torch.cat([api.render_bwd(ctx, proj, cam, bins, nc, dQ[:, k:k + d]) for k in range(0, 64, d)], 1)
        assert float((parts - whole).norm() / whole.norm()) <= 2e-6
