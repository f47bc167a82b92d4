"""Tile lists of synthetic projections at the edges of the binning kernels, exactly (integers): scan
blocks of 64 tiles (one tile, 64, 65, more than 32 blocks), splats of many tiles beside splats of
none, lists of 255 to 258 keys (counted or sorted by the network), lists above 4,096 keys with more pairs than the merge buffers start with (the second sort),
depth ties, no pairs at all, and a buffer that is too small."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_2602_12314_gb300 import api as _api
    return _api


def _camera(width, height):
    from paper_2602_12314_gb300 import _lib as L
    c = L.Camera(fx=50.0, fy=50.0, cx=width / 2, cy=height / 2, z_near=0.01, width=width, height=height)
    c.R[:] = [1, 0, 0, 0, 1, 0, 0, 0, 1]
    return c


def _scene(api, n, cam, span, seed, visible):
    """Random rects of up to span x span tiles; depths with ties."""
    tx, ty = (cam.width + 15) // 16, (cam.height + 15) // 16
    g = np.random.default_rng(seed)
    x0, y0 = g.integers(0, tx, n), g.integers(0, ty, n)
    x1, y1 = np.minimum(tx, x0 + g.integers(1, span + 1, n)), np.minimum(ty, y0 + g.integers(1, span + 1, n))
    rect = np.stack([x0, y0, x1, y1], 1).astype(np.int32)
    touched = ((x1 - x0) * (y1 - y0) * (g.random(n) < visible)).astype(np.int32)
    depth = (g.integers(1, 200, n) / 16).astype(np.float32)
    dev = lambda a: torch.as_tensor(a, device="cuda")
    proj = api.Projection(dev(np.zeros((n, 2), np.float32)), dev(np.zeros((n, 4), np.float32)), dev(depth), dev(rect),
                          dev(touched))
    own = np.repeat(np.arange(n), touched)
    k = np.arange(len(own)) - np.repeat(np.cumsum(touched) - touched, touched)
    w = (x1 - x0)[own]
    tile = (y0[own] + k // w) * tx + x0[own] + k % w
    at = np.lexsort((own, depth[own], tile))
    ends = np.cumsum(np.bincount(tile, minlength=tx * ty))
    ranges = np.stack([np.concatenate([[0], ends[:-1]]), ends], 1)
    ranges[ranges[:, 0] == ranges[:, 1]] = 0
    return proj, own[at], ranges


@pytest.mark.parametrize("n,width,height,span,visible", [
    (1, 16, 16, 1, 1.0), (700, 128, 128, 3, 0.7), (999, 1040, 16, 70, 0.5), (20_000, 1200, 680, 9, 0.3),
    (3_000, 700, 500, 40, 0.9), (90_001, 64, 64, 4, 1.0), (4_097, 16, 16, 1, 1.0), (255, 16, 16, 1, 1.0),
    (256, 16, 16, 1, 1.0), (257, 16, 16, 1, 1.0), (4_096, 16, 16, 1, 1.0), (515, 640, 480, 8, 0.0)])
def test_lists_equal_a_sort(api, n, width, height, span, visible):
    from paper_2602_12314_gb300 import _lib as L
    cam = _camera(width, height)
    proj, ids, ranges = _scene(api, n, cam, span, n, visible)
    P = len(ids)
    with api.Context(0) as ctx:
        for rep in range(4):  # plain launches, then the captured and the replayed ones
            bins = api.sort(ctx, proj, cam, capacity=max(P, 1))
            assert bins.num_pairs == P
            np.testing.assert_array_equal(bins.tile_ranges.cpu().numpy(), ranges)
            np.testing.assert_array_equal(bins.pair_ids[:P].cpu().numpy(), ids)
        if P > 1:
            bins = api.TileBins(torch.full((P,), -1, dtype=torch.int32, device="cuda"), bins.tile_ranges, 0)
            bs, ps = bins.struct(), proj.struct()
            bs.capacity = P - 1
            assert L.load().latentam_sort(ctx.handle, n, ctypes.byref(ps), ctypes.byref(cam), ctypes.byref(bs),
                                          api._stream()) == L.ERR_CAPACITY
            assert bs.num_pairs == P and int(bins.tile_ranges.abs().sum()) == 0
            assert bool((bins.pair_ids == -1).all())


def test_pair_count_is_exact_when_a_look_back_gives_up(api):
    """The last block's look-back is made to give up: no tile keeps a list, the pair count is still that
    of the splats (a call that finds its buffer too small asks for the right size), and the next
    binning reports the wait, the one after it is complete."""
    from paper_2602_12314_gb300 import _lib as L
    cam = _camera(1200, 680)  # 3,225 tiles: 51 scan blocks
    proj, ids, ranges = _scene(api, 20_000, cam, 9, 7, 0.3)
    P = len(ids)
    with api.Context(0) as ctx:
        ctx.test_wait_timeout(0)
        bins = api.sort(ctx, proj, cam, capacity=P)
        assert bins.num_pairs == P and int(bins.tile_ranges.abs().sum()) == 0
        with pytest.raises(L.LatentamError) as e:
            api.sort(ctx, proj, cam, capacity=P)
        assert e.value.status == L.ERR_TIMEOUT
        bins = api.sort(ctx, proj, cam, capacity=P)
        assert bins.num_pairs == P
        np.testing.assert_array_equal(bins.tile_ranges.cpu().numpy(), ranges)
        np.testing.assert_array_equal(bins.pair_ids[:P].cpu().numpy(), ids)


@pytest.mark.parametrize("n,width,height,span", [(1, 2000, 1500, 125), (5, 2000, 1500, 125), (33, 640, 480, 40),
                                                 (1216, 640, 480, 12), (1217, 300, 200, 9), (2433, 320, 240, 20),
                                                 (20_000, 320, 240, 3)])
def test_splats_shared_by_several_warps(api, n, width, height, span):
    """Few splats of many tiles, at the counts where one warp more or fewer shares 32 splats' pairs."""
    cam = _camera(width, height)
    proj, ids, ranges = _scene(api, n, cam, span, 3 * n, 0.9)
    P = len(ids)
    with api.Context(0) as ctx:
        for _ in range(3):
            bins = api.sort(ctx, proj, cam, capacity=max(P, 1))
            assert bins.num_pairs == P
            np.testing.assert_array_equal(bins.tile_ranges.cpu().numpy(), ranges)
            np.testing.assert_array_equal(bins.pair_ids[:P].cpu().numpy(), ids)
