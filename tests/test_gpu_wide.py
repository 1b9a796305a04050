"""The wide hierarchies against the binary one: the grouped traversals (8, 16
and 32 lanes on a pixel) must return the hits of the per-lane packets, which
read the binary nodes, at the sizes where the cut of the wide nodes changes
(one node, exactly full, one more, two levels) and on trees of equal codes."""
import numpy as np
import pytest

import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = (1, 2, 3, 8, 9, 16, 17, 32, 33, 65, 257, 1024, 1025, 7000)


@pytest.fixture(scope="module")
def gs():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2504_06598_gb300 as m
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for gpu tests")
    return m


def _cloud(M, coincident):
    cloud = scenes.tiny_cloud(M, M=M)
    cloud.log_scales[:] += 1.0
    if coincident:
        cloud.means[M // 2:] = cloud.means[0]
    return cloud


@pytest.mark.parametrize("fmt", ["binary", "binary_q8"])
@pytest.mark.parametrize("coincident", [False, True])
def test_grouped_hits_equal_packet_hits(gs, fmt, coincident):
    cam = scenes.Pinhole(width=21, height=13, eye=(0.4, 0.3, 2.8))
    for M in SIZES:
        g = gs.Gaussians.from_cloud(_cloud(M, coincident))
        bvh = gs.build_bvh(g, node_format=fmt)
        for lanes in (8, 16, 32):
            kw = dict(seed=M, spp=lanes, want_hits=True)
            assert gs.trace_layout(bvh, spp=lanes, samples_per_lane=1)["grouped"]
            _, a, ta = gs.trace_stochastic(bvh, g, cam, samples_per_lane=1, **kw)
            # eight samples per lane: fewer than eight lanes a pixel; an
            # explicit stack depth keeps the per-lane walk of the binary nodes
            _, b, tb = gs.trace_stochastic(bvh, g, cam, samples_per_lane=8, stack_depth=96, **kw)
            bvh.sync_status()
            assert torch.equal(a, b) and torch.equal(ta, tb), (M, lanes)
        assert M < 100 or (a >= 0).any()
        bvh.free()


SMALL = [scenes.Pinhole(width=37, height=19, eye=(0.4, 0.3, 2.8)),
         scenes.Pinhole(width=41, height=23, eye=(0.05, 0.02, 0.1), look_at=(1.0, 0.3, -0.4)),
         scenes.Pinhole(width=5, height=3, eye=(0.0, 0.0, 0.5), fov_y_deg=170.0),
         scenes.Pinhole(width=1, height=1, eye=(0.3, 0.1, 2.0)),
         scenes.Pinhole(width=33, height=9, eye=(0.0, 3.0, 0.0), up=(0.0, 0.0, 1.0))]
# more tiles than one wave of warps, where the tiles are taken
LARGE = [scenes.Pinhole(width=613, height=401, eye=(0.4, 0.3, 2.8)),
         scenes.Pinhole(width=517, height=403, eye=(0.05, 0.02, 0.1), look_at=(1.0, 0.3, -0.4),
                        fov_y_deg=150.0)]


@pytest.mark.parametrize("fmt", ["binary", "binary_q8"])
@pytest.mark.parametrize("spp,spl", [(1, 0), (3, 1), (5, 2), (7, 0), (16, 0), (32, 8)])
def test_tile_hits_equal_packet_hits(gs, fmt, spp, spl):
    """The tile traversal, and the warp per pixel of images too small for it,
    against the binary walk: an eye inside the cloud, a view so wide that a
    tile has no pyramid, one pixel, odd sizes, a range, and a range that ends
    before everything."""
    for cams, M, coincident in ((SMALL, 1, False), (SMALL, 2, False), (SMALL, 33, True),
                                (SMALL, 1025, False), (LARGE, 1, False), (LARGE, 33, False),
                                (LARGE, 1025, True)):
        g = gs.Gaussians.from_cloud(_cloud(M, coincident))
        bvh = gs.build_bvh(g, node_format=fmt)
        for cam in cams:
            for lim in ({}, dict(t_min=1.5, t_max=3.0), dict(t_max=1e-3)):
                kw = dict(seed=M, spp=spp, samples_per_lane=spl, want_hits=True, **lim)
                assert gs.trace_layout(bvh, spp=spp, samples_per_lane=spl)["lanes_per_pixel"] < 8
                rgb, a, ta = gs.trace_stochastic(bvh, g, cam, **kw)
                ref, b, tb = gs.trace_stochastic(bvh, g, cam, stack_depth=96, **kw)
                bvh.sync_status()
                assert torch.equal(a, b) and torch.equal(ta, tb), (M, cam)
                # sums of spp colours in another order
                assert (rgb - ref).abs().max() <= 2 * spp * 2.0 ** -24 * ref.abs().max()
        bvh.free()


@pytest.mark.parametrize("fmt", ["binary", "binary_q8"])
@pytest.mark.parametrize("spp,n_hits", [(33, 1), (64, 1), (65, 1), (200, 1), (16, 4), (17, 8)])
def test_shared_walk_hits_equal_packet_hits(gs, fmt, spp, n_hits):
    """Above 32 samples a pixel the library's own choice walks once for four
    pixels: against one pixel at a time, with odd image sizes, sample counts
    around 64, a range, and the stored payloads."""
    for cams, M, coincident in ((SMALL, 1, False), (SMALL, 2, False), (SMALL, 33, True),
                                (SMALL, 1025, False), (SMALL, 7000, True)):
        g = gs.Gaussians.from_cloud(_cloud(M, coincident))
        bvh = gs.build_bvh(g, node_format=fmt)
        for cam in cams:
            for lim in ({}, dict(t_min=1.5, t_max=3.0)):
                kw = dict(seed=M, spp=spp, n_hits=n_hits, **lim)
                rgb, a, ta = gs.trace_stochastic(bvh, g, cam, want_hits=True, **kw)
                ref, b, tb = gs.trace_stochastic(bvh, g, cam, want_hits=True, stack_depth=96, **kw)
                keys = gs.sample_keys(cam, spp, n_hits)
                again = gs.trace_stochastic(bvh, g, cam, keys=keys, **kw)
                bvh.sync_status()
                assert torch.equal(a, b) and torch.equal(ta, tb), (M, cam)
                assert torch.equal(again, rgb) and torch.equal(ref, rgb)
                gid = gs.decode_keys(keys)[2].reshape(cam.height, cam.width, spp, n_hits)
                assert torch.equal(gid.permute(2, 3, 0, 1), a.long())
        bvh.free()


@pytest.mark.parametrize("M", [1023, 1025, 8192, 8193, 10240, 10241, 70001])
@pytest.mark.parametrize("coincident", [False, True])
def test_sort_is_stable_and_complete(gs, M, coincident):
    """The one-block build up to 8,192 Gaussians and the tiled sort above:
    at the limit, at whole tiles of 2,048 keys and one past them, with half of
    the codes equal."""
    bvh = gs.build_bvh(gs.Gaussians.from_cloud(_cloud(M, coincident)))
    bvh.sync_status()
    ex = bvh.export()
    bvh.free()
    codes, order = ex["codes"], ex["order"].astype(np.int64)
    assert np.all(codes[1:] >= codes[:-1])
    eq = codes[1:] == codes[:-1]
    assert np.all(order[1:][eq] > order[:-1][eq])
    assert eq.any() or not coincident
    assert np.array_equal(np.sort(order), np.arange(M))


@pytest.mark.parametrize("fmt", ["binary", "binary_q8"])
@pytest.mark.parametrize("spp,n_hits,degree", [(1, 1, 0), (3, 1, 1), (16, 1, 3), (5, 4, 2), (70, 1, 3)])
def test_tile_gradients_equal_packet_gradients(gs, fmt, spp, n_hits, degree):
    """Gradients of the tile form (ten sums, one chain rule per Gaussian)
    against those of the per-lane form, which an explicit stack depth keeps:
    small images, and one with more tiles than a wave. Both add the same terms
    in float32 in different orders: the bound is that of the parity tests."""
    cams = SMALL[:2] + (LARGE[:1] if spp <= 16 else [])
    for M in (2, 33, 1025):
        cloud = scenes.shell_cloud(M, M=M, n_clusters=4, sh_degree=degree)
        cloud.log_scales[:] += 1.5
        g = gs.Gaussians.from_cloud(cloud)
        bvh = gs.build_bvh(g, node_format=fmt)
        for cam in cams:
            d = torch.randn((cam.height, cam.width, 3), device="cuda",
                            generator=torch.Generator("cuda").manual_seed(M))
            kw = dict(seed=M, spp=spp, n_hits=n_hits, bg=(0.2, 0.1, 0.4))
            keys = gs.sample_keys(cam, spp, n_hits)
            gs.trace_stochastic(bvh, g, cam, keys=keys, **kw)
            ref = gs.trace_backward(bvh, g, cam, d, stack_depth=96, **kw)
            for k in (None, keys):
                got = gs.trace_backward(bvh, g, cam, d, keys=k, **kw)
                bvh.sync_status()
                for name in ref:
                    bound = 1e-4 * ref[name].abs().max() + 1e-6
                    assert (got[name] - ref[name]).abs().max() <= bound, (name, M, cam)
        bvh.free()


@pytest.mark.parametrize("fmt", ["binary", "binary_q8"])
@pytest.mark.parametrize("spp,spl,n_hits", [(3, 1, 1), (5, 1, 1), (7, 1, 1), (17, 0, 1), (20, 0, 1), (24, 0, 1), (6, 1, 8),
                                            (5, 0, 4), (13, 2, 2), (20, 4, 1)])
def test_small_images_add_samples_in_the_layouts_order(gs, fmt, spp, spl, n_hits):
    """The warp per pixel of small images adds a pixel's samples in the order
    of the layout that gs_trace_layout reports: the image of the per-lane walk
    (which an explicit stack depth keeps) bit for bit."""
    cloud = scenes.tiny_cloud(5, M=700)
    cloud.log_scales[:] += 1.0
    g = gs.Gaussians.from_cloud(cloud)
    bvh = gs.build_bvh(g, node_format=fmt)
    for cam in SMALL[:2]:
        kw = dict(seed=6, spp=spp, n_hits=n_hits, samples_per_lane=spl, bg=(0.3, 0.2, 0.9))
        rgb = gs.trace_stochastic(bvh, g, cam, **kw)
        ref = gs.trace_stochastic(bvh, g, cam, stack_depth=96, **kw)
        assert torch.equal(rgb, ref)
    bvh.sync_status()
    bvh.free()


@pytest.mark.parametrize("fmt", ["binary", "binary_q8"])
@pytest.mark.parametrize("seed", [0, 2, 4, 5])
def test_far_outliers_hide_nothing(gs, fmt, seed):
    """Gaussians far outside the scene make nodes as long as they are far; what
    lies beside them in such a node is still found."""
    M, n = 4000, 1500
    cloud = scenes.tiny_cloud(seed, M=M)
    rng = np.random.default_rng(seed)
    far = 10.0 ** rng.uniform(0.5, 8, (n, 3)) * rng.choice([-1, 1], (n, 3))
    cloud.means[:n, 0] = far[:, 0]
    cloud.log_scales[:] -= 1.0
    cloud = cloud.subset(rng.permutation(M))
    g = gs.Gaussians.from_cloud(cloud)
    bvh = gs.build_bvh(g, node_format=fmt)
    for cam in LARGE[:1] + SMALL[:2]:
        for spp in (1, 16, 64):
            kw = dict(seed=1, spp=spp, want_hits=True)
            _, a, ta = gs.trace_stochastic(bvh, g, cam, **kw)
            _, b, tb = gs.trace_stochastic(bvh, g, cam, stack_depth=96, **kw)
            assert torch.equal(a, b) and torch.equal(ta, tb), (cam, spp)
    bvh.sync_status()
    bvh.free()
