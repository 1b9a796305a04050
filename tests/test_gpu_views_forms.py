"""The forms of the batched launch against one another: which of them a frame
takes follows from its size, its samples and the handle's nodes, and must not
show in any sample's outcome. The 4-wide handles, whose camera and shadow rays
walk as per-lane packets, are the other side."""
import numpy as np
import pytest

import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gs():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2504_06598_gb300 as m
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for gpu tests")
    return m


def _render(gs, g, cams, ex, fmt, **kw):
    bvh = gs.build_bvh(g, node_format=fmt)
    rgb, smp = gs.render_views(bvh, g, cams, ex, seed=5, want_samples=True, **kw)
    bvh.sync_status()
    bvh.free()
    return rgb, smp


@pytest.mark.parametrize("fmt", ["binary", "binary_q8"])
@pytest.mark.parametrize("spp", [56, 57, 60, 63, 64])
@pytest.mark.parametrize("size", [(23, 17), (171, 120)])
def test_samples_up_to_64(gs, fmt, spp, size):
    """Eight samples a lane make eight passes from 57 samples on: a warp per
    pixel in the small frame, tiles in the large one, packets with an explicit
    stack depth."""
    g = gs.Gaussians.from_cloud(scenes.shell_cloud(7, M=6000))
    cams = scenes.wavefront_views(1, seed=2, fixed_res=size)
    ex = scenes.ground_and_lights(2, seed=1)
    ref, smp = _render(gs, g, cams, ex, "wide4", spp=spp)
    assert (smp[..., 0] == -2).any() and (smp[..., 0] >= 0).any() and (smp[..., 1] >= 0).any()
    for depth in (0, 96):
        rgb, got = _render(gs, g, cams, ex, fmt, spp=spp, stack_depth=depth)
        assert torch.equal(got, smp)
        # sums of spp colours in another order
        assert (rgb - ref).abs().max() <= 2 * spp * 2.0 ** -24 * ref.abs().max()


@pytest.mark.parametrize("spp", [1, 3, 5, 17, 20, 24, 56, 60])
def test_small_frames_add_samples_in_the_layouts_order(gs, spp):
    """A warp per pixel, as small frames take it: the packets' image to the
    last bit."""
    g = gs.Gaussians.from_cloud(scenes.shell_cloud(7, M=6000))
    cams = scenes.wavefront_views(2, seed=4, fixed_res=(31, 23))
    ex = scenes.ground_and_lights(3, seed=1)
    ref, smp = _render(gs, g, cams, ex, "wide4", spp=spp)
    for fmt in ("binary", "binary_q8"):
        rgb, got = _render(gs, g, cams, ex, fmt, spp=spp)
        assert torch.equal(got, smp) and torch.equal(rgb, ref), fmt


@pytest.mark.parametrize("fmt", ["binary", "binary_q8"])
@pytest.mark.parametrize("spp", [1, 3, 4, 16])
def test_tiles(gs, fmt, spp):
    """Frames large enough for the tile walk: camera rays and the shadow rays
    toward lights above the scene, in its middle and close to the ground (whose
    nearest pixels have no pyramid), at odd sizes."""
    g = gs.Gaussians.from_cloud(scenes.shell_cloud(7, M=6000))
    cams = scenes.wavefront_views(2, seed=4, fixed_res=(401, 299))
    ex = scenes.ground_and_lights(2, seed=1)
    ex.lights += [((0.0, 0.0, 0.0), (1.0, 2.0, 3.0)), ((0.4, -1.29, 0.3), (0.1, 0.1, 0.1))]
    ref, smp = _render(gs, g, cams, ex, "wide4", spp=spp)
    rgb, got = _render(gs, g, cams, ex, fmt, spp=spp)
    assert torch.equal(got, smp) and torch.equal(rgb, ref)


@pytest.mark.parametrize("fmt", ["binary", "binary_q8"])
@pytest.mark.parametrize("spp", [1, 4])
@pytest.mark.parametrize("size", [1e-3, 1e-4])
def test_shadows_of_gaussians_beside_the_light(gs, fmt, spp, size):
    """A light a hundred units above the ground, inside a cloud as small as
    `size`: shadow rays pass the light by the rounding of their direction, a
    length not far below that of the cloud's Gaussians."""
    cloud = scenes.tiny_cloud(9, M=2000)
    cloud.means[:] *= np.float32(size)
    cloud.log_scales[:] += np.float32(np.log(size))
    g = gs.Gaussians.from_cloud(cloud)
    cams = [scenes.Pinhole(width=401, height=299, eye=(x, 60.0, 0.1), look_at=(0.0, -100.0, 0.0),
                           up=(0.0, 0.0, 1.0), ray_id_offset=o) for x, o in ((0.0, 0), (90.0, 401 * 299))]
    ex = scenes.SceneExtras(lights=[((0.0, 0.0, 0.0), (1.0, 1.0, 1.0))], has_ground=True,
                            ground_y=-100.0, ground_half_extent=300.0)
    _, smp = _render(gs, g, cams, ex, "wide4", spp=spp)
    _, got = _render(gs, g, cams, ex, fmt, spp=spp)
    lit, got_lit = smp[..., 2] != 0, got[..., 2] != 0
    assert lit.any() and not lit[smp[..., 0] == -2].all()
    # a shadow is a hit that was found. (The packets miss a few of these: their
    # slabs are taken from the ground point, a hundred units away.)
    assert torch.equal(got[..., :2], smp[..., :2])
    assert not (got_lit & ~lit).any()


@pytest.mark.parametrize("fmt", ["binary", "binary_q8"])
def test_bounce_rays_at_a_small_stack(gs, fmt):
    """An opaque sheet above the ground is the root's left child: a bounce ray
    that evaluates it first never pushes a node."""
    cloud = scenes.tiny_cloud(2, M=65)
    cloud.means[1:, 0] = 0.55 + 0.45 * np.abs(cloud.means[1:, 0])
    cloud.means[1:, 1] += 2.0
    cloud.log_scales[1:] += 1.0
    cloud.means[0] = (0.0, 0.0, 0.0)
    cloud.log_scales[0] = (5.0, -4.0, 5.0)
    cloud.quats[0] = (1.0, 0.0, 0.0, 0.0)
    cloud.opacity_logits[0] = 40.0
    g = gs.Gaussians.from_cloud(cloud)
    ex = scenes.SceneExtras(lights=[], has_ground=True, ground_y=-0.5, ground_half_extent=3.0, bounce=True, shadow_eps=1e-4)
    bvh = gs.build_bvh(g, node_format=fmt)
    cnt = torch.zeros(4, dtype=torch.int64, device="cuda")
    # eight rays at a time: too few for the warp to evaluate at once
    for x in np.linspace(-0.4, 1.2, 60):
        cams = [scenes.Pinhole(width=1, height=1, eye=(0.3, -0.1, 0.4), look_at=(float(x), -0.5, 0.0))]
        _, s0 = gs.render_views(bvh, g, cams, ex, seed=1, spp=8, want_samples=True)
        # (counters: camera rays in groups, which have a stack of their own)
        _, s1 = gs.render_views(bvh, g, cams, ex, seed=1, spp=8, counters=cnt, stack_depth=1,
                                want_samples=True)
        bvh.sync_status()
        assert torch.equal(s0, s1)
        assert (s0[..., 1] == 0).any()
    bvh.free()


@pytest.mark.parametrize("fmt", ["binary", "binary_q8"])
@pytest.mark.parametrize("spp", [1, 16])
def test_tiles_that_test_each_leaf(gs, fmt, spp):
    """More Gaussians than a sixteenth of a view's pixels, a light among them."""
    cloud = scenes.shell_cloud(7, M=20000)
    g = gs.Gaussians.from_cloud(cloud)
    cams = scenes.wavefront_views(2, seed=4, fixed_res=(401, 299))
    ex = scenes.ground_and_lights(1, seed=1)
    ex.lights += [((0.0, 0.0, 0.0), (1.0, 2.0, 3.0)),
                  (tuple(float(v) for v in cloud.means[0] + 0.01), (0.1, 0.1, 0.1))]
    ref, smp = _render(gs, g, cams, ex, "wide4", spp=spp)
    rgb, got = _render(gs, g, cams, ex, fmt, spp=spp)
    assert torch.equal(got, smp) and torch.equal(rgb, ref)
