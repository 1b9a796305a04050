"""The walks that gs_trace_stochastic chooses among, each reached through a size
that takes it: the hits and the image of the per-lane walk of the binary nodes
(which an explicit stack depth keeps), bit for bit."""
import functools

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


@functools.lru_cache(maxsize=2)
def _cloud(M):
    cloud = scenes.shell_cloud(3, M=M, n_clusters=8, sh_degree=1)
    cloud.log_scales[:] += 0.5
    return cloud


# Gaussians, width, height, samples, hits
CASES = [
    (1025, 64, 48, 3, 1), (1025, 63, 47, 24, 1), (1025, 33, 21, 60, 1), (5000, 33, 21, 15, 4),  # warp per pixel
    (1025, 613, 401, 1, 1), (1025, 613, 401, 5, 2), (600, 613, 401, 60, 1),  # tiles
    (20000, 613, 401, 3, 1), (20000, 613, 401, 16, 1),  # with each leaf's box tested
    (5000, 613, 401, 40, 1), (5000, 613, 401, 64, 1), (1025, 613, 401, 127, 1), (33, 613, 401, 25, 4),  # shared
    (300, 613, 401, 4, 1), (5000, 160, 121, 100, 1), (1025, 613, 401, 129, 1),  # the layout's own
    (1000000, 500, 403, 8, 1),  # packets of a dense scene
    (70000, 61, 930, 2, 1), (70000, 930, 61, 2, 1),  # narrow and wide: tiles, warp per pixel
]


@pytest.mark.parametrize("fmt", ["binary", "binary_q8"])
@pytest.mark.parametrize("M,spp,spl,n_hits", [(5000, 12, 1, 1), (5000, 31, 2, 1), (70000, 16, 1, 1),
                                              (70000, 62, 2, 1), (5000, 24, 4, 2)])
def test_passes_of_8_to_31(gs, fmt, M, spp, spl, n_hits):
    """The caller's samples per lane: whole warps in place of groups, in the
    layout's order of sums."""
    g = gs.Gaussians.from_cloud(_cloud(M))
    bvh = gs.build_bvh(g, node_format=fmt)
    cam = scenes.Pinhole(width=161, height=93, eye=(0.5, 0.8, 2.4))
    kw = dict(seed=4, spp=spp, n_hits=n_hits, samples_per_lane=spl, bg=(0.3, 0.1, 0.7),
              want_hits=True)
    rgb, a, ta = gs.trace_stochastic(bvh, g, cam, **kw)
    ref, b, tb = gs.trace_stochastic(bvh, g, cam, stack_depth=96, **kw)
    bvh.sync_status()
    bvh.free()
    assert torch.equal(a, b) and torch.equal(ta, tb) and torch.equal(rgb, ref)


@pytest.mark.parametrize("fmt", ["binary", "binary_q8"])
@pytest.mark.parametrize("M,w,h,spp,n_hits", CASES)
def test_walks_agree(gs, fmt, M, w, h, spp, n_hits):
    if M > 100000 and fmt != "binary":
        pytest.skip("once is enough")
    g = gs.Gaussians.from_cloud(_cloud(M))
    bvh = gs.build_bvh(g, node_format=fmt)
    cam = scenes.Pinhole(width=w, height=h, eye=(0.5, 0.8, 2.4))
    kw = dict(seed=4, spp=spp, n_hits=n_hits, bg=(0.3, 0.1, 0.7), want_hits=True)
    rgb, a, ta = gs.trace_stochastic(bvh, g, cam, **kw)
    ref, b, tb = gs.trace_stochastic(bvh, g, cam, stack_depth=96, **kw)
    bvh.sync_status()
    bvh.free()
    assert (a >= 0).any()
    assert torch.equal(a, b) and torch.equal(ta, tb) and torch.equal(rgb, ref)
