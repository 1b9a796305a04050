"""What the kernels do when a limit is reached that no scene of these sizes
reaches: a second library is built with the walks' stacks cut to an eighth and
no patience between the tiles of the sort, and must give the same bits."""
import os

import numpy as np
import pytest

import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FLAGS = ("-DGSRT_POOL_SHIFT=3", "-DGSRT_LOOKBACK_LIMIT=0", "--split-compile", "0")


@pytest.fixture(scope="module")
def gs():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2504_06598_gb300 as m
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for gpu tests")
    return m


@pytest.fixture(scope="module")
def run(gs, tmp_path_factory):
    """run(fn): fn() with the usual library and with the cut one."""
    from paper_2504_06598_gb300 import build as gbuild
    mp = pytest.MonkeyPatch()
    out = str(tmp_path_factory.mktemp("limits"))
    mp.setattr(gbuild, "BUILD", out)
    mp.setattr(gbuild, "LIB", os.path.join(out, "libgsrt_limits.so"))
    cut = gbuild.build(force=True, extra_flags=FLAGS)
    mp.undo()

    def both(fn):
        usual = fn()
        torch.cuda.synchronize()
        with pytest.MonkeyPatch.context() as m:
            m.setattr(gs, "LIB_PATH", cut)
            m.setattr(gs, "_lib", None)
            other = fn()
            torch.cuda.synchronize()
        return usual, other

    return both


@pytest.mark.parametrize("M", [8193, 70001])
def test_sort_without_waiting(gs, run, M):
    cloud = scenes.tiny_cloud(1, M=M)
    cloud.means[M // 2:] = cloud.means[0]
    g = gs.Gaussians.from_cloud(cloud)

    def order():
        bvh = gs.build_bvh(g)
        bvh.sync_status()
        ex = bvh.export()
        bvh.free()
        return ex["order"]

    usual, other = run(order)
    assert np.array_equal(usual, other)


@pytest.mark.parametrize("fmt", ["binary", "binary_q8"])
def test_walks_start_over(gs, run, fmt):
    """Warps per pixel, groups, tiles and shared walks whose stack fills."""
    cloud = scenes.shell_cloud(3, M=60000, sh_degree=1)
    cloud.log_scales[:] += 0.7
    g = gs.Gaussians.from_cloud(cloud)
    small = scenes.Pinhole(width=37, height=19, eye=(0.4, 0.3, 2.8))
    large = scenes.Pinhole(width=613, height=401, eye=(0.05, 0.02, 0.1), look_at=(1.0, 0.3, -0.4),
                           fov_y_deg=100.0)
    calls = [(small, 3, 0), (small, 16, 1), (small, 32, 1), (small, 8, 1), (small, 70, 0),
             (large, 1, 0), (large, 16, 0), (large, 50, 0)]
    views = scenes.wavefront_views(2, seed=4, fixed_res=(401, 299))

    def render():
        bvh = gs.build_bvh(g, node_format=fmt)
        out = []
        for cam, spp, spl in calls:
            out += gs.trace_stochastic(bvh, g, cam, seed=2, spp=spp, samples_per_lane=spl,
                                       want_hits=True)
        out += gs.render_views(bvh, g, views, scenes.ground_and_lights(2, seed=1), seed=5, spp=3,
                               want_samples=True)
        bvh.sync_status()
        bvh.free()
        return out

    for a, b in zip(*run(render)):
        assert torch.equal(a, b)
