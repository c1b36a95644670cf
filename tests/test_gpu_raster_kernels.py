"""The rasterizer's kernels: configurations that run the same one are tuned as one, and
both block shapes of the 16-pixel kernel (256 threads on one square when squares are few,
128 on each of two otherwise) give the images of the 8-pixel kernels bit for bit, with
pair counting off.
"""
import pytest

from paper_2609_30741_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_30741_gb300 import build
    build.build()
    from paper_2609_30741_gb300 import gs as gsmod
    return gsmod


def _kernel(cfg):
    tile, pix, batch = cfg
    return tile, pix if tile == 8 else 0, min(batch, 64)


def test_configurations_of_one_kernel_share_their_time(gs):
    scene, cam, dom, aff = synth.workload_small()
    ctx = gs.Context(scene.n, cam.width, cam.height, max_instances=1 << 22, min_tile=8)
    best, ms, results = gs.autotune_stereo(ctx, gs.DeviceScene(scene), dom, aff, cam, reps=3, use_cache=False)
    times = {}
    for c, t in results:
        times.setdefault(_kernel(c), set()).add(t)
    assert len(results) == 28 and len(times) == 8
    assert all(len(v) == 1 and min(v) > 0 for v in times.values())
    assert times[_kernel(best)] == {ms} and ms == min(min(v) for v in times.values())


# 16-pixel squares of the image: 192, 1216 (as many as groups on 152 SMs), 1248 and 7500
@pytest.mark.parametrize("size", [(256, 192), (608, 512), (611, 500), (1600, 1200)])
@pytest.mark.parametrize("ellipsoids", [False, True])
def test_both_block_shapes_of_the_16_pixel_kernel(gs, size, ellipsoids):
    scene = synth.scene_object_ground(1305, n=30_000, sh_degree=1)
    if ellipsoids:
        scene = synth.to_ellipsoids(scene)
    cam = synth.centred_camera(size[0], size[1], float(size[0]))
    pose = synth.arc_poses()[3]
    ds = gs.DeviceScene(scene)
    ctx = gs.Context(scene.n, cam.width, cam.height, max_instances=1 << 24, min_tile=8)
    ref = None
    for cfg in ((8, 1, 32), (8, 2, 64), (16, 2, 32), (16, 4, 128), (32, 2, 32), (32, 8, 256)):
        ctx.set_raster(*cfg)
        got = [t.clone() for t in ctx.render_mono(ds, pose, cam, bg=(0.1, 0.2, 0.3))]
        ctx.check_ok()
        if ref is None:
            ref = got
            assert float(ref[2].min()) < 0.1
        for a, b in zip(ref, got):
            assert torch.equal(a, b), cfg
