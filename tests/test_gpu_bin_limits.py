"""The binning's capacities at their edges. A tile list holds every surfel that reaches
one of the tile's pixel centres, whatever the tile edge, so images at 8- and 32-pixel
tiles are equal bit for bit as long as every instance and span fits.
"""
import numpy as np
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


def _discs(n, scale, seed=1):
    """n nearly frontal discs in front of the camera, thin enough in opacity to be blended on."""
    r = np.random.default_rng(seed)
    pos = np.zeros((n, 4), np.float32)
    pos[:, :2] = r.uniform(-0.3, 0.3, (n, 2))
    pos[:, 2] = r.uniform(2.0, 3.0, n)
    quat = np.tile(np.array([1, 0, 0, 0], np.float32), (n, 1)) + 0.05 * r.standard_normal((n, 4)).astype(np.float32)
    quat /= np.linalg.norm(quat, axis=1, keepdims=True)
    sh = r.uniform(-1, 1, (n, 1, 3)).astype(np.float32)
    return synth.Scene(pos, quat.astype(np.float32), np.full((n, 2), scale, np.float32),
                       np.full(n, 0.05, np.float32), sh, 0)


def _images(gs, ctx, ds, cam, cfg):
    ctx.set_raster(*cfg)
    out = ctx.render_mono(ds, synth.identity_pose(), cam, bg=(0.1, 0.2, 0.3))
    ctx.check_ok()
    return [t.clone() for t in out]


def test_large_surfels_at_small_tiles(gs):
    """A hundred surfels over 64 bands of four 8-pixel tile rows each."""
    scene, cam = _discs(100, 2.0), synth.centred_camera(1920, 2048, 1500.0)
    ds = gs.DeviceScene(scene)
    ctx = gs.Context(scene.n, cam.width, cam.height, max_instances=1 << 23, min_tile=8)
    small = _images(gs, ctx, ds, cam, (8, 2, 64))
    assert ctx.usage()["band_entries"][0] > 60 * scene.n
    for a, b in zip(small, _images(gs, ctx, ds, cam, (32, 2, 64))):
        assert torch.equal(a, b)


def test_tall_image_at_the_most_tile_rows(gs):
    """8192 rows at 8-pixel tiles: 1024 tile rows, the row lists' largest shared memory."""
    scene, cam = _discs(400, 0.02), synth.centred_camera(65, 8192, 6000.0)
    ds = gs.DeviceScene(scene)
    ctx = gs.Context(scene.n, cam.width, cam.height, max_instances=1 << 20, min_tile=8)
    small = _images(gs, ctx, ds, cam, (8, 1, 32))
    assert float(small[2].min()) < 1.0 - 0.04  # surfels of opacity 0.05 were blended
    for a, b in zip(small, _images(gs, ctx, ds, cam, (32, 2, 64))):
        assert torch.equal(a, b)


@pytest.mark.parametrize("kind", ["discs", "mixed"])
def test_capacity_of_exactly_the_reported_counts(gs, kind):
    """A context of max(instances, spans) renders the frame; one instance less does not."""
    cam = synth.centred_camera(333, 257, 300.0)
    scene = _discs(60, 0.6) if kind == "discs" else synth.random_scene(5, 3000)
    ds = gs.DeviceScene(scene)
    big = gs.Context(scene.n, cam.width, cam.height, max_instances=1 << 22, min_tile=8)
    want = _images(gs, big, ds, cam, (8, 2, 64))
    u = big.usage()
    need = max(u["instances"][0], u["spans"][0])
    ctx = gs.Context(scene.n, cam.width, cam.height, max_instances=need, max_instances_aff=1, min_tile=8,
                     paths=gs.PATH_MONO)
    for a, b in zip(want, _images(gs, ctx, ds, cam, (8, 2, 64))):
        assert torch.equal(a, b)
    less = gs.Context(scene.n, cam.width, cam.height, max_instances=need - 1, max_instances_aff=1, min_tile=8,
                      paths=gs.PATH_MONO)
    with pytest.raises(gs.GsError) as e:
        _images(gs, less, ds, cam, (8, 2, 64))
    assert e.value.status == gs.GS_ERR_CAPACITY
