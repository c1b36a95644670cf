"""GPU SSIM (gs_ssim) of images that differ little, against the FP64 oracle.

With d the images' difference the map is (1 - D^2 / (..)) (1 - vd / (..)): d^2 is at most
1e-6 here, so the rounding of the filters (22 FP32 steps, 2^-19 relative) moves a map
value by less than 1e-8, and what is left is the rounding of the map's own seven
operations and of the result: 8 x 2^-24 in all.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 8 * 2.0 ** -24


@pytest.fixture(scope="module")
def gs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_30741_gb300 import build
    build.build()
    from paper_2609_30741_gb300 import gs as gsmod
    return gsmod


@pytest.mark.parametrize("noise", [1e-4, 1e-3])
@pytest.mark.parametrize("kind", ["white", "bright", "grey"])
@pytest.mark.parametrize("shape", [(3, 37, 53), (1, 240, 321)])
def test_ssim_of_close_images(gs, shape, kind, noise):
    from oracle import metrics
    rng = np.random.default_rng(shape[1])
    x = {"white": np.ones(shape), "bright": 0.9 + 0.1 * rng.random(shape), "grey": np.full(shape, 0.5)}[kind]
    y = x + noise * np.clip(rng.standard_normal(shape), -3.0, 3.0)
    a, b = (torch.tensor(v, dtype=torch.float32, device="cuda") for v in (x, y))
    ctx = gs.Context(16, 512, 512, max_instances=1 << 12)
    want = metrics.ssim(a.double().cpu().numpy(), b.double().cpu().numpy())
    for p, q in ((a, b), (b, a)):
        assert abs(float(ctx.ssim(p, q)) - want) <= TOL, (float(ctx.ssim(p, q)), want)
    assert float(ctx.ssim(b, b)) == 1.0


@pytest.mark.parametrize("noise", [1e-4, 1e-3])
@pytest.mark.parametrize("shape", [(3, 37, 53), (3, 1199, 1599)])
def test_ssim_next_to_one_is_rounded_once(gs, shape, noise):
    """Uniform noise in [0, 1] and a copy with a little more: 1 - SSIM is below 1e-5, of
    which 2^-16 is the most the filters' rounding makes (22 steps of 2^-24 on squares up to 4
    against a variance of 0.3), and the result is rounded to a float once."""
    from oracle import metrics
    rng = np.random.default_rng(shape[2])
    x = rng.random(shape)
    y = x + noise * np.clip(rng.standard_normal(shape), -3.0, 3.0)
    a, b = (torch.tensor(v, dtype=torch.float32, device="cuda") for v in (x, y))
    ctx = gs.Context(16, 1600, 1200, max_instances=1 << 12)
    want = metrics.ssim(a.double().cpu().numpy(), b.double().cpu().numpy())
    assert 0.0 < 1.0 - want < 1e-5
    for p, q in ((a, b), (b, a)):
        assert abs(float(ctx.ssim(p, q)) - want) <= 2.0 ** -25 + 1e-5 * 2.0 ** -16


@pytest.mark.parametrize("size", [(480, 640), (1079, 1919)])
def test_window_weights_sum_to_one(gs, size):
    """A smooth image and a noisy copy. A window that sums to 1 - e adds e A^2 to every
    variance, 1.6e-7 of the SSIM for the weights' own rounding; without it what is left is
    the result's rounding (2^-25) and the mean of the map's, far below as much again."""
    from oracle import metrics
    h, w = size
    v, u = np.mgrid[:h, :w] / 24.0
    rng = np.random.default_rng(h)
    x = np.stack([0.5 + 0.2 * np.cos(u + c) + 0.2 * np.sin(0.7 * v - c) for c in range(3)])
    y = x + 0.05 * rng.standard_normal(x.shape)
    a, b = (torch.tensor(t, dtype=torch.float32, device="cuda") for t in (x, y))
    ctx = gs.Context(16, w, h, max_instances=1 << 12)
    want = metrics.ssim(a.double().cpu().numpy(), b.double().cpu().numpy())
    assert abs(float(ctx.ssim(a, b)) - want) <= 2.0 ** -24, (float(ctx.ssim(a, b)), want)
