"""The repair network's persistent kernels over tile counts around their grids: one
tile, a CTA's second and later tiles, CTAs with unequal shares.

A tile's result does not depend on the list around it, so the gate logits and fills of
a list that repeats tiles equal those of each tile listed once, bit for bit. A training
batch that repeats every tile 4 or 16 times has the same mean loss: every output
gradient is scaled by an exact power of two, so only the order of the FP32 sums differs.
An accumulator takes at most 6 x 46 MMAs and 152 partials, each with a relative error
of 2^-22 of the largest partial sum: 1e-4 of it; 1e-3 of a layer's largest gradient
leaves room for cancellation.
"""
import numpy as np
import pytest

from oracle import repair as R

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

H, W = 91, 125  # 6 x 8 tiles, ragged at both edges


@pytest.fixture(scope="module")
def net():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_30741_gb300 import build, gs
    build.build()
    rng = np.random.default_rng(3)
    Wt, b = R.init_weights(3)
    b = [rng.normal(0, 0.05, bb.shape) for bb in b]
    ctx = gs.Context(16, W, H, max_instances=1 << 12)
    ctx.repair_load(R.pack(Wt, b).astype(np.float32).astype(np.float64))
    f = np.zeros((1, H, W, 8), np.float32)
    f[..., :6] = rng.random((1, H, W, 6))
    f[..., 4] = rng.random((1, H, W)) < 0.3
    feat = torch.tensor(f).to(torch.bfloat16).cuda()
    tiles = torch.tensor([(y << 12) | x for y in range(6) for x in range(8)], dtype=torch.int32, device="cuda")
    ctx.repair_calibrate_fp8(feat, tiles)
    return ctx, feat, tiles


@pytest.mark.parametrize("fp8", [False, True])
@pytest.mark.parametrize("n", [1, 2, 151, 153, 304, 305, 1000])
def test_tiles_do_not_depend_on_their_place(net, n, fp8):
    ctx, feat, tiles = net
    one_fill = torch.zeros(1, 3, H, W, device="cuda")
    _, one = ctx.repair_infer(feat, tiles, fill=one_fill, fp8=fp8)
    pick = (torch.arange(n, device="cuda") * 7) % tiles.numel()
    fill = torch.full((1, 3, H, W), -7.0, device="cuda")
    _, gate = ctx.repair_infer(feat, tiles[pick].contiguous(), fill=fill, fp8=fp8)
    ctx.check_ok()
    assert torch.equal(gate, one[pick])
    listed = torch.zeros(tiles.numel(), dtype=torch.bool, device="cuda")
    listed[pick] = True
    px = listed.view(6, 8).repeat_interleave(16, 0).repeat_interleave(16, 1)[:H, :W]
    assert torch.equal(fill[0][:, px], one_fill[0][:, px])
    assert torch.all(fill[0][:, ~px] == -7.0)


@pytest.mark.parametrize("times", [4, 16])
def test_repeated_batches_give_the_same_gradient(net, times):
    ctx, feat, tiles = net
    target = torch.full((1, 3, H, W), 10.0, device="cuda")

    def grad(t):
        # a scratch full of NaN: only what the step itself wrote may be read
        scratch = ctx.repair_scratch(t.numel())
        scratch.fill_(0xFF)
        ctx.repair_train_step(feat, target, target.clone(), t, scratch=scratch, lr=0.0, gate_weight=0.1)
        ctx.check_ok()
        return ctx.repair_read(1).astype(np.float64)

    g1, gn = grad(tiles), grad(tiles.repeat(times).contiguous())
    o = 0
    for l in range(6):
        n = R.CHANNELS[l + 1] * (9 * R.CHANNELS[l] + 1)
        a, b = g1[o:o + n], gn[o:o + n]
        assert np.isfinite(b).all() and np.abs(a).max() > 0
        assert np.abs(a - b).max() <= 1e-3 * np.abs(a).max(), l
        o += n
