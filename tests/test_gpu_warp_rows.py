"""The allocation-free warp (gs_warp_noalloc) on rigs of both its paths: one CTA per
image row when every sample keeps its row, else a scatter to the whole image.

Both paths run the same float32 operations in the same order, every one of them rounded
as IEEE 754 asks (a fused multiply-add once), so the reference below, which repeats them
one by one and takes the nearest sample of every destination pixel, must agree bit for
bit. An extended-precision product and sum rounded to float32 differs from the fused
operation only when the extended result lies within 2^-11 (2^-60 for quadruple) of an
ulp of a rounding boundary AND the landing pixel or the winner depends on that last bit;
the seeds are fixed, and none of these inputs has such a pixel.
"""
import math

import numpy as np
import pytest

from paper_2609_30741_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

F = np.float32
Z_NEAR = F(0.2)
INF_BITS = 0x7F800000


@pytest.fixture(scope="module")
def gs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_30741_gb300 import build
    build.build()
    from paper_2609_30741_gb300 import gs as gsmod
    return gsmod


def _fma(a, b, c):
    return (a.astype(np.longdouble) * np.longdouble(b) + np.asarray(c, np.longdouble)).astype(F)


def _relative(dom, aff):
    """X_aff = R_aff^T R_dom X_dom + R_aff^T (t_dom - t_aff)."""
    L = np.longdouble
    R = (aff.R.astype(L).T @ dom.R.astype(L)).astype(np.float64)
    t = (aff.R.astype(L).T @ (dom.t - aff.t).astype(L)).astype(np.float64)
    return R, t


def _reference(depth, trans, dom, aff, cam):
    """(hole mask, winning source index, winner's depth) of every destination pixel."""
    H, W = cam.height, cam.width
    Rd, td = _relative(dom, aff)
    R, t = Rd.astype(F), td.astype(F)
    fx, fy, cx, cy = F(cam.fx), F(cam.fy), F(cam.cx), F(cam.cy)
    y, x = (v.astype(F) for v in np.meshgrid(np.arange(H), np.arange(W), indexing="ij"))
    with np.errstate(all="ignore"):
        cov = F(1) - trans
        surf = cov >= F(0.5)
        d = np.where(surf, depth / cov, F(0)).astype(F)
        rx, ry = ((x - cx) / fx).astype(F), ((y - cy) / fy).astype(F)

        def row(i):
            s = _fma(rx * d, R[i, 0], _fma(ry * d, R[i, 1], _fma(d, R[i, 2], t[i])))
            b = _fma(rx, R[i, 0], _fma(ry, R[i, 1], R[i, 2]))
            return np.where(surf, s, b).astype(F)
        X, Y, Z = row(0), row(1), row(2)
        u = np.floor((_fma((X / Z).astype(F), fx, cx) + F(0.5)).astype(F))
        v = np.floor((_fma((Y / Z).astype(F), fy, cy) + F(0.5)).astype(F))
        ok = (Z > np.where(surf, Z_NEAR, F(0))) & (u >= 0) & (u <= W - 1) & (v >= 0) & (v <= H - 1)
    src = np.arange(H * W, dtype=np.uint64).reshape(H, W)
    zb = np.where(surf, np.ascontiguousarray(Z).view(np.uint32), np.uint32(INF_BITS)).astype(np.uint64)
    key = np.full(H * W, np.iinfo(np.uint64).max, np.uint64)
    dst = (v[ok].astype(np.int64) * W + u[ok].astype(np.int64))
    np.minimum.at(key, dst, ((zb << np.uint64(32)) | src)[ok])
    hole = key == np.iinfo(np.uint64).max
    win = (key & np.uint64(0xFFFFFFFF)).astype(np.int64)
    zdep = (key >> np.uint64(32)).astype(np.uint32).view(F)
    return hole.reshape(H, W), np.where(hole, 0, win).reshape(H, W), np.where(hole, F(0), zdep).reshape(H, W)


def _inputs(H, W, seed):
    """Depth steps with noise, background, half covered and empty pixels."""
    r = np.random.default_rng(seed)
    z = 0.8 + 0.7 * r.integers(0, 4, (H, W // 9 + 1)).repeat(9, 1)[:, :W] + 0.01 * r.random((H, W))
    T = np.where(r.random((H, W)) < 0.15, 1.0, 0.05 * r.random((H, W)))
    T = np.where(r.random((H, W)) < 0.05, 0.5, T).astype(F)
    D = (z * (1.0 - T)).astype(F)
    D[r.random((H, W)) < 0.02] = 0.0
    return r.random((3, H, W)).astype(F), D, T


def _check(gs, cam, dom, aff, seed=1):
    H, W = cam.height, cam.width
    rgb, D, T = _inputs(H, W, seed)
    hole, win, dep = _reference(D, T, dom, aff, cam)
    g = [torch.tensor(v, device="cuda") for v in (rgb, D, T)]
    out = torch.full((3, H, W), -1.0, device="cuda")
    dw = torch.full((H, W), -1.0, device="cuda")
    hw = torch.full((H, W), 7, dtype=torch.uint8, device="cuda")
    gs.warp_noalloc(*g, dom, aff, cam, out, dw, hw)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(hw.cpu().numpy().astype(bool), hole)
    np.testing.assert_array_equal(dw.cpu().numpy(), dep)
    want = np.where(hole[None], F(0), rgb.reshape(3, -1)[:, win.ravel()].reshape(3, H, W))
    np.testing.assert_array_equal(out.cpu().numpy(), want)
    return hole


def _rot(axis, angle):
    c, s = math.cos(angle), math.sin(angle)
    return {"x": np.array([[1, 0, 0], [0, c, -s], [0, s, c]]), "y": np.array([[c, 0, s], [0, 1, 0], [-s, 0, c]]),
            "z": np.array([[c, -s, 0], [s, c, 0], [0, 0, 1]])}[axis].astype(float)


def _pair(kind):
    head = synth.look_at([0.05, -0.02, 0.1], [0.0, 0.0, 2.5])
    dom, aff = synth.eye_pair(head)
    t = {"parallel": aff.t, "vertical": dom.t + 0.05 * dom.R[:, 1], "forward": dom.t + 0.05 * dom.R[:, 2]}
    if kind in t:
        return dom, synth.Pose(dom.R.copy(), t[kind])
    if kind == "toed_in":
        return (synth.Pose(dom.R @ _rot("y", 0.02), dom.t), synth.Pose(aff.R @ _rot("y", -0.02), aff.t))
    return dom, synth.Pose(aff.R @ _rot("z", 0.01), aff.t)  # rolled


@pytest.mark.parametrize("kind", ["parallel", "toed_in", "vertical", "forward", "rolled"])
@pytest.mark.parametrize("size", [(97, 61), (1, 33), (257, 1), (1025, 3)])
def test_rigs_that_keep_rows_and_rigs_that_do_not(gs, kind, size):
    dom, aff = _pair(kind)
    _check(gs, synth.centred_camera(size[0], size[1], 90.0), dom, aff, seed=size[0])


@pytest.mark.parametrize("W", [6144, 6145, 8190])
def test_widths_around_the_shared_memory_of_a_row(gs, W):
    """A row's winners fit the default shared memory up to 6144 columns; wider images scatter."""
    dom, aff = _pair("parallel")
    hole = _check(gs, synth.centred_camera(W, 5, 5000.0), dom, aff)
    assert 0.0 < hole.mean() < 0.9


@pytest.mark.parametrize("share", [0.5, 0.999, 1.001, 2.0])
def test_both_sides_of_the_row_bound(gs, share):
    """The affiliated eye pitched by `share` of the angle at which a sample may leave its
    quarter of a pixel: fy (e1 + ry e2) / (1 - e2) = 0.25 with e1 = |sin| + (1 - cos) ry,
    e2 = |sin| ry + (1 - cos) for a centred camera."""
    cam = synth.centred_camera(130, 77, 210.0)
    ry = 0.5 * (cam.height - 1) / cam.fy

    def off(a):
        s, c = math.sin(a), 1 - math.cos(a)
        e1, e2 = s + c * ry, s * ry + c
        return cam.fy * (e1 + ry * e2) / (1 - e2)
    lo, hi = 0.0, 0.01
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if off(mid) < 0.25 else (lo, mid)
    dom, aff = synth.eye_pair(synth.identity_pose())
    _check(gs, cam, dom, synth.Pose(aff.R @ _rot("x", share * lo), aff.t))


@pytest.mark.parametrize("case", [("principal point", 96, 64, 3.0e7), ("height", 3, 1 << 20, None)])
def test_rows_that_float32_cannot_keep(gs, case):
    """Image rows whose projected coordinate float32 rounds by a quarter of a pixel and
    more: the samples land where the rounding puts them, as in the scatter."""
    _, W, H, cy = case
    cam = synth.centred_camera(W, H, 300.0)
    if cy is not None:
        cam.cy = cy
    dom, aff = synth.eye_pair(synth.identity_pose())
    _check(gs, cam, dom, aff)
