"""The compositing's walk, which skips per 8x8 block of pixels the records that
cannot reach it, against a walk that visits every record of the tile's list at
every pixel (lodge_debug_composite): plain frames for every bin size, and
frames kept for the adjoint, whose lists the adjoint and the scoring walk
filter the same way.  The bar is equality of every bit."""
import numpy as np
import pytest

from paper_2505_23158_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_23158_gb300 import build
    build.build()
    from paper_2505_23158_gb300 import api
    ctx = api.Lodge(0)
    yield torch, ctx
    ctx.close()


def _params(torch, lv):
    return [torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()
            for a in (lv.means, lv.log_scales, lv.quats, lv.opacity_logits, lv.sh.reshape(lv.n, 48))]


def _check(torch, ctx, ps, cam):
    saved, st, h = ctx.render_params(*ps, cam, save=True)
    want = ctx.debug_composite(h, cam.height, cam.width)
    ctx.release(h)
    assert torch.equal(saved, want)
    try:
        for log2 in (0, 1, 2, 3):
            ctx.set_bin_size(log2)
            assert torch.equal(ctx.render_params(*ps, cam)[0], want), f"bins {log2}"
    finally:
        ctx.set_bin_size(-1)
    return want, st


def test_plain_scene(env):
    torch, ctx = env
    scene, cams = synth.workload_plain(0)
    for cam in cams[:2]:
        _check(torch, ctx, _params(torch, scene.levels[0]), cam)


def test_outdoor_scene(env):
    torch, ctx = env
    scene, cams = synth.workload_outdoor(seed=3, n_poses=6, scale=0.01, width=331, height_px=187)
    for cam in cams[:3]:
        _check(torch, ctx, _params(torch, scene.levels[0]), cam)


@pytest.mark.parametrize("seed,wh", [(0, (64, 48)), (1, (37, 61)), (2, (1600, 24)), (3, (20000, 17))])
def test_thin_rotated_splats_at_the_threshold(env, seed, wh):
    """Splats from a pixel to thousands of pixels long, hair-thin, at every
    angle, centred on and off the image, most of them just above opacity
    1/255."""
    torch, ctx = env
    r = np.random.default_rng(seed)
    n = 3000
    cam = synth.look_at((0.0, 0.0, 0.0), (0.0, 0.0, 1.0), (0.0, -1.0, 0.0), wh[0], wh[1], 60.0)
    z = r.uniform(1.0, 20.0, n)
    half = 0.6 * np.array(wh) / cam.fx
    means = np.stack([r.uniform(-half[0], half[0], n) * z, r.uniform(-half[1], half[1], n) * z, z], 1)
    long_axis = np.exp(r.uniform(np.log(0.5), np.log(3000.0), n)) * z / cam.fx
    logs = np.log(np.stack([long_axis, long_axis * np.exp(r.uniform(-9, 0, n)), long_axis * 1e-3], 1))
    th = r.uniform(0, np.pi, n)
    quats = np.stack([np.cos(th / 2), 0 * th, 0 * th, np.sin(th / 2)], 1) + r.normal(0, 1e-3, (n, 4))
    o = np.exp(r.uniform(np.log(1.0005 / 255), np.log(0.05), n))
    lv = synth.Level(means.astype(np.float32), logs.astype(np.float32), quats.astype(np.float32),
                     np.log(o / (1 - o)).astype(np.float32), r.normal(0, 0.3, (n, 16, 3)).astype(np.float32))
    img, st = _check(torch, ctx, _params(torch, lv), cam)
    assert st["n_visible"] > n // 4 and float(img.max()) > 0.05


@pytest.mark.parametrize("seed,pixels", [(4, (3e3, 3e4)), (5, (3e4, 1e6)), (6, (1e6, 3e7))])
def test_splats_that_reach_the_image_from_afar(env, seed, pixels):
    """Splats of up to 3e7 pixels, a few pixels wide, whose means lie up to two
    standard deviations off the image along their long axis: the terms of the
    exponent are then far larger than the exponent, and its rounding larger
    than any fixed margin."""
    torch, ctx = env
    r = np.random.default_rng(seed)
    n, w, h = 4000, 61, 45
    cam = synth.look_at((0.0, 0.0, 0.0), (0.0, 0.0, 1.0), (0.0, -1.0, 0.0), w, h, 60.0)
    R, t = np.asarray(cam.R, np.float64), np.asarray(cam.t, np.float64)
    sigma = np.exp(r.uniform(*np.log(pixels), n))           # standard deviation along the axis, pixels
    th = r.uniform(0, np.pi, n)
    along = r.uniform(-2.0, 2.0, n) * sigma
    px = r.uniform(0, w, n) + along * np.cos(th)
    py = r.uniform(0, h, n) + along * np.sin(th)
    z = r.uniform(1.0, 3.0, n)
    p = np.stack([(px - cam.cx) / cam.fx * z, (py - cam.cy) / cam.fy * z, z], 1)
    means = (p - t) @ R
    axis = np.stack([np.cos(th), np.sin(th), 0 * th], 1) @ R    # in the image plane: world direction
    phi = np.arctan2(axis[:, 1], axis[:, 0])
    assert np.abs(axis[:, 2]).max() < 1e-6                      # the camera looks along z
    logs = np.log(np.stack([sigma, np.exp(r.uniform(np.log(0.01), np.log(3), n)), np.full(n, 1e-3)], 1)
                  * (z / cam.fx)[:, None])
    quats = np.stack([np.cos(phi / 2), 0 * phi, 0 * phi, np.sin(phi / 2)], 1)
    o = np.exp(r.uniform(np.log(1.02 / 255), np.log(5 / 255), n))
    lv = synth.Level(means.astype(np.float32), logs.astype(np.float32), quats.astype(np.float32),
                     np.log(o / (1 - o)).astype(np.float32), r.normal(0, 0.3, (n, 16, 3)).astype(np.float32))
    img, st = _check(torch, ctx, _params(torch, lv), cam)
    assert st["n_visible"] > n // 4 and float(img.max()) > 0.05
