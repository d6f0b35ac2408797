"""Emission paths that take other frames than the key-list tests: one warp per
record (32 keys a record or more), the count / scan / write launches with the
counts on the device below their capacities, and scoring views that outgrow
their slot's key capacity.  The bars are equality."""
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
    return torch, api


def _cam(w, h, position=(0.0, 0.0, -3.0), forward=(0.0, 0.0, 1.0)):
    return synth.look_at(position, forward, (0.0, -1.0, 0.0), w, h, 40.0)


def _level(n, seed, log_scale, lo, hi):
    r = np.random.default_rng(seed)
    return synth.Level(r.uniform(lo, hi, (n, 3)).astype(np.float32),
                       (r.normal(0, 0.3, (n, 3)) + log_scale).astype(np.float32),
                       r.normal(size=(n, 4)).astype(np.float32), r.normal(-1, 1, n).astype(np.float32),
                       r.normal(0, 0.2, (n, 16, 3)).astype(np.float32))


def _scene(lv):
    return synth.Scene(levels=[lv], d_thresholds=np.zeros(0), chunk_centers=np.zeros((1, 3)))


@pytest.mark.parametrize("n,wh", [(1, (641, 479)), (7, (333, 222)), (33, (641, 479)), (300, (500, 500))])
def test_records_of_many_keys(env, n, wh):
    """A saved frame of screen-filling splats takes one warp per record; its
    key list holds every tile of every record's rect in depth order."""
    torch, api = env
    lv = _level(n, n, 0.0, -0.3, 0.3)
    with api.Lodge(0) as ctx:
        sid = ctx.load_scene(_scene(lv))
        img, st, h = ctx.render(sid, api.FULL, _cam(*wh), save=True)
        keys, gids = ctx.debug_keys(h)
        rec = ctx.debug_records(h)
        want_img = ctx.debug_composite(h, wh[1], wh[0])
        ctx.release(h)
        plain = ctx.render(sid, api.FULL, _cam(*wh))[0]
    assert st["n_visible"] == n and st["n_keys"] >= 32 * n
    tiles_x = (wh[0] + 15) // 16
    want = []
    for r, d, g in zip(rec["rect"].tolist(), rec["depth"].view(torch.int32).tolist(), rec["gid"].tolist()):
        want += [(y * tiles_x + x, d, g) for y in range(r[1], r[3] + 1) for x in range(r[0], r[2] + 1)]
    want.sort()                                      # depths are positive: bits order as values
    assert [(k >> 32, k & 0xFFFFFFFF, g) for k, g in zip(keys.tolist(), gids.tolist())] == want
    assert torch.equal(img, want_img) and torch.equal(plain, want_img)


def test_split_emission_with_device_counts(env):
    """Frames of more than 2^21 Gaussians, half of them behind the camera: the
    first waits for its counts, the later ones leave them on the device."""
    torch, api = env
    n = (1 << 21) + 4321
    lv = _level(n, 5, -7.5, (-1.0, -1.0, -7.0), (1.0, 1.0, 1.0))
    cam = _cam(400, 300)
    with api.Lodge(0) as ctx:
        sid = ctx.load_scene(_scene(lv))
        _, st, h = ctx.render(sid, api.FULL, cam, save=True)
        want = ctx.debug_composite(h, 300, 400)
        ctx.release(h)
        assert n // 4 < st["n_visible"] < 3 * n // 4
        for _ in range(3):
            img, s = ctx.render(sid, api.FULL, cam)
            assert torch.equal(img, want) and s["n_keys"] == st["n_keys"]
        for img in ctx.render(sid, api.FULL, [cam] * 9)[0]:
            assert torch.equal(img, want)


@pytest.mark.parametrize("views", [2, 5, 9])
def test_scores_of_views_that_outgrow_their_capacity(env, views):
    """Views that see nothing size their slots' key capacity small; the views
    behind them outgrow it, raise no score and are rendered again."""
    torch, api = env
    lv = _level(60_000, 9, -3.0, -1.0, 1.0)
    away = _cam(400, 300, forward=(0.0, 0.0, -1.0))
    cams = [_cam(400, 300, position=(0.1 * i, 0.0, -3.0)) for i in range(views)]
    with api.Lodge(0) as ctx:
        sid = ctx.load_scene(_scene(lv))
        want = torch.stack([ctx.importance(sid, api.FULL, [c]) for c in cams]).amax(0)
        assert int((want > 0).sum()) > 1000
    with api.Lodge(0) as ctx:
        sid = ctx.load_scene(_scene(lv))
        ctx.profile_enable()
        assert torch.equal(ctx.importance(sid, api.FULL, [away] * 4 + cams), want)
        assert ctx.profile_read()["redone"] > 0
        ctx.profile_enable(False)
        assert torch.equal(ctx.importance(sid, api.FULL, [away] * 4 + cams), want)
