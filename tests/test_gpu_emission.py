"""Key emission at the sizes where its tiles of depth-sorted records change
(32 records near, 256 or 1024 behind, a split emission above 2^21).  The key
list is compared whole, so the bars are exact."""
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
    yield torch, api, ctx
    ctx.close()


def _params(torch, n, seed, log_mean, big=0):
    """n Gaussians in front of the camera, the first `big` of them large."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    r = lambda *s: torch.randn(*s, generator=g, device="cuda")
    means = torch.rand(n, 3, generator=g, device="cuda") * 1.2 - 0.6
    logs = r(n, 3) * 0.3 + log_mean
    logs[:big] += 3.5
    return [means, logs, r(n, 4), r(n) - 1.0, r(n, 48) * 0.2]


def _cam(w, h):
    return synth.look_at((0.0, 0.0, -3.0), (0.0, 0.0, 1.0), (0.0, -1.0, 0.0), w, h, 40.0)


def _expected_keys(torch, rec, tiles_x):
    """(tile, depth) keys and gids of every record, sorted by tile, depth and
    record."""
    r = rec["rect"].long()
    w, cnt = r[:, 2] - r[:, 0] + 1, (r[:, 2] - r[:, 0] + 1) * (r[:, 3] - r[:, 1] + 1)
    who = torch.repeat_interleave(torch.arange(r.shape[0], device=r.device), cnt)
    k = torch.arange(who.numel(), device=r.device) - (cnt.cumsum(0) - cnt)[who]
    tile = (r[who, 1] + k // w[who]) * tiles_x + r[who, 0] + k % w[who]
    depth = rec["depth"].view(torch.int32).long()[who]      # positive: bits order as values
    o = torch.argsort(depth, stable=True)                   # records ascend already
    o = o[torch.argsort(tile[o], stable=True)]
    return ((tile << 32) | depth)[o], rec["gid"][who][o]


@pytest.mark.parametrize("n,big,log_mean,wh", [(1, 1, -2.5, (65, 33)), (31, 3, -2.5, (160, 96)), (33, 0, -3.0, (33, 200)),
                                               (4095, 40, -4.0, (320, 200)), (4096, 0, -4.0, (320, 200)),
                                               (4097, 4097, -6.0, (129, 65)), (4353, 300, -4.5, (640, 48)),
                                               (70_000, 50, -5.0, (333, 222)), (2_200_000, 60, -8.0, (400, 300))])
def test_key_lists(env, n, big, log_mean, wh):
    torch, api, ctx = env
    p = _params(torch, n, n, log_mean, big)
    cam = _cam(*wh)
    img, st, h = ctx.render_params(*p, cam, save=True)
    try:
        keys, gids = ctx.debug_keys(h)
        want, want_gid = _expected_keys(torch, ctx.debug_records(h), (wh[0] + 15) // 16)
    finally:
        ctx.release(h)
    assert st["n_keys"] == want.numel() == keys.numel()
    assert torch.equal(keys, want) and torch.equal(gids, want_gid)


@pytest.mark.parametrize("n", [33, 4097, 70_000])
def test_bins_and_lone_frames_agree(env, n):
    """Lone frames (their second call runs without a mid-frame sync) and the
    frames of a list, for every bin size, give the saved frame's image."""
    torch, api, ctx = env
    p = [t.cpu().numpy() for t in _params(torch, n, n, -4.5, 20)]
    sc = synth.Scene(levels=[synth.Level(p[0], p[1], p[2], p[3], p[4].reshape(n, 16, 3))], d_thresholds=np.zeros(0),
                     chunk_centers=np.zeros((1, 3)))
    cam = _cam(223, 131)
    sid = ctx.load_scene(sc)
    try:
        want, _, h = ctx.render(sid, api.FULL, cam, save=True)
        ctx.release(h)
        for log2 in (0, 1, 2, 3):
            ctx.set_bin_size(log2)
            for _ in range(3):
                assert torch.equal(ctx.render(sid, api.FULL, cam)[0], want)
            for img in ctx.render(sid, api.FULL, [cam] * 9)[0]:
                assert torch.equal(img, want)
    finally:
        ctx.set_bin_size(-1)
        ctx.unload_scene(sid)
