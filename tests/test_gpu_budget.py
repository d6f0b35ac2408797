"""Device memory of the frame calls: what a frame's scratch holds, and calls
on several streams in a context whose memory holds one stream's scratch."""
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


def _scene(n, seed=0, log_scale=-5.5):
    """n small Gaussians in front of _cam, all visible."""
    r = np.random.default_rng(seed)
    lv = synth.Level(r.uniform(-0.8, 0.8, (n, 3)).astype(np.float32),
                     r.normal(log_scale, 0.3, (n, 3)).astype(np.float32), r.normal(size=(n, 4)).astype(np.float32),
                     r.normal(0, 0.5, n).astype(np.float32), r.normal(0, 0.2, (n, 16, 3)).astype(np.float32))
    return synth.Scene(levels=[lv], d_thresholds=np.zeros(0), chunk_centers=np.zeros((1, 3)))


def _cam(w, h, shift=0.0):
    return synth.look_at((shift, 0.0, -3.0), (0.0, 0.0, 1.0), (0.0, -1.0, 0.0), w, h, 50.0)


def test_scratch_of_a_frame(env):
    """A frame of small splats holds its records, its sorts and its keys, with
    the quarter that growing buffers keep in hand, and nothing per record that
    its emission does not read."""
    torch, api = env
    n = 300_000
    with api.Lodge(0) as ctx:
        sid = ctx.load_scene(_scene(n))
        ctx.set_bin_size(0)
        before = ctx.residency_stats()["hbm_used"]
        for _ in range(2):   # with and without a mid-frame sync
            _, st = ctx.render(sid, api.FULL, _cam(320, 240))
        used = ctx.residency_stats()["hbm_used"] - before
    assert st["n_visible"] == n and st["n_keys"] < 8 * n
    cap = st["n_keys"] + st["n_keys"] // 2 + 65536      # the key capacity a slot keeps
    record = 16 + 16 + 4 + 8 + 4                        # two halves, blue, rect, gid
    depth = 4 * 4 + 4                                   # keys and records twice, look-back words of 4 passes
    key = 4 * 2 + 2                                     # packed twice, look-back words of at most 2 passes
    assert used <= 1.25 * ((record + depth) * n + key * cap) + (1 << 20)


@pytest.mark.parametrize("call", ["importance", "importance_chunk", "full", "chunk_blend", "lod"])
def test_several_streams_in_the_memory_of_one(env, call):
    """A list of cameras in a context whose budget holds the scene and the
    scratch of one frame at a time: the images and scores are those of the
    cameras one by one."""
    torch, api = env
    scene, cams = synth.workload_outdoor(seed=6, n_poses=40, scale=0.05, width=320, height_px=180)
    cams = cams[::4]
    mode = {"importance": api.FULL, "full": api.FULL, "lod": api.LOD}.get(call, api.CHUNK_BLEND)

    def run(ctx, sid, cs):
        if call == "importance":
            return ctx.importance(sid, mode, cs)
        if call == "importance_chunk":
            return ctx.importance(sid, api.CHUNK, cs, chunk=1)
        out = torch.empty(len(cs), 180, 320, 3, device="cuda")
        return torch.stack(ctx.render(sid, mode, cs, out=out.view(-1))[0])

    with api.Lodge(0) as ctx:
        sid = ctx.load_scene(scene)
        want = [run(ctx, sid, [c]) for c in cams for _ in range(2)][::2]
        alone = ctx.residency_stats()["hbm_used"]
        run(ctx, sid, cams)
        assert ctx.residency_stats()["hbm_used"] > 1.05 * alone    # several streams hold more
    want = torch.stack(want).amax(0) if call.startswith("importance") else torch.cat(want)
    budget = alone + (1 << 16)
    with api.Lodge(0, hbm_budget_bytes=budget) as ctx:
        sid = ctx.load_scene(scene)
        for _ in range(2):
            assert torch.equal(run(ctx, sid, cams), want)
            assert ctx.residency_stats()["hbm_used"] <= budget


def test_scratch_left_behind_is_given_back(env):
    """The scratch that a call over several views leaves on its streams' slots
    yields to what the context needs next."""
    torch, api = env
    a, b = _scene(60_000), _scene(200_000, seed=1)
    cams = [_cam(160, 120, 0.05 * i) for i in range(6)]
    with api.Lodge(0) as ctx:
        sid = ctx.load_scene(a)
        base = ctx.residency_stats()["hbm_used"]
        want = torch.stack([ctx.importance(sid, api.FULL, [c]) for c in cams for _ in range(2)]).amax(0)
        one = ctx.residency_stats()["hbm_used"]
        ctx.importance(sid, api.FULL, cams)
        several = ctx.residency_stats()["hbm_used"]
        ctx.load_scene(b)
        scene_b = ctx.residency_stats()["hbm_used"] - several
    assert several - one < 0.9 * scene_b                    # the budget below holds the slots' scratch at first
    with api.Lodge(0, hbm_budget_bytes=one + int(1.05 * scene_b)) as ctx:
        sid = ctx.load_scene(a)
        assert torch.equal(ctx.importance(sid, api.FULL, cams), want)
        assert ctx.residency_stats()["hbm_used"] > base + 1.5 * (one - base)
        ctx.load_scene(b)
        assert torch.equal(ctx.importance(sid, api.FULL, cams), want)
