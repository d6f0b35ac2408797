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
