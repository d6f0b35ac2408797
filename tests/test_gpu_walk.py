"""The walks over a tile's key list at the sizes where they can go wrong:
list lengths around a staged batch (128 records) and a turn of the walk (4),
on images that are not whole blocks or tiles, against the FP64 oracle.

Bars: pixels max-abs 2e-4 and mean-abs 1e-5 with knife-edge pixels checked
against the oracle's reachable range, as in the parity tests."""
import numpy as np
import pytest

import oracle as O
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


def _stack_scene(n, seed, opacity=-3.0):
    """n faint, anisotropic Gaussians on the view axis: every pixel of a
    small image composites most of them without saturating."""
    r = np.random.default_rng(seed)
    means = np.zeros((n, 3), np.float32)
    means[:, :2] = r.normal(0, 0.25, (n, 2))
    means[:, 2] = r.uniform(-1, 1, n)
    lv = synth.Level(means, r.normal(-2.2, 0.7, (n, 3)).astype(np.float32),
                     r.normal(size=(n, 4)).astype(np.float32),
                     r.normal(opacity, 0.5, n).astype(np.float32),
                     r.normal(0, 0.3, (n, 16, 3)).astype(np.float32))
    return synth.Scene(levels=[lv], d_thresholds=np.zeros(0), chunk_centers=np.zeros((1, 3)))


@pytest.mark.parametrize("n,wh", [(1, (8, 8)), (3, (16, 16)), (4, (7, 9)), (5, (31, 17)), (127, (16, 16)),
                                  (128, (15, 16)), (129, (33, 16)), (131, (16, 40)), (256, (24, 24)),
                                  (257, (9, 23)), (1000, (40, 33))])
def test_list_lengths(env, n, wh):
    torch, api, ctx = env
    scene = _stack_scene(n, n)
    cam = synth.look_at((0.0, 0.0, -3.0), (0.0, 0.0, 1.0), (0.0, -1.0, 0.0), wh[0], wh[1], 30.0)
    osc = O.OracleScene(scene)
    ref = O.render(osc, cam, np.arange(n))
    sid = ctx.load_scene(scene)
    try:
        for log2 in (0, 1, 3):
            ctx.set_bin_size(log2)
            img, st = ctx.render(sid, api.FULL, cam)
            assert st["n_visible"] == ref["n_visible"] and st["n_keys"] == ref["n_keys"]
            O.compare_pixels(img.cpu().numpy(), ref, max_abs=2e-4, mean_abs=1e-5)
            saved, _, h = ctx.render(sid, api.FULL, cam, save=True)
            ctx.release(h)
            assert torch.equal(img, saved)
    finally:
        ctx.set_bin_size(-1)
        ctx.unload_scene(sid)


@pytest.mark.parametrize("n,wh", [(1, (8, 8)), (3, (16, 16)), (127, (15, 16)), (128, (33, 16)), (129, (16, 40)),
                                  (300, (9, 23))])
def test_gradients_of_list_lengths(env, n, wh):
    """The adjoint's walk on the same stacks: relative L2 error of every
    parameter group at most 1e-3 against the FP64 oracle (the bar of the
    gradient tests), and a non-finite image gradient reaches no record that
    its pixel does not composite."""
    torch, api, ctx = env
    from oracle import grad as G
    scene = _stack_scene(n, 50 + n, opacity=-1.0)
    lv = scene.levels[0]
    cam = synth.look_at((0.0, 0.0, -3.0), (0.0, 0.0, 1.0), (0.0, -1.0, 0.0), wh[0], wh[1], 30.0)
    w = np.random.default_rng(n).normal(size=(wh[1], wh[0], 3))
    g_ref, _ = G.grads(lv, cam, w)
    ps = [torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()
          for a in (lv.means, lv.log_scales, lv.quats, lv.opacity_logits, lv.sh.reshape(n, 48))]

    def grads(image_grad):
        _, _, h = ctx.render_params(*ps, cam, save=True)
        gs = [torch.zeros_like(p) for p in ps]
        ctx.render_backward(h, torch.from_numpy(image_grad.astype(np.float32)).cuda(), *gs)
        ctx.release(h)
        return gs

    for g, r in zip(grads(w), g_ref):
        r = np.asarray(r)
        e = np.linalg.norm(g.cpu().numpy().reshape(r.shape) - r) / max(np.linalg.norm(r), 1e-30)
        assert e < 1e-3
    w[0, 0] = np.inf
    alone = np.zeros_like(w)
    alone[0, 0] = 1.0
    touched = (grads(alone)[4].abs().sum(1) > 0)          # records that pixel (0, 0) composites
    hurt = ~torch.isfinite(grads(w)[4]).all(1)
    assert not (hurt & ~touched).any()


@pytest.mark.parametrize("n,wh", [(1, (8, 8)), (3, (16, 16)), (4, (7, 9)), (127, (15, 16)), (128, (33, 16)),
                                  (129, (16, 40)), (300, (9, 23))])
def test_importance_of_list_lengths(env, n, wh):
    """The scoring walk on the same stacks: every score within 2e-4 of the
    oracle's bracket (the bar of the importance tests), and the same for
    every bin size, whose lists hold the same records in the same order."""
    torch, api, ctx = env
    scene = _stack_scene(n, 90 + n, opacity=-1.0)
    cam = synth.look_at((0.0, 0.0, -3.0), (0.0, 0.0, 1.0), (0.0, -1.0, 0.0), wh[0], wh[1], 30.0)
    ref, clean = O.importance(O.OracleScene(scene), cam, np.arange(n))
    sid = ctx.load_scene(scene)
    try:
        scores = []
        for log2 in (0, 1, 3):
            ctx.set_bin_size(log2)
            scores.append(ctx.importance(sid, api.FULL, [cam]))
            s = scores[-1].cpu().numpy().astype(np.float64)
            assert (s >= np.minimum(clean, ref) - 2e-4).all() and (s <= ref + 2e-4).all()
            assert torch.equal(scores[-1], scores[0])
    finally:
        ctx.set_bin_size(-1)
        ctx.unload_scene(sid)
