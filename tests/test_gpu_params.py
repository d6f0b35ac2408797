"""The parameter path (raw arrays read in place, the adjoint's staged rows) at
the sizes of a warp, with levels beside the trained one and at both
alignments of the SH gradients."""
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


def _params(torch, n, seed, log_mean):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    r = lambda *s: torch.randn(*s, generator=g, device="cuda")
    means = torch.rand(n, 3, generator=g, device="cuda") * 1.2 - 0.6
    logs = r(n, 3) * 0.3 + log_mean
    return [means, logs, r(n, 4), r(n) - 1.0, r(n, 48) * 0.2]


def _cam(w, h):
    return synth.look_at((0.0, 0.0, -3.0), (0.0, 0.0, 1.0), (0.0, -1.0, 0.0), w, h, 40.0)


@pytest.mark.parametrize("n,degree", [(1, 3), (31, 2), (32, 1), (33, 0), (129, 3)])
def test_parameter_levels_and_gradient_alignment(env, n, degree):
    """A level's image and gradients do not depend on the levels beside it (an
    empty one among them; thresholds of 0 leave only the last active) nor on
    the alignment of the SH gradients."""
    torch, api, ctx = env
    p, other = _params(torch, n, n, -2.5), _params(torch, 40, 7, -2.5)
    empty = [t[:0] for t in other]
    cam = _cam(72, 56)
    fv = [0.0, 1e-3, 2e-3]
    a, _, ha = ctx.render_params(*p, cam, sh_degree=degree, filter_var=fv[2], save=True)
    b, _, hb = ctx.render_params_lod([other, empty, p], cam, [0.0, 0.0], fv, sh_degree=degree, train_level=2, save=True)
    assert torch.equal(a, b)
    w = torch.randn(a.shape, generator=torch.Generator(device="cuda").manual_seed(n), device="cuda")
    shifted = torch.zeros(48 * n + 1, device="cuda")[1:].view(n, 48)
    ga = [torch.zeros_like(t) for t in p]
    gb = [torch.zeros_like(t) for t in p[:4]] + [shifted]
    assert shifted.data_ptr() % 16 != 0
    ctx.render_backward(ha, w, *ga)
    ctx.render_backward(hb, w, *gb)
    ctx.release(ha)
    ctx.release(hb)
    for x, y in zip(ga, gb):   # the same FP64 sums of warp partials, in any order, rounded once
        assert float((x - y).abs().max()) <= 1e-6 * float(x.abs().max() + 1e-30)
    assert float(ga[4][:, 3 * (degree + 1) ** 2:].abs().sum()) == 0.0


@pytest.mark.parametrize("n,hidden,degree", [(1, 0, 3), (33, 0, 2), (1023, 500, 1), (1024, 1024, 3), (1025, 1, 0),
                                             (5000, 4000, 3)])
def test_written_gradients_equal_accumulated(env, n, hidden, degree):
    """lodge_render_gradients sets every row: the accumulated gradients where
    a Gaussian is seen, 0 elsewhere (`hidden` ones behind the camera, in one
    run of the list and scattered), at both alignments."""
    torch, api, ctx = env
    p = _params(torch, n, n, -3.0)
    half = hidden // 2
    p[0][:half, 2] = -50.0
    p[0][torch.randperm(n, generator=torch.Generator().manual_seed(n))[:hidden - half].cuda(), 2] = -50.0
    cam = _cam(90, 70)
    img, st, h = ctx.render_params(*p, cam, sh_degree=degree, save=True)
    w = torch.randn(img.shape, generator=torch.Generator(device="cuda").manual_seed(n), device="cuda")
    want = [torch.zeros_like(t) for t in p]
    ctx.render_backward(h, w, *want)
    for shift in (0, 1):
        got = [torch.full((t.numel() + shift,), float("nan"), device="cuda")[shift:].view(t.shape) for t in p]
        ctx.render_gradients(h, w, *got)
        for x, y in zip(got, want):   # the same FP64 sums of warp partials, in any order, rounded once
            assert float((x - y).abs().max()) <= 1e-6 * float(y.abs().max() + 1e-30)
    ctx.release(h)
