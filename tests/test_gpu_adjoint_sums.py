"""What the compositing's adjoint works out in FP32: partial sums over at most
32 pixels before they are added in FP64, and the transmittance restored by
IEEE quotients.  Each test is built so that the exact value is known; the bars
are derived beside it."""
import numpy as np
import pytest

from paper_2505_23158_gb300 import synth

pytestmark = pytest.mark.gpu
Y0 = np.float32(0.28209479177387814)


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


def _cam(w, h):
    """A camera at the origin looking along z."""
    return synth.Camera(R=np.eye(3, dtype=np.float32), t=np.zeros(3, np.float32), fx=64.0, fy=64.0, cx=w / 2,
                        cy=h / 2, width=w, height=h, znear=0.2, center=np.zeros(3))


def _stack(torch, logits, log_scale, rgb):
    """Gaussians on the view axis, the first one nearest, all of one colour."""
    n = len(logits)
    z = torch.arange(n, device="cuda", dtype=torch.float32) + 2.0
    means = torch.stack([torch.zeros_like(z), torch.zeros_like(z), z], 1)
    quats = torch.zeros(n, 4, device="cuda")
    quats[:, 0] = 1.0
    sh = torch.zeros(n, 48, device="cuda")
    sh[:, :3] = (torch.as_tensor(rgb, dtype=torch.float32, device="cuda") - 0.5) / float(Y0)
    return [means, torch.full((n, 3), log_scale, device="cuda"), quats,
            torch.tensor(np.asarray(logits, np.float32), device="cuda"), sh]


def _render(ctx, torch, ps, cam, g_img):
    img, _, h = ctx.render_params(*ps, cam, save=True)
    gs = [torch.zeros_like(p) for p in ps]
    ctx.render_backward(h, g_img.cuda().contiguous(), *gs)
    ctx.release(h)
    return img, gs


def test_partials_span_32_pixels(env):
    """One splat that every pixel takes with the clamped weight 0.99.  In two
    8x8 blocks the rows 0, 1, 4 and 5, whose pixels one half of a warp holds,
    carry image gradients of +-2^26, and the other half's rows 1: a sum over
    a half's 32 pixels is exact in FP32 (equal terms), and the large ones
    cancel in FP64.  A partial that spans 64 pixels loses the ones (a unit in
    the last place of 2^26 is 8)."""
    torch, ctx = env
    ps = _stack(torch, [12.0], 6.0, (1.0, 1.0, 1.0))
    g = torch.zeros(16, 16, 3)
    g[[2, 3, 6, 7], :, 0] = 1.0
    for y in (0, 1, 4, 5):
        g[y, 0:8, 0] = 2.0 ** 26
        g[y, 8:16, 0] = -(2.0 ** 26)
    img, gs = _render(ctx, torch, ps, _cam(16, 16), g)
    assert (img == img[0, 0]).all() and float(img[0, 0, 0]) == float(np.float32(0.99))
    want = float(Y0) * 64 * float(np.float32(0.99))
    # FP32 roundings after the sum: its cast and the product with Y0
    assert abs(float(gs[4][0, 0]) - want) <= 2 * 2.0 ** -24 * want


# logits of two splats on the pixel's centre and their alphas on the device
@pytest.mark.parametrize("l1,l2,a1,a2", [
    ("-0x1.8331cp-1", "-0x1.d553dp+1", "0x1.472168p-2", "0x1.98615ap-6"),
    ("-0x1.5296cp+0", "-0x1.affe28p+1", "0x1.aeddcp-3", "0x1.0f0e1ap-5"),
    ("0x1.781c9p+0", "-0x1.cad6fp+1", "0x1.a038d4p-1", "0x1.ba4f1ap-6"),
    ("-0x1.ff5638p+1", "-0x1.71af4p+1", "0x1.28307p-6", "0x1.b00fd4p-5"),
    ("0x1.bb198p-2", "-0x1.8869a4p+1", "0x1.368a02p-1", "0x1.6ce666p-5")])
def test_transmittance_restored_by_ieee_quotients(env, l1, l2, a1, a2):
    """The colour gradient that one pixel gives the splat behind is Y0 T alpha
    with T = T_final / (1 - alpha), each operation rounded as IEEE has it (the
    bar is equality).  An approximate quotient with one remainder correction
    is off by a unit in the last place for these pairs."""
    torch, ctx = env
    l1, l2, a1, a2 = (np.float32(float.fromhex(x)) for x in (l1, l2, a1, a2))
    one = np.float32(1)
    ps = _stack(torch, [l1, l2], -12.0, (0.5, 0.5, 0.5))
    g = torch.zeros(17, 17, 3)
    g[8, 8, 0] = 1.0
    img, gs = _render(ctx, torch, ps, _cam(17, 17), g)
    T1 = one - a1
    T2 = T1 * (one - a2)
    want = (np.float64(a1) * 0.5 + np.float64(T1 * a2) * 0.5).astype(np.float32)   # the alphas are as given
    assert np.float32(float(img[8, 8, 0])) == want
    T = T2 / (one - a2)
    assert np.float32(float(gs[4][1, 0])) == Y0 * (T * a2)
    assert np.float32(float(gs[4][0, 0])) == Y0 * ((T / (one - a1)) * a1)
