"""A frame's status word reaches the call that renders the frame, whichever
of a call's frames it is and however the slot's next frame runs: a slot's
first frame is waited for in its middle only, and the frames behind it leave
their counts on the device.  The status is injected on the host's side (the
word is set after the frame's last kernel); nothing waits or faults."""
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
    scene, cams = synth.workload_outdoor(seed=5, n_poses=24, scale=0.01, width=160, height_px=96)
    return torch, api, scene, cams


@pytest.mark.parametrize("warm", [False, True])
@pytest.mark.parametrize("call", ["importance", "importance_chunk", "render", "render_full", "render_host"])
def test_status_of_any_frame_is_reported(env, call, warm):
    torch, api, scene, cams = env
    host = np.zeros(24 * 160 * 96 * 3, np.float32)

    def run(ctx, sid):
        if call == "importance":
            return ctx.importance(sid, api.CHUNK_BLEND, cams)
        if call == "importance_chunk":
            return ctx.importance(sid, api.CHUNK, cams, chunk=0)
        if call == "render":
            return torch.stack(ctx.render(sid, api.CHUNK_BLEND, cams)[0])
        if call == "render_full":
            return torch.stack(ctx.render(sid, api.FULL, cams)[0])
        ctx.render_host(sid, api.CHUNK_BLEND, cams, host)
        return torch.from_numpy(host.copy())

    with api.Lodge(0) as ctx:
        sid = ctx.load_scene(scene)
        want = run(ctx, sid)
    with api.Lodge(0) as ctx:
        sid = ctx.load_scene(scene)
        if warm:
            run(ctx, sid)
        ctx.inject_frame_timeouts(1)
        with pytest.raises(api.LodgeError) as e:
            run(ctx, sid)
        assert e.value.status == 5                      # LODGE_E_TIMEOUT
        assert torch.equal(run(ctx, sid), want)         # and the next call is sound
