"""A background copied from a server's scene to the device, then the scene's
next frame: the copy runs on the server stream, behind whatever is queued
there, and has to get the frame it was asked for."""
import ctypes

import numpy as np
import pytest

from paper_2511_02852_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    yield
    torch.cuda.synchronize()


@pytest.mark.parametrize("whole", [True, False])
def test_background_copied_before_the_next_frame(whole):
    from paper_2511_02852_gb300 import scwp
    cfg, other = wl.small_jonswap(), wl.tiny()
    alone = scwp.Scene(cfg)
    alone.set_batched(True)
    want = []
    for _ in range(3):
        alone.step(cfg["dt"])
        want.append(np.stack(alone.maps(-1)))
    alone.close()
    assert not np.array_equal(want[0], want[1])
    sv = scwp.Server(max_inflight=3)
    a, b = sv.add_scene(cfg), sv.add_scene(other)
    view = sv.scene(a)
    n = want[0][0].size
    rid, done, got = 0, 0, []

    def copy(dst):
        if whole:
            scwp.scwp_height_maps(view.ctx, -1, ctypes.c_void_p(dst.data_ptr()), 3 * n, 1)
        else:
            for f in range(3):
                scwp.scwp_height_map(view.ctx, -1, f, ctypes.c_void_p(dst[f].data_ptr()), n, 1)

    for _ in range(3):
        sv.submit(a, cfg["dt"], rid)
        sv.submit(b, other["dt"], rid + 1)
        rid += 2
        assert sv.tick() >= 1
        while done < rid:   # (the host's own wait for the frame)
            done += len(sv.poll())
            if done < rid:
                sv.tick()
        # the server stream has work ahead of the copy; the next tick comes meanwhile
        dst = torch.empty((3, n), device="cuda")
        torch.cuda._sleep(20_000_000)   # about 10 ms
        copy(dst)
        got.append(dst)
    torch.cuda.synchronize()
    for f, (g, w) in enumerate(zip(got, want)):
        assert np.array_equal(g.cpu().numpy().reshape(w.shape), w), "frame %d" % (f + 1)
    sv.close()
