"""Edges of the launches that take several patches at once, of the step
kernel's tiles, of the partial planes' pitch and of the map copies, on the
summed-area path: integer state and bins bit-exact against the oracle, maps
within the contract of test_gpu_parity.py, copies bit for bit."""
import numpy as np
import pytest

from oracle.scene import OracleScene
from paper_2511_02852_gb300 import workloads as wl
from test_gpu_parity import compare_bins, compare_maps, compare_state

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    yield
    torch.cuda.synchronize()


def _scene(cfg, batched=False):
    from paper_2511_02852_gb300 import scwp
    sc = scwp.Scene(cfg, device=0)
    sc.set_batched(batched)
    return sc


def _patches(n, **kw):
    """n uneven patches of 20 to 77 cells a side, every third with a wake."""
    rng = np.random.default_rng(5 + n)
    out = []
    for i in range(n):
        w, h = (int(v) for v in rng.integers(20, 78, 2))
        p = dict(origin_x=float(rng.uniform(-50, 50)), origin_y=float(rng.uniform(-50, 50)), cell=0.5, width=w,
                 height=h, max_particles=6000, prefill=int(rng.integers(0, 900)), emitter=1 if i % 3 == 0 else 0,
                 obj_radius=2.0, obj_speed=4.0, obj_path_radius=4.0, wake_amp=0.02, wake_rate=2)
        p.update(kw)
        out.append(wl.patch(**p))
    return out


# packs hold 1, 8 or 32 patches
@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("n", [1, 2, 8, 9, 32, 33])
def test_patches_per_launch(n, batched):
    spec = wl.spectrum(wind_speed=9.0, fetch=40e3, n_buckets=5, n_theta=8, fft_n=64, fft_L=120.0, seed=40 + n)
    cfg = wl.scene("pack%d" % n, spec, _patches(n), frames=3)
    sc, orc = _scene(cfg, batched), OracleScene(cfg)
    for _ in range(3):
        sc.step(cfg["dt"])
        orc.step(cfg["dt"])
    bg = orc.background()
    for p in range(n):
        compare_state(sc, orc, p)
        compare_bins(sc, orc, p)
        st = sc.stats(p)
        assert st.live_particles == len(orc.patches[p].X) and st.error_flags == 0
        if p in (0, n // 2, n - 1):
            ref, ev = orc.patch_maps(p, bg)
            assert st.eval_count == ev
            compare_maps(sc.maps(p), ref, orc.spec.Hs(), "pack of %d, patch %d" % (n, p))
    sc.close()


def test_injection_plans_beyond_one_launch():
    """Eight patches whose plans, 128 segments each, do not fit one launch's
    parameters."""
    spec = wl.spectrum(wind_speed=9.0, fetch=40e3, n_buckets=64, n_theta=4, fft_n=64, fft_L=120.0, seed=3)
    cfg = wl.scene("plans", spec, _patches(8, prefill=50, max_particles=60000, inject_scale=500.0, width=60, height=60),
                   frames=2)
    sc, orc = _scene(cfg), OracleScene(cfg)
    for _ in range(2):
        sc.step(cfg["dt"])
        orc.step(cfg["dt"])
    for p in range(8):
        compare_state(sc, orc, p)
        compare_bins(sc, orc, p)
    sc.close()


# tiles of 1024 particles, 32 look-back words read at a time
@pytest.mark.parametrize("n", [0, 1, 1023, 1024, 1025, 32 * 1024, 33 * 1024 + 7])
def test_step_compacts_across_tiles(n):
    spec = wl.spectrum(wind_speed=9.0, fetch=40e3, n_buckets=5, n_theta=8, fft_n=64, fft_L=120.0, seed=8)
    cfg = wl.scene("tiles", spec, [wl.patch(cell=0.5, width=70, height=45, max_particles=40000, prefill=0)], frames=2)
    sc, orc = _scene(cfg), OracleScene(cfg)
    rng = np.random.default_rng(n)
    ps = orc.patches[0]
    # from well inside to far outside: whole runs die, others live
    far = np.repeat(rng.uniform(0.2, 30.0, n // 64 + 1), 64)[:n]
    X = np.rint(rng.normal(35, 30, n) * far * 65536 * 0.5).astype(np.int64)
    Y = np.rint(rng.normal(22, 20, n) * far * 65536 * 0.5).astype(np.int64)
    B, J = rng.integers(0, 5, n), rng.integers(0, 8, n)
    ps.X, ps.Y, ps.B, ps.J = X, Y, B.astype(np.int64), J.astype(np.int64)
    sc.set_particles(0, X.astype(np.int32), Y.astype(np.int32), ((B << 16) | J).astype(np.uint32))
    for _ in range(2):
        sc.step(cfg["dt"])
        orc.step(cfg["dt"])
        compare_state(sc, orc, 0)
    compare_bins(sc, orc, 0)
    ref, ev = orc.patch_maps(0)
    assert sc.stats(0).eval_count == ev
    compare_maps(sc.maps(0), ref, orc.spec.Hs(), "%d particles" % n)
    sc.close()


# the partial planes' rows are whole quads, the maps' rows are not
@pytest.mark.parametrize("width", [1, 3, 61, 62, 63, 64, 65, 130])
def test_group_blend_of_any_width(width):
    spec = wl.spectrum(wind_speed=9.0, fetch=40e3, n_buckets=6, n_theta=8, fft_n=64, fft_L=120.0, seed=width)
    cfg = wl.scene("width", spec, [wl.patch(cell=0.5, width=width, height=37, max_particles=4000, prefill=800)], frames=1)
    sc, orc = _scene(cfg), OracleScene(cfg)
    sc.step(cfg["dt"])
    orc.step(cfg["dt"])
    assert sc.info(0).sat_groups > 1
    ref, _ = orc.patch_maps(0)
    compare_maps(sc.maps(0), ref, orc.spec.Hs(), "width %d" % width)
    sc.close()


@pytest.mark.parametrize("width,height", [(1, 1), (5, 3), (64, 64), (333, 41)])
@pytest.mark.parametrize("offset", [0, 1, 2])
def test_maps_to_a_device_buffer(width, height, offset):
    """The same words as the copy to the host, nothing beside them written,
    from any float of a device buffer."""
    import ctypes
    from paper_2511_02852_gb300 import scwp
    spec = wl.spectrum(wind_speed=9.0, fetch=40e3, n_buckets=4, n_theta=8, fft_n=32, fft_L=60.0, seed=2)
    cfg = wl.scene("copy", spec, [wl.patch(cell=0.5, width=width, height=height, max_particles=2000, prefill=300)], frames=1)
    sc = _scene(cfg)
    sc.step(cfg["dt"])
    for pid, n in ((0, width * height), (-1, 32 * 32)):
        want = np.concatenate([np.asarray(m).ravel() for m in sc.maps(pid)])
        buf = torch.full((3 * n + 8,), -7.0, device="cuda")
        scwp.scwp_height_maps(sc.ctx, pid, ctypes.c_void_p(buf.data_ptr() + 4 * offset), 3 * n, 1)
        got = buf.cpu().numpy()
        assert np.array_equal(got[offset:offset + 3 * n], want)
        assert (got[:offset] == -7.0).all() and (got[offset + 3 * n:] == -7.0).all()
        buf.fill_(-7.0)
        scwp.scwp_height_map(sc.ctx, pid, 1, ctypes.c_void_p(buf.data_ptr() + 4 * offset), n, 1)
        assert np.array_equal(buf.cpu().numpy()[offset:offset + n], want[n:2 * n])
    sc.close()


@pytest.mark.parametrize("N", [8, 64, 512])
def test_noalloc_output_on_any_float(N):
    """An output that starts on an odd float gets the same words as an
    aligned one."""
    from paper_2511_02852_gb300 import scwp
    g = torch.Generator().manual_seed(N)
    h0 = torch.randn((N, N, 2), generator=g).cuda()
    om = torch.stack([torch.rand((N, N), generator=g) * 3.0, torch.zeros(N, N)], -1).contiguous().cuda()
    fn, st = scwp.lib().scwp_background_noalloc, torch.cuda.current_stream().cuda_stream
    a, b = torch.empty(3 * N * N, device="cuda"), torch.empty(3 * N * N + 1, device="cuda")
    assert fn(h0.data_ptr(), om.data_ptr(), N, 2.0 * N, 1.0, 3.25, a.data_ptr(), st) == 0
    assert fn(h0.data_ptr(), om.data_ptr(), N, 2.0 * N, 1.0, 3.25, b.data_ptr() + 4, st) == 0
    torch.cuda.synchronize()
    assert torch.equal(a, b[1:])
