"""Edges of a server tick's shared launches: 16 backgrounds of one grid size a
launch, packs of 32 patches over the plans of several scenes, grid sizes
interleaved.  Each scene is the same as when it is stepped alone."""
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


def _scene(i, fft_n, patches):
    rng = np.random.default_rng(i)
    spec = wl.spectrum(wind_speed=6.0 + 0.3 * i, fetch=40e3, n_buckets=4, n_theta=8, fft_n=fft_n, fft_L=90.0 + i, seed=i)
    ps = [wl.patch(origin_x=float(rng.uniform(-40, 40)), cell=0.5, width=int(rng.integers(20, 90)),
                   height=int(rng.integers(20, 90)), max_particles=3000, prefill=int(rng.integers(0, 500)),
                   emitter=k % 2, obj_radius=2.0, obj_speed=4.0, obj_path_radius=4.0, wake_amp=0.02, wake_rate=2)
          for k in range(patches)]
    return wl.scene("s%d" % i, spec, ps, frames=2)


# scenes of a 32^2 grid, of other grids, patches each
@pytest.mark.parametrize("n,others,patches", [(15, 2, 1), (16, 0, 2), (16, 3, 2), (17, 3, 2), (33, 1, 1)])
def test_scenes_of_one_tick_are_as_when_alone(n, others, patches):
    from paper_2511_02852_gb300 import scwp
    cfgs = [_scene(i, 32, patches) for i in range(n)]
    for k in range(others):
        cfgs.insert(3 * k + 1, _scene(100 + k, (64, 8, 128)[k], 1 + k))
    sv = scwp.Server(max_inflight=2)
    ids = [sv.add_scene(c) for c in cfgs]
    frames = 2
    for f in range(frames):
        for k, (s, c) in enumerate(zip(ids, cfgs)):
            sv.submit(s, c["dt"], f * len(cfgs) + k)
        assert sv.tick() == len(cfgs)   # all in one tick
        done = 0
        while done < len(cfgs):
            done += len(sv.poll())
    torch.cuda.synchronize()
    for s, c in zip(ids, cfgs):
        alone = scwp.Scene(c)
        alone.set_batched(True)
        for _ in range(frames):
            alone.step(c["dt"])
        view = sv.scene(s)
        for a, m in zip(alone.maps(-1), view.maps(-1)):
            assert np.array_equal(a, m), "background of %s" % c["name"]
        for p in range(len(c["patches"])):
            for a, m in zip(alone.particles(p), view.particles(p)):
                assert np.array_equal(a, m), "%s patch %d" % (c["name"], p)
            for a, m in zip(alone.bins(p), view.bins(p)):
                assert np.array_equal(a, m), "%s patch %d" % (c["name"], p)
            for a, m in zip(alone.maps(p), view.maps(p)):
                assert np.array_equal(a, m), "%s patch %d" % (c["name"], p)
            assert alone.stats(p).eval_count == view.stats(p).eval_count
        alone.close()
    sv.close()
