"""When and how often a frame's plan is made: for the mode that runs, once the
scene has changed, in device memory that is reused."""
import numpy as np
import pytest

from oracle.scene import OracleScene
from paper_2511_02852_gb300 import workloads as wl
from test_gpu_parity import compare_maps

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    yield
    torch.cuda.synchronize()


def _cfg(n=4, nb=12):
    rng = np.random.default_rng(n)
    spec = wl.spectrum(wind_speed=9.0, fetch=40e3, n_buckets=nb, n_theta=8, fft_n=64, fft_L=120.0, seed=11)
    ps = [wl.patch(origin_x=5.0 * i, cell=0.5, width=int(rng.integers(60, 300)), height=int(rng.integers(60, 300)),
                   max_particles=8000, prefill=2000) for i in range(n)]
    return wl.scene("plan", spec, ps, frames=2)


class _Counted:
    """A scene whose allocator calls are counted."""

    def __init__(self, cfg):
        from paper_2511_02852_gb300 import scwp
        self.calls = self.held = 0
        self.sizes = {}
        orig_alloc = torch.cuda.caching_allocator_alloc
        orig_free = torch.cuda.caching_allocator_delete

        def alloc(nbytes, device, stream):
            p = orig_alloc(nbytes, device, stream)
            self.calls += 1
            self.held += nbytes
            self.sizes[int(p)] = nbytes
            return p

        def free(p):
            self.held -= self.sizes.pop(int(p), 0)
            orig_free(p)

        torch.cuda.caching_allocator_alloc, torch.cuda.caching_allocator_delete = alloc, free
        self._undo = (orig_alloc, orig_free)
        self.sc = scwp.Scene(cfg, device=0)

    def close(self):
        self.sc.close()
        torch.cuda.caching_allocator_alloc, torch.cuda.caching_allocator_delete = self._undo


def test_a_plain_scene_makes_no_tensor_core_plan():
    """Descriptors, parameters and the summed-area frame plan: four blocks at
    most; the tensor-core frame plan is made once the scene is batched."""
    cfg = _cfg()
    c = _Counted(cfg)
    try:
        before = c.calls
        c.sc.step(cfg["dt"])
        torch.cuda.synchronize()
        assert c.calls - before <= 4
    finally:
        c.close()


@pytest.mark.parametrize("first_batched", [False, True])
def test_modes_in_turn(first_batched):
    """Either synthesis, in either mode, whichever came first."""
    from paper_2511_02852_gb300 import scwp
    cfg = _cfg()
    sc, orc = scwp.Scene(cfg, device=0), OracleScene(cfg)
    sc.step(cfg["dt"])
    orc.step(cfg["dt"])
    bg = orc.background()
    ref = [orc.patch_maps(p, bg)[0] for p in range(len(cfg["patches"]))]
    for batched in (first_batched, not first_batched):
        sc.set_batched(batched)
        for mode in (scwp.SYNTH_GATHER, scwp.SYNTH_SAT, scwp.SYNTH_GATHER):
            sc.resynthesize(mode)
            for p, r in enumerate(ref):
                compare_maps(sc.maps(p), r, orc.spec.Hs(), "batched %d mode %d patch %d" % (batched, mode, p))
    sc.close()


def test_the_first_frame_takes_one_block():
    cfg = _cfg()
    c = _Counted(cfg)
    try:
        before = c.calls
        c.sc.step(cfg["dt"])
        torch.cuda.synchronize()
        assert c.calls - before <= 1
    finally:
        c.close()


@pytest.mark.parametrize("batched", [False, True])
def test_planning_again_holds_no_more_memory(batched):
    """A second round of the same settings takes no device memory that the
    first did not."""
    cfg = _cfg()
    c = _Counted(cfg)
    try:
        sc = c.sc
        sc.set_batched(batched)

        def settings():
            for lo, hi in ((0, 3), (3, 12), (0, 64)):
                sc.set_bucket_range(lo, hi)
                sc.step(cfg["dt"])
            for gmul in (0.5, 2.0, 8.0, 1.0):
                sc.set_sat_plan(0, gmul)
                sc.step(cfg["dt"])
            sc.set_batched(not batched)
            sc.step(cfg["dt"])
            sc.set_batched(batched)
            sc.step(cfg["dt"])
            torch.cuda.synchronize()

        settings()
        held = c.held
        for _ in range(3):
            settings()
            assert c.held == held
    finally:
        c.close()


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("n,side", [(1, 300), (2, 100), (32, 512)])
def test_patch_info_describes_the_plan_that_runs(n, side, batched):
    """A group-sum blend runs if and only if some patch has more than one
    plane, and every patch has one item per tile, group and part."""
    from paper_2511_02852_gb300 import scwp
    spec = wl.spectrum(wind_speed=9.0, fetch=40e3, n_buckets=12, n_theta=8, fft_n=64, fft_L=120.0, seed=11)
    cfg = wl.scene("info", spec, [wl.patch(cell=0.5, width=side, height=side, max_particles=4000, prefill=500)
                                  for _ in range(n)], frames=1)
    sc = scwp.Scene(cfg, device=0)
    sc.set_batched(batched)
    count = lambda: scwp_launches(scwp, sc)
    sc.step(cfg["dt"])
    for gmul in (1.0, 8.0, 0.125):
        sc.set_sat_plan(0, gmul)
        infos = [sc.info(p) for p in range(n)]
        before = count()
        sc.resynthesize(scwp.SYNTH_SAT)
        passes = (int(infos[0].total_bins).bit_length() + 7) // 8
        blend = any(i.sat_groups * i.sat_parts > 1 for i in infos)
        assert count() - before == 1 + passes + 1 + 1 + blend   # keys, sort, records, synthesis, blend
        for i in infos:
            assert i.sat_items == ((side + 63) // 64) ** 2 * i.sat_groups * i.sat_parts
    sc.close()


def test_three_group_plans_keep_their_waves():
    """The three-group kernel (two CTAs an SM, one item each) gets at least
    three waves of items on a patch that has the buckets for it."""
    from paper_2511_02852_gb300 import scwp
    sc = scwp.Scene(wl.realistic(), device=0)
    sc.set_sat_plan(1, 1.0)
    i = sc.info(0)
    assert i.sat_variant == 1 and i.sat_items >= 3 * i.sat_slots, (i.sat_items, i.sat_slots)
    sc.set_sat_plan(0, 1.0)
    assert sc.info(0).sat_variant == 0
    sc.close()


def scwp_launches(scwp, sc):
    import ctypes
    n = ctypes.c_int64()
    assert scwp.lib().scwp_launch_count(sc.ctx, ctypes.byref(n)) == 0
    return n.value
