"""A step kernel whose look-back runs out.

scwp_debug_step_timeout runs the real step kernel with the word of its first
tile never published and a short limit, then the frame's binning.  The counts,
digit totals and keys of such a frame do not agree, so every later stage must
take the patch as empty: the call checks that no bump was binned and reports
the timeout.  Nothing faults, traps or hangs: a tile that gives up stores
within bounds, and a fresh scene afterwards is bit-exact against the oracle."""
import time

import pytest

from oracle.scene import OracleScene
from paper_2511_02852_gb300 import workloads as wl

from test_gpu_parity import compare_bins, compare_state

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

E_INVALID, E_TIMEOUT = 1, 5


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    yield
    torch.cuda.synchronize()


# two, three and forty tiles of 1024 particles (32 look-back words at a time)
@pytest.mark.parametrize("n,stepped", [(2000, True), (3000, False), (40000, True)])
def test_step_lookback_wait_runs_out_and_leaves_the_patch_empty(n, stepped):
    from paper_2511_02852_gb300 import scwp
    L = scwp.lib()
    spec = wl.spectrum(wind_speed=9.0, fetch=40e3, n_buckets=5, n_theta=8, fft_n=64, fft_L=120.0, seed=8)
    cfg = wl.scene("stall", spec, [wl.patch(cell=0.5, width=160, height=120, max_particles=50000, prefill=n)], frames=2)
    sc = scwp.Scene(cfg, device=0)
    if stepped:
        sc.step(cfg["dt"])
    assert sc.stats(0).live_particles > 1024
    assert L.scwp_debug_step_timeout(sc.ctx, 0, 0.0) == E_INVALID
    assert L.scwp_debug_step_timeout(sc.ctx, 1, 0.05) == E_INVALID
    wait = 0.05
    t0 = time.perf_counter()
    rc = L.scwp_debug_step_timeout(sc.ctx, 0, wait)
    took = time.perf_counter() - t0
    assert rc == E_TIMEOUT, (scwp.STATUS.get(rc, rc), L.scwp_last_error(sc.ctx))
    assert took >= 0.8 * wait
    assert L.scwp_step(sc.ctx, cfg["dt"]) == E_TIMEOUT   # sticky
    sc.close()
    fresh, orc = scwp.Scene(cfg, device=0), OracleScene(cfg)
    for _ in range(2):
        fresh.step(cfg["dt"])
        orc.step(cfg["dt"])
    assert fresh.stats(0).error_flags == 0
    compare_state(fresh, orc, 0)
    compare_bins(fresh, orc, 0)
    fresh.close()


def test_too_few_particles_for_two_tiles():
    from paper_2511_02852_gb300 import scwp
    spec = wl.spectrum(wind_speed=9.0, fetch=40e3, n_buckets=5, n_theta=8, fft_n=64, fft_L=120.0, seed=8)
    cfg = wl.scene("one", spec, [wl.patch(cell=0.5, width=64, height=64, max_particles=5000, prefill=1000)], frames=1)
    sc = scwp.Scene(cfg, device=0)
    assert scwp.lib().scwp_debug_step_timeout(sc.ctx, 0, 0.05) == E_INVALID
    sc.step(cfg["dt"])   # refused arguments leave the context usable
    assert sc.stats(0).error_flags == 0
    sc.close()
