"""Which way a map goes to a device buffer: the copy kernel only where the
whole buffer lies in one allocation; a range that runs out of its allocation,
even into the next one, is the copy API's to take or refuse.  The calls are
captured and the graphs never launched: nothing is written."""
import ctypes as C

import pytest

from paper_2511_02852_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KERNEL_NODE = 0
SIZE = 2 << 20


@pytest.fixture(scope="module")
def rt():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.init()
    R = C.CDLL("libcudart.so.13")
    for name in ("cudaMalloc", "cudaFree", "cudaStreamBeginCapture", "cudaStreamEndCapture", "cudaGraphGetNodes",
                 "cudaGraphNodeGetType", "cudaGraphDestroy", "cudaGetLastError"):
        getattr(R, name).restype = C.c_int
    yield R
    torch.cuda.synchronize()


def _captured(R, stream, call):
    """Status of call() under capture on the stream, and the node types."""
    st = C.c_void_p(stream.cuda_stream)
    assert R.cudaStreamBeginCapture(st, C.c_int(2)) == 0
    rc = call()
    graph, kinds = C.c_void_p(), []
    if R.cudaStreamEndCapture(st, C.byref(graph)) == 0 and graph.value:
        n = C.c_size_t(16)
        nodes = (C.c_void_p * 16)()
        assert R.cudaGraphGetNodes(graph, nodes, C.byref(n)) == 0
        for k in range(n.value):
            t = C.c_int()
            assert R.cudaGraphNodeGetType(C.c_void_p(nodes[k]), C.byref(t)) == 0
            kinds.append(t.value)
        R.cudaGraphDestroy(graph)
    R.cudaGetLastError()
    return rc, kinds


def test_a_range_past_its_allocation_is_not_written_by_a_kernel(rt):
    from paper_2511_02852_gb300 import scwp
    R = rt
    bufs = []
    for _ in range(16):
        p = C.c_void_p()
        assert R.cudaMalloc(C.byref(p), C.c_size_t(SIZE)) == 0
        bufs.append(p.value)
    try:
        s = torch.cuda.Stream()
        spec = wl.spectrum(wind_speed=9.0, fetch=40e3, n_buckets=4, n_theta=8, fft_n=32, fft_L=60.0, seed=2)
        cfg = wl.scene("route", spec, [wl.patch(cell=0.5, width=512, height=512, max_particles=2000, prefill=300)],
                       frames=1)
        sc = scwp.Scene(cfg, device=0, stream=s)
        sc.step(cfg["dt"])
        s.synchronize()
        n = 512 * 512
        at = lambda p: (lambda: scwp.lib().scwp_height_map(sc.ctx, 0, 0, C.c_void_p(p), n, 1))
        # from the first byte, and up to the last one, of an allocation
        for p in (bufs[0], bufs[0] + SIZE - 4 * n):
            assert _captured(R, s, at(p)) == (0, [KERNEL_NODE])
        addr = sorted(bufs)
        pair = [a for a, b in zip(addr, addr[1:]) if b - (a + SIZE) < 2 * n]
        if not pair:
            pytest.skip("no two allocations next to each other")
        # starts in one allocation, ends in the next
        rc, kinds = _captured(R, s, at(pair[0] + SIZE - 2 * n))
        assert KERNEL_NODE not in kinds, (rc, kinds)
        sc.close()
    finally:
        torch.cuda.synchronize()
        for p in bufs:
            R.cudaFree(C.c_void_p(p))
