"""fr_set_state from device memory (marked gpu): a buffer shorter than the state is refused, as the
device copy refuses it, and never read past its end; whole allocations and parts of larger ones are read.

The short buffer is followed by another allocation in the same mapped block, so that no read of this test could leave
mapped memory, whatever the library did with it."""
import ctypes as C

import numpy as np
import pytest

from paper_2308_06605_gb300 import fr
from paper_2308_06605_gb300 import inputs as I

from helpers import ensure_lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rt():
    """The CUDA runtime that the library loaded."""
    ensure_lib()
    with open("/proc/self/maps") as fh:
        path = next(ln.split()[-1] for ln in fh if "libcudart" in ln)
    return C.CDLL(path)


def _malloc(rt, n):
    p = C.c_void_p()
    assert rt.cudaMalloc(C.byref(p), C.c_size_t(n)) == 0
    return p.value


@pytest.mark.parametrize("precision", [fr.FR_PREC_FP64, fr.FR_PREC_MIXED])
def test_short_device_buffer_is_refused(rt, precision):
    ph = I.tgv_physics(Ma=0.2, Re=400.0)
    ph.precision = precision
    with fr.Mesh(I.hex_box_mesh((4, 4, 4)), ph, 2) as m:
        need = int(np.prod(m.shape)) * 8
        bufs = [_malloc(rt, 4096) for _ in range(64)]
        try:
            # The lowest of the short buffers, with at least the state's size mapped behind its start.
            bufs.sort()
            short = next((b for b in bufs if any(b + need <= c + 4096 and b >> 21 == (c + 4095) >> 21 for c in bufs)), None)
            if short is None:
                pytest.skip("no neighbouring allocations")
            st = fr.load().fr_set_state(m._h, C.c_void_p(short), fr.FR_DEVICE)
            assert st == fr.FR_ECUDA
        finally:
            for b in bufs:
                rt.cudaFree(C.c_void_p(b))
    rt.cudaGetLastError()


@pytest.mark.parametrize("precision", [fr.FR_PREC_FP64, fr.FR_PREC_MIXED])
def test_whole_and_inner_device_buffers(precision):
    torch = pytest.importorskip("torch")
    ensure_lib()
    ph = I.tgv_physics(Ma=0.2, Re=400.0)
    ph.precision = precision
    with fr.Mesh(I.hex_box_mesh((4, 4, 4)), ph, 2) as m:
        Q = np.ascontiguousarray(I.tgv_state(m.solution_points(), Ma=0.2))
        n = Q.size
        big = torch.zeros(2 * n + 3, dtype=torch.float64, device="cuda")
        for at in (0, 1, n + 3):
            big[at:at + n] = torch.from_numpy(Q.ravel()).cuda()
            m.set_state(np.zeros(m.shape) + 1.0)
            m.set_state(big[at:at + n])
            np.testing.assert_array_equal(m.get_state(), Q)
            big.zero_()


@pytest.mark.parametrize("where", ["host", "device"])
def test_short_state_is_refused_by_the_binding(where):
    torch = pytest.importorskip("torch")
    ensure_lib()
    with fr.Mesh(I.hex_box_mesh((2, 2, 2)), I.tgv_physics(), 2) as m:
        short = np.zeros(int(np.prod(m.shape)) - 1)
        with pytest.raises(ValueError):
            m.set_state(short if where == "host" else torch.from_numpy(short).cuda())


def test_set_state_under_stream_capture():
    torch = pytest.importorskip("torch")
    ensure_lib()
    st = torch.cuda.Stream()
    with fr.Mesh(I.hex_box_mesh((4, 4, 4)), I.tgv_physics(Ma=0.2, Re=400.0), 2, stream=st.cuda_stream) as m:
        Q = np.ascontiguousarray(I.tgv_state(m.solution_points(), Ma=0.2))
        src = torch.from_numpy(Q).cuda()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            m.set_state(src)
        m.set_state(np.ones(m.shape))
        graph.replay()
        torch.cuda.synchronize()
        np.testing.assert_array_equal(m.get_state(), Q)
