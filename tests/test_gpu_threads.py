"""Host threads that use the library side by side (marked gpu): kernels whose shared memory differs
from call to call (a closure or none, the orders of a projection) must launch whatever another thread launches."""
import threading

import numpy as np
import pytest

from paper_2308_06605_gb300 import fr
from paper_2308_06605_gb300 import inputs as I

from helpers import ensure_lib
from test_gpu_closure import _random_net

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def _together(*jobs):
    """Run the jobs in one thread each; the first failure of each."""
    errors, gate = [], threading.Barrier(len(jobs))

    def body(job):
        try:
            gate.wait()
            job()
        except Exception as e:                      # reported by the test, not by the thread
            errors.append(e)
    ts = [threading.Thread(target=body, args=(j,)) for j in jobs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    return errors


@pytest.mark.parametrize("p,box,vcjh_c", [(1, (3, 3, 3), 0.0), (2, (3, 3, 3), 0.0), (2, (7, 7, 7), 0.0), (4, (3, 3, 3), 0.0),
                                          (2, (3, 3, 3), 1e-4)])
def test_closure_beside_a_mesh_without(p, box, vcjh_c):
    torch = pytest.importorskip("torch")
    d, ph = I.hex_box_mesh(box), I.tgv_physics(Ma=0.2, Re=300.0)
    ph.vcjh_c = vcjh_c
    scales = np.concatenate([np.zeros(11), [1.0] * 9, [1.5, 0.2], [0.8]]).astype(np.float32)
    streams = [torch.cuda.Stream() for _ in range(2)]
    with fr.Mesh(d, ph, p, stream=streams[0].cuda_stream) as a, fr.Mesh(d, ph, p, stream=streams[1].cuda_stream) as b:
        Q = np.ascontiguousarray(I.tgv_state(a.solution_points(), Ma=0.2))
        a.set_closure(_random_net(2), scales)
        for m in (a, b):
            m.set_state(Q)

        def steps(m):
            for _ in range(400):
                m.rk_step(0.0, 1e-6)
        assert _together(lambda: steps(a), lambda: steps(b)) == []


def test_projections_from_two_orders():
    torch = pytest.importorskip("torch")
    d, ph = I.hex_box_mesh((2, 2, 1), prisms="all"), I.tgv_physics(Ma=0.2, Re=300.0)
    pairs = []
    for p in (1, 1, 7):
        st = torch.cuda.Stream().cuda_stream
        a, b = fr.Mesh(d, ph, p, stream=st), fr.Mesh(d, ph, 1, stream=st)
        a.set_state(np.ascontiguousarray(I.tgv_state(a.solution_points(), Ma=0.2)))
        pairs.append((a, b))

    done = threading.Event()

    def project(a, b):
        if a.p == 7:                       # its host part takes long: the others run beside it
            try:
                for _ in range(100):
                    fr.project_state(a, b)
            finally:
                done.set()
        while not done.is_set():
            fr.project_state(a, b)
    try:
        assert _together(*[lambda q=q: project(*q) for q in pairs]) == []
    finally:
        for q in pairs:
            for m in q:
                m.close()
