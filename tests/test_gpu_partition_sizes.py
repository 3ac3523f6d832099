"""Parts small enough for the small-mesh kernels against a whole mesh that takes the large ones (marked gpu).

The whole mesh lies above every limit on the element count (small viscous meshes: 1216 at p = 1, 304 at p = 2 and
3, 152 at p = 4; two elements per thread: 1824 at p = 2, 1216 at p = 3, 608 at p = 4) and on the point count
(38912), each part below: residual and one step of every Runge-Kutta scheme, with and without a
body acceleration and a sponge, agree bit for bit in all three precisions, as they do where parts and whole
run the same kernels."""
import numpy as np
import pytest

from paper_2308_06605_gb300 import fr
from paper_2308_06605_gb300 import inputs as I

from helpers import ensure_lib
from test_gpu_partition import Parts

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("viscous", [0, 1, 2])
@pytest.mark.parametrize("precision", [fr.FR_PREC_FP64, fr.FR_PREC_MIXED, fr.FR_PREC_MIXED_VF32])
@pytest.mark.parametrize("p,box,n_parts", [(1, (17, 17, 17), 5), (2, (13, 13, 11), 7), (3, (11, 11, 11), 5), (4, (9, 9, 9), 5)])
def test_small_parts_equal_a_large_whole(p, box, n_parts, precision, viscous):
    torch = pytest.importorskip("torch")
    ensure_lib()
    desc = I.hex_box_mesh(box, seed=6, shuffle=True, rotate=True, perturb=0.05)
    ph = I.tgv_physics(Ma=0.2, Re=400.0)
    ph.precision, ph.viscous = precision, viscous
    whole = fr.Mesh(desc, ph, p)
    parts = Parts(desc, ph, p, n_parts)
    try:
        low, high = {1: (1216, 1216), 2: (304, 1824), 3: (304, 1216), 4: (152, 608)}[p]
        assert whole.n_elem > high and whole.n_points > 38912
        assert all(m.n_elem <= low and m.n_points <= 38912 for m in parts.meshes)
        x = whole.solution_points()
        Q = np.ascontiguousarray(I.tgv_state(x, Ma=0.2, perturb=1e-2, seed=1))
        sigma, ref = 2.0 + np.sin(x[..., 0]), np.ascontiguousarray(Q * (1 + 1e-2 * np.cos(x[..., 1:2])))
        for source in (None, "body", "both"):
            for m, eg in [(whole, slice(None))] + [(m, h["elem_global"]) for m, h in zip(parts.meshes, parts.halo)]:
                m.set_source(accel=(0.3, -0.2, 0.1) if source else None,
                             sigma=sigma[eg] if source == "both" else None, Q_ref=ref[eg] if source == "both" else None)
            whole.set_state(Q)
            parts.set_state(Q)
            R = whole.residual()
            Rd = [torch.empty(m.shape, dtype=torch.float64, device="cuda") for m in parts.meshes]
            parts.stage(R=Rd)
            torch.cuda.synchronize()
            np.testing.assert_array_equal(parts.gather([r.cpu().numpy() for r in Rd], R.shape), R, err_msg=f"residual, source {source}")
            for scheme, stages in ((fr.FR_RK44, 4), (fr.FR_SSPRK33, 3), (fr.FR_SSPRK104, 10)):
                whole.set_state(Q)
                parts.set_state(Q)
                whole.rk_step(0.0, 1e-3, scheme)
                for s in range(stages):
                    parts.stage(scheme, s, 1e-3)
                got = parts.gather([m.get_state() for m in parts.meshes], Q.shape)
                np.testing.assert_array_equal(got, whole.get_state(), err_msg=f"scheme {scheme}, source {source}")
    finally:
        parts.close()
        whole.close()


@pytest.mark.parametrize("viscous", [1, 2])
@pytest.mark.parametrize("p", [5, 7])
def test_one_and_two_elements_per_thread_agree(p, viscous):
    """FP32 viscous branch: 175 elements take the kernel with two elements per thread (its last block one), the parts
    of 88 and 87 the one with an element per block."""
    torch = pytest.importorskip("torch")
    ensure_lib()
    desc = I.hex_box_mesh((7, 5, 5), seed=6, shuffle=True, rotate=True, perturb=0.05)
    ph = I.tgv_physics(Ma=0.2, Re=400.0)
    ph.precision, ph.viscous = fr.FR_PREC_MIXED_VF32, viscous
    parts = Parts(desc, ph, p, 2)
    try:
        with fr.Mesh(desc, ph, p) as whole:
            Q = np.ascontiguousarray(I.tgv_state(whole.solution_points(), Ma=0.2, perturb=1e-2, seed=1))
            whole.set_state(Q)
            R = whole.residual()
        assert sorted(m.n_elem for m in parts.meshes) == [87, 88]
        parts.set_state(Q)
        Rd = [torch.empty(m.shape, dtype=torch.float64, device="cuda") for m in parts.meshes]
        parts.stage(R=Rd)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(parts.gather([r.cpu().numpy() for r in Rd], R.shape), R)
    finally:
        parts.close()
