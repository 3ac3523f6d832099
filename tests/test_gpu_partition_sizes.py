"""Parts small enough for the small-mesh kernels against a whole mesh that takes the large ones (marked gpu).

The whole mesh lies above every limit on the element count (304 at p = 2 and 3, 152 at p = 4) and on the
point count (38912), each part below: residual and one step of every Runge-Kutta scheme, with and without a
body acceleration and a sponge, agree bit for bit in all three precisions, as they do where parts and whole
run the same kernels."""
import numpy as np
import pytest

from paper_2308_06605_gb300 import fr
from paper_2308_06605_gb300 import inputs as I

from helpers import ensure_lib
from test_gpu_partition import Parts

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("viscous", [1, 2])
@pytest.mark.parametrize("precision", [fr.FR_PREC_FP64, fr.FR_PREC_MIXED, fr.FR_PREC_MIXED_VF32])
@pytest.mark.parametrize("p,box,n_parts", [(2, (12, 11, 11), 5), (3, (9, 9, 9), 3), (4, (9, 6, 6), 3)])
def test_small_parts_equal_a_large_whole(p, box, n_parts, precision, viscous):
    torch = pytest.importorskip("torch")
    ensure_lib()
    desc = I.hex_box_mesh(box, seed=6, shuffle=True, rotate=True, perturb=0.05)
    ph = I.tgv_physics(Ma=0.2, Re=400.0)
    ph.precision, ph.viscous = precision, viscous
    whole = fr.Mesh(desc, ph, p)
    parts = Parts(desc, ph, p, n_parts)
    try:
        limit = 152 if p == 4 else 304
        assert whole.n_elem > limit and whole.n_points > 38912
        assert all(m.n_elem <= limit and m.n_points <= 38912 for m in parts.meshes)
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
