"""Inviscid residuals on every element kernel against the oracle (marked gpu): hexahedra (DG-equivalent correction
and c != 0), mixed and all-prism meshes; per entry 1e-12 (FP64, flux from the contravariant velocity) and 1e-9
(double-float) of the magnitude scale, and a batch's persistent kernel against the mesh's own kernels, 1e-13."""
import numpy as np
import pytest

from paper_2308_06605_gb300 import fr
from paper_2308_06605_gb300 import inputs as I
from oracle.hexfr import HexFR
from oracle.mixedfr import MixedFR

from helpers import assert_residual_parity, ensure_lib, vcjh_c

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def flat(arrs):
    return np.concatenate([np.asarray(a).reshape(-1, 5) for a in arrs])


@pytest.mark.parametrize("kind", ["hex", "vcjh", "checker", "all"])
@pytest.mark.parametrize("p", [1, 2, 3, 4, 5])
def test_inviscid_residual(p, kind):
    d = I.hex_box_mesh((3, 3, 2), prisms=None if kind in ("hex", "vcjh") else kind, seed=p, rotate=True, shuffle=True, perturb=0.1)
    ph = I.tgv_physics(Ma=0.2, Re=400.0)
    ph.viscous = 0
    if kind == "vcjh":
        ph.vcjh_c = vcjh_c(p, "hu")
    ora = (HexFR if kind in ("hex", "vcjh") else MixedFR)(d, ph, p)
    if kind in ("hex", "vcjh"):
        Q = [np.ascontiguousarray(I.tgv_state(ora.x, Ma=0.2, perturb=1e-2, seed=1))]
        R, S = ora.residual(Q[0]).reshape(-1, 5), ora.residual(Q[0], magnitude=True).reshape(-1, 5)
    else:
        Q = [np.ascontiguousarray(I.tgv_state(x, Ma=0.2, perturb=1e-2, seed=1)) for x in ora.x]
        R, S = flat(ora.residual(Q)), flat(ora.residual(Q, magnitude=True))
    for precision, bar in [(fr.FR_PREC_FP64, 1e-12), (fr.FR_PREC_MIXED, 1e-9)]:
        ph.precision = precision
        with fr.Mesh(d, ph, p) as g:
            g.set_state(flat(Q))
            assert_residual_parity(g.residual().reshape(-1, 5), R, S, bar)


@pytest.mark.parametrize("prisms", [None, "checker"])
def test_batch_and_mesh_agree(prisms):
    d = I.hex_box_mesh((3, 3, 2), prisms=prisms, seed=1, rotate=True, shuffle=True, perturb=0.1)
    ph = I.tgv_physics(Ma=0.2, Re=400.0)
    ph.viscous = 0
    with fr.Mesh(d, ph, 3) as a, fr.Mesh(d, ph, 3) as b:
        Q = np.ascontiguousarray(I.tgv_state(a.solution_points(), Ma=0.2, perturb=1e-2, seed=1))
        a.set_state(Q)
        b.set_state(Q)
        a.rk_step(0.0, 1e-3)
        with fr.Batch([b]) as bt:
            bt.select(0)
            bt.set_dt([1e-3])
            bt.rk_step()
        np.testing.assert_allclose(b.get_state(), a.get_state(), rtol=1e-13, atol=1e-13)
