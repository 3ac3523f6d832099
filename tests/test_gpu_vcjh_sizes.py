"""Steps with a correction function c != 0 below and above the 38912 points up to which the correction runs with
one thread per point (marked gpu), against the oracle: states within 1e-12 (FP64) and 1e-9 (double-float) of
|Q| + dt S, with and without a body acceleration."""
import numpy as np
import pytest

from paper_2308_06605_gb300 import fr
from paper_2308_06605_gb300 import inputs as I
from oracle import timeint as TI
from oracle.mixedfr import MixedFR

from helpers import assert_state_parity, ensure_lib, vcjh_c

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [4, 9])
def test_steps(n):
    ensure_lib()
    p = 3
    d = I.hex_box_mesh((n, n, n), hi=(2 * np.pi * round(n / 4),) * 3, seed=2, shuffle=True, rotate=True, perturb=0.1)
    ph = I.tgv_physics(Ma=0.2, Re=400.0)
    ph.vcjh_c = vcjh_c(p, "hu")
    ora = MixedFR(d, ph, p)
    Q = [np.ascontiguousarray(I.tgv_state(x, Ma=0.2, perturb=1e-2, seed=1)) for x in ora.x]
    dt = 2e-3
    for accel in (None, (0.3, -0.2, 0.1)):
        ora.set_source(accel=accel)
        S = ora.residual(Q, magnitude=True)[0]
        for scheme, name in ((fr.FR_RK44, "rk44"), (fr.FR_SSPRK33, "ssprk33")):
            want = TI.SCHEMES[name](ora.residual, Q, dt)[0]
            for precision, bar in ((fr.FR_PREC_FP64, 1e-12), (fr.FR_PREC_MIXED, 1e-9)):
                ph.precision = precision
                with fr.Mesh(d, ph, p) as g:
                    g.set_source(accel=accel)
                    g.set_state(Q[0])
                    g.rk_step(0.0, dt, scheme)
                    assert_state_parity(g.get_state(), want, S, dt, bar)
