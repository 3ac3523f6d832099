"""Kernels of large meshes against the oracle (marked gpu), on meshes just large enough to take them.

Up to 304 elements at p = 2 and 3 and 152 at p = 4 a viscous mesh takes the volume kernel that spreads an
element's variables over thread groups, up to 1216 at p = 1 the one with an element per warp, and up to 38912
points the correction kernel with one thread per point; the suite's other meshes with LDG, boundaries,
non-affine elements or the closure are that small.  Here: the full volume kernels at odd element counts on shuffled,
rotated and perturbed elements with BR2 and LDG, periodic and between a wall and a characteristic boundary, a
residual and a step each; the staged correction without source terms under the three Runge-Kutta schemes; the
closure with one element per block, with the split kernel and with sixteen per block (three in the last).  Bars of the
suite: per entry 1e-12 (FP64), 1e-9 (double-float), 2e-8 (FP32 viscous branch, Re >= 400 at these cell sizes)
of the magnitude scale; closure: nu 1e-5 relative, residual 1e-6."""
import numpy as np
import pytest

from paper_2308_06605_gb300 import fr
from paper_2308_06605_gb300 import inputs as I
from oracle import timeint as TI
from oracle.hexfr import HexFR

from helpers import assert_residual_parity, assert_state_parity, ensure_lib
from test_gpu_closure import _random_net, bf16_round

pytestmark = pytest.mark.gpu

BARS = [(fr.FR_PREC_FP64, 1e-12), (fr.FR_PREC_MIXED, 1e-9), (fr.FR_PREC_MIXED_VF32, 2e-8)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def _case(kind, box):
    """Mesh (cells as large as those of the suite's 4^3 and 4 x 2 x 2 boxes), physics and state."""
    if kind == "periodic":
        d = I.hex_box_mesh(box, hi=tuple(2 * np.pi * round(b / 4) for b in box), seed=5, shuffle=True, rotate=True, perturb=0.1)
        return d, I.tgv_physics(Ma=0.2, Re=400.0), lambda x: I.tgv_state(x, Ma=0.2, perturb=1e-2, seed=1)
    d = I.hex_box_mesh(box, hi=tuple(float(round(b / 2)) for b in box), periodic=(False, True, True), seed=3, rotate=True,
                       shuffle=True, perturb=0.1,
                       wall_tags={1: (I.BC_WALL_ISOTHERMAL, (1.1,)), 2: (I.BC_CHAR_OUTFLOW, (0.7,))})
    ph = I.Physics(gamma=1.4, R=1.0, mu=5e-4, Pr=0.71, viscous=1)
    return d, ph, lambda x: I.conserved(1 + 0.1 * np.sin(x[..., 0]), 0.2 * np.cos(2 * np.pi * x[..., 1]), 0.1 + 0 * x[..., 0],
                                        0.05 * np.sin(2 * np.pi * x[..., 2]), 0.7 + 0.02 * x[..., 0], 1.4)


@pytest.mark.parametrize("viscous", [1, 2])
@pytest.mark.parametrize("kind", ["periodic", "walls"])
@pytest.mark.parametrize("p,box", [(1, (11, 11, 11)), (2, (9, 7, 7)), (3, (9, 7, 7)), (4, (9, 5, 5))])
def test_volume_kernels_above_the_small_mesh_limit(p, box, kind, viscous):
    d, ph, state = _case(kind, box)
    ph.viscous = viscous
    ora = HexFR(d, ph, p)
    Q = np.ascontiguousarray(state(ora.x))
    R, S = ora.residual(Q), ora.residual(Q, magnitude=True)
    dt = 0.3 * ora.max_dt(Q, 0.3)
    Q1 = ora.rk44_step(Q, 0.0, dt)
    for precision, bar in BARS:
        ph.precision = precision
        with fr.Mesh(d, ph, p) as g:
            g.set_state(Q)
            assert_residual_parity(g.residual(), R, S, bar)
            g.rk_step(0.0, dt)
            assert_state_parity(g.get_state(), Q1, S, dt, bar)


# Odd element counts at which the kernel with two elements per thread runs (FP32 viscous branch, or no viscous branch in
# double-float), its last block with one.
@pytest.mark.parametrize("p,box,viscous", [(3, (11, 11, 11), 1), (3, (11, 11, 11), 2), (4, (9, 9, 9), 1), (4, (9, 9, 9), 2),
                                           (5, (7, 5, 5), 1), (5, (7, 5, 5), 2), (5, (9, 9, 7), 2), (2, (13, 13, 11), 0), (3, (11, 11, 11), 0), (4, (9, 9, 7), 0)])
def test_two_elements_per_thread(p, box, viscous):
    d, ph, state = _case("walls" if viscous == 2 else "periodic", box)
    ph.viscous = viscous
    ora = HexFR(d, ph, p)
    Q = np.ascontiguousarray(state(ora.x))
    ph.precision = fr.FR_PREC_MIXED_VF32 if viscous else fr.FR_PREC_MIXED
    with fr.Mesh(d, ph, p) as g:
        g.set_state(Q)
        assert_residual_parity(g.residual(), ora.residual(Q), ora.residual(Q, magnitude=True), 2e-8 if viscous else 1e-9)


@pytest.mark.parametrize("p,box", [(3, (9, 9, 9)), (4, (7, 7, 7))])
def test_staged_correction_without_source(p, box):
    d, ph, state = _case("periodic", box)
    ora = HexFR(d, ph, p)
    Q = np.ascontiguousarray(state(ora.x))
    S, dt = ora.residual(Q, magnitude=True), 0.3 * ora.max_dt(Q, 0.3)
    for name, scheme in (("rk44", fr.FR_RK44), ("ssprk33", fr.FR_SSPRK33), ("ssprk104", fr.FR_SSPRK104)):
        want = TI.SCHEMES[name](lambda q: [ora.residual(q[0])], [Q], dt)[0]
        for precision, bar in BARS[:2]:
            ph.precision = precision
            with fr.Mesh(d, ph, p) as g:
                g.set_state(Q)
                g.rk_step(0.0, dt, scheme)
                assert_state_parity(g.get_state(), want, S, dt * TI.STAGES[name] / 4, bar)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("p,box", [(1, (17, 1, 1)), (1, (4, 4, 4)), (1, (11, 11, 11)), (2, (9, 7, 7)), (3, (9, 7, 7)), (4, (3, 3, 3)),
                                   (4, (9, 5, 5)), (5, (3, 3, 2))])
def test_closure(p, box, precision):
    d = I.hex_box_mesh(box, seed=5, rotate=True, shuffle=True, perturb=0.05)
    ph = I.tgv_physics(Ma=0.2, Re=300.0)
    ph.precision = precision
    ora = HexFR(d, ph, p)
    Q = np.ascontiguousarray(I.tgv_state(ora.x, Ma=0.2, perturb=2e-2, seed=1))
    P = _random_net(2)
    scales = np.concatenate([np.zeros(11), [1.0] * 9, [1.5, 0.2], [0.8]]).astype(np.float32)
    with fr.Mesh(d, ph, p) as g:
        g.set_closure(P, scales)
        g.set_state(Q)
        R = g.residual()
        nu = g.closure_nu()
    ora.set_closure(bf16_round(P).astype(np.float64),
                    (scales[:11].astype(np.float64), scales[11:22].astype(np.float64), float(scales[22])))
    Ro = ora.residual(Q)
    assert np.ptp(ora.last_nu) > 1e-2 * ora.last_nu.mean()     # an element's value is not its neighbour's
    np.testing.assert_allclose(nu, ora.last_nu, rtol=1e-5)
    assert_residual_parity(R, Ro, ora.residual(Q, magnitude=True), rel=1e-6)
