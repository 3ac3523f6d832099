"""Kernels that share a block between several elements, samples or values, at the counts where a block is
partly filled (marked gpu), against the oracle.

Volume kernel at p = 1, 2 (16 and 7 elements per block), double-float face interpolation (its own
count per order) and the correction kernels (256 points per block): residual and one RK44 step with one
element fewer and more than a full block, viscous and inviscid, at the suite's bars per entry (FP64 1e-12,
double-float 1e-9, FP32 viscous branch 2e-8 of the magnitude scale at Re 400).  Odd element counts leave the
packed volume kernel's last block with one element.  Closure training (32 samples per block, at most 304 blocks,
partial rows limited by the workspace): loss and gradient at the suite's FP32 bars.  Order projection
with the most elements per block, 1e-13.  Meshes just below and above the sizes where the kernels for few
elements or points give way to the full ones."""
import numpy as np
import pytest

from paper_2308_06605_gb300 import fr
from paper_2308_06605_gb300 import inputs as I
from oracle import mlp
from oracle import project as PJ
from oracle import timeint as TI
from oracle.hexfr import HexFR
from oracle.mixedfr import MixedFR

from helpers import assert_residual_parity, assert_state_parity, ensure_lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


@pytest.mark.parametrize("viscous", [0, 1, 2])
@pytest.mark.parametrize("precision,bar", [(fr.FR_PREC_FP64, 1e-12), (fr.FR_PREC_MIXED, 1e-9), (fr.FR_PREC_MIXED_VF32, 2e-8)])
@pytest.mark.parametrize("p,box", [(1, (5, 3, 1)), (1, (4, 2, 2)), (1, (17, 1, 1)), (2, (3, 2, 1)), (2, (7, 1, 1)),
                                   (2, (2, 2, 2)), (3, (3, 1, 1)), (3, (5, 1, 1)), (4, (3, 2, 1)), (4, (5, 1, 1)),
                                   (5, (3, 1, 1)), (6, (3, 1, 1)), (7, (3, 1, 1))])
def test_partly_filled_blocks(p, box, precision, bar, viscous):
    d = I.hex_box_mesh(box, seed=4, shuffle=True, rotate=True, affine=((1.0, 0.2, 0.0), (0.0, 1.0, 0.1), (0.1, 0.0, 1.0)))
    ph = I.tgv_physics(Ma=0.2, Re=400.0)
    ph.viscous = viscous
    ora = HexFR(d, ph, p)
    rng = np.random.default_rng(p + 10 * viscous)
    Q = np.ascontiguousarray(I.tgv_state(ora.x, Ma=0.2, perturb=1e-2, seed=1)) * (1 + 1e-3 * rng.standard_normal(ora.x.shape[:2] + (1,)))
    S = ora.residual(Q, magnitude=True)
    gph = I.Physics(**{**ph.__dict__, "precision": precision})
    with fr.Mesh(d, gph, p) as g:
        g.set_state(Q)
        assert_residual_parity(g.residual(), ora.residual(Q), S, bar)
        dt = 0.1 * ora.max_dt(Q, 0.3)
        g.rk_step(0.0, dt)
        assert_state_parity(g.get_state(), ora.rk44_step(Q, 0.0, dt), S, dt, bar)


@pytest.mark.parametrize("n", [1, 23, 24, 31, 32, 33, 64, 9728, 9761])
def test_training_tiles(n):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(n)
    X = (rng.standard_normal((n, 11)) * np.linspace(0.5, 3, 11)).astype(np.float32)
    y = np.abs(rng.standard_normal(n)).astype(np.float32)
    scales = np.concatenate([np.full(11, 0.1), np.linspace(0.5, 3, 11), [1.0]]).astype(np.float32)
    P = (0.25 * rng.standard_normal(mlp.N_PARAMS)).astype(np.float32)
    tr = fr.MLPTrainer(P, scales, max_batch=n)
    tr.g.fill_(7.0)                                     # every entry has to be written
    tr.loss.fill_(7.0)
    loss, g = tr.loss_grad(torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda())
    out = tr.forward(torch.from_numpy(X).cuda()).cpu().numpy()
    Xn = (X.astype(np.float64) - scales[:11].astype(np.float64)) / scales[11:22].astype(np.float64)
    lo, go = mlp.loss_and_grad(P.astype(np.float64), Xn, y.astype(np.float64))
    gg = g.cpu().numpy().astype(np.float64)
    assert abs(float(loss.item()) - lo) <= 1e-5 * lo
    assert np.abs(gg - go).max() <= 1e-4 * np.abs(go).max()
    np.testing.assert_allclose(out, mlp.forward(P.astype(np.float64), Xn)[0], rtol=1e-5, atol=1e-6)


@pytest.mark.parametrize("p,q", [(1, 7), (7, 1), (2, 1), (1, 2)])
def test_projection_blocks(p, q):
    d = I.hex_box_mesh((5, 3, 1), seed=2)
    ph = I.tgv_physics(Ma=0.2, Re=300.0)
    Q = np.random.default_rng(p).standard_normal((15, (p + 1) ** 3, 5)) + 3.0
    want = PJ.project([Q, np.zeros((0, (p + 1) ** 2 * (p + 2) // 2, 5))], p, q)[0]
    ph.precision = fr.FR_PREC_MIXED
    with fr.Mesh(d, ph, p) as a, fr.Mesh(d, ph, q) as b:
        a.set_state(Q)
        fr.project_state(a, b)
        np.testing.assert_allclose(b.get_state(), want, rtol=1e-13, atol=1e-13 * np.abs(want).max())


def test_one_mesh_twice_in_a_batch_keeps_its_order():
    """A batch that lists a mesh twice advances it twice per stage, one after the other: not side by side."""
    import torch
    d = I.hex_box_mesh((4, 4, 4), lo=(-5, -5, -5), hi=(5, 5, 5))
    ph = I.Physics(gamma=1.4, R=1.0, mu=0.0, viscous=0)
    st = torch.cuda.Stream()
    got = []
    with fr.Mesh(d, ph, 2, stream=st.cuda_stream) as m:
        Q = np.ascontiguousarray(I.isentropic_vortex_state(m.solution_points(), period=(10, 10)))
        for _ in range(2):
            m.set_state(Q)
            with fr.Batch([m, m]) as b:
                b.set_dt([1e-3, 1e-3])
                b.select(1)
                b.rk_step()
            got.append(m.get_state())
        m.set_state(Q)
        for s in range(4):
            m.rk_stage(s, 0.0, 1e-3)
            m.rk_stage(s, 0.0, 1e-3)
        want = m.get_state()
    assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], want)


def _flat(arrs):
    return np.concatenate([np.asarray(a).reshape(-1, 5) for a in arrs])


# Element counts at the limits of the volume kernel that splits an element's variables over thread groups (304 at
# p = 2 and 3, 152 at p = 4) and of the correction kernel with one thread per point (38912 points).
@pytest.mark.parametrize("p,box", [(1, (17, 17, 17)), (2, (19, 4, 4)), (2, (61, 5, 1)), (2, (12, 12, 11)),
                                   (3, (19, 4, 4)), (3, (61, 5, 1)), (3, (19, 8, 4)), (3, (29, 7, 3)), (4, (19, 4, 2)),
                                   (4, (17, 3, 3)), (4, (13, 6, 4)), (5, (8, 6, 4)), (6, (5, 5, 5)), (7, (5, 4, 4))])
def test_small_mesh_limits(p, box):
    d = I.hex_box_mesh(box, seed=6, rotate=True, affine=((1.0, 0.2, 0.0), (0.0, 1.0, 0.1), (0.1, 0.0, 1.0)))
    ph = I.tgv_physics(Ma=0.2, Re=400.0)
    ora = MixedFR(d, ph, p)
    Qs = [np.ascontiguousarray(I.tgv_state(x, Ma=0.2, perturb=1e-2, seed=1)) for x in ora.x]
    R, S, dt = _flat(ora.residual(Qs)), _flat(ora.residual(Qs, magnitude=True)), 2e-5
    ora.set_source(accel=(0.3, -0.2, 0.1))
    S1 = _flat(ora.residual(Qs, magnitude=True))
    want = [_flat(TI.rk44(ora.residual, Qs, dt))]
    if p == 3:
        want.append(_flat(TI.SCHEMES["ssprk33"](ora.residual, Qs, dt)))
    for precision, bar in [(fr.FR_PREC_FP64, 1e-12), (fr.FR_PREC_MIXED, 1e-9), (fr.FR_PREC_MIXED_VF32, 2e-8)]:
        ph.precision = precision
        with fr.Mesh(d, ph, p) as g:
            g.set_state(_flat(Qs))
            got = g.residual().reshape(-1, 5)
            if precision == fr.FR_PREC_MIXED_VF32:      # thin cells are mostly viscous: the suite's normwise bar
                assert (np.abs(got - R).max(axis=0) <= 1e-6 * np.abs(R).max(axis=0)).all()
            else:
                assert_residual_parity(got, R, S, bar)
            g.set_source(accel=(0.3, -0.2, 0.1))
            for scheme, w in zip((fr.FR_RK44, fr.FR_SSPRK33), want):
                g.set_state(_flat(Qs))
                g.rk_step(0.0, dt, scheme)
                assert_state_parity(g.get_state().reshape(-1, 5), w, S1, dt, bar)


@pytest.mark.parametrize("flux", [0, 1])
def test_zero_and_subnormal_values(flux):
    """Double-float values that the integer conversion to FP64 leaves to the instruction: zeros and FP32 subnormals."""
    d = I.hex_box_mesh((4, 3, 3), seed=2, rotate=True, perturb=0.1)
    ph = I.tgv_physics(Ma=0.2, Re=400.0)
    ph.inviscid_flux = flux
    ora = HexFR(d, ph, 3)
    Q = np.ascontiguousarray(I.tgv_state(ora.x, Ma=0.2, perturb=1e-2, seed=1))
    Q[:, ::3, 1:4] = (0.0, 1e-39, -3e-42)
    Q[:, 1::3, 0] = np.float32(1.25)
    S, dt = ora.residual(Q, magnitude=True), 1e-4
    ph.precision = fr.FR_PREC_MIXED
    with fr.Mesh(d, ph, 3) as g:
        g.set_state(Q)
        assert_residual_parity(g.residual(), ora.residual(Q), S, 1e-9)
        for scheme, f in ((fr.FR_RK44, TI.rk44), (fr.FR_SSPRK33, TI.SCHEMES["ssprk33"])):
            g.set_state(Q)
            g.rk_step(0.0, dt, scheme)
            assert_state_parity(g.get_state(), f(lambda q: [ora.residual(q[0])], [Q], dt)[0], S, dt, 1e-9)
