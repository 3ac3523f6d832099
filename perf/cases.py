"""What the framework's users have it compute, as measurable cases.

Each case is one pass of a user's program through the public binding (`paper_2308_06605_gb300.fr`):
a flow solver that is handed a state, advances it by whole Runge-Kutta steps and gives the new
state back; a single residual; a batched ensemble; one training step of the eddy-viscosity network;
the change of order at start-up.  Sizes are those of the benchmark, the configurations and the
tests, or smaller ones of the same kind where the host-side mesh build would take long.
`exact` evaluates the same scheme in plain torch in 64 bits with dense operators (module-level class
`Scheme`), independent of the library.
"""
import functools
import math

import numpy as np
import torch

from paper_2308_06605_gb300 import fr, inputs, perfmodel

PRECISION = {"fp64": 0, "mixed": 1, "vf32": 3}
SCHEME = {"rk44": 0, "ssp33": 1}


def listed():
    return [
        # The benchmark's workload, Taylor-Green vortex at p = 4 on the double-float path, 48^3 hexahedra.
        dict(name="tgv_mixed_48_p4", do="step", flow="tgv", n=48, p=4, precision="mixed", steps=1),
        # The same flow on the FP64 path (the binding's default precision).
        dict(name="tgv_fp64_32_p4", do="step", flow="tgv", n=32, p=4, precision="fp64", steps=1),
        # High order: the p-sweep's last member, on a smaller box.
        dict(name="tgv_mixed_20_p7", do="step", flow="tgv", n=20, p=7, precision="mixed", steps=1),
        # Fine runs of the closure's data generation: FP32 viscous branch.
        dict(name="tgv_vf32_40_p3", do="step", flow="tgv", n=40, p=3, precision="vf32", steps=1),
        # The small configuration: 8^3 hexahedra, p = 3, ten RK44 steps in FP64.
        dict(name="tgv_fp64_8_p3", do="step", flow="tgv", n=8, p=3, precision="fp64", steps=10),
        # The smallest call: one residual on a test-size unstructured mesh (perturbed, renumbered).
        dict(name="residual_fp64_4_p2", do="residual", flow="tgv", n=4, p=2, precision="fp64"),
        # Turbine-cascade passage: a quarter of the elements prisms, walls, characteristic in- and outflow.
        dict(name="passage_mixed_72_p4", do="step", flow="passage", n=72, p=4, precision="mixed", steps=1),
        # Body-force-driven channel between isothermal walls on an unstructured (perturbed, renumbered)
        # mesh with the paper's other options: Roe, LDG and the three-stage SSP scheme.
        dict(name="channel_mixed_15_p5", do="step", flow="channel", n=15, p=5, precision="mixed", steps=1),
        # Large-eddy run of the closure pipeline: coarse order, learned eddy viscosity, FP64.
        dict(name="les_fp64_24_p2", do="step", flow="les", n=24, p=2, precision="fp64", steps=1),
        # Ensemble of isentropic vortices of different sizes and orders, batched and tuned.
        dict(name="ensemble_mixed_16", do="batch", count=16, pick=0, precision="mixed", steps=1),
        # One optimiser step of the closure network at the pipeline's batch size.
        dict(name="closure_train_4096", do="train", n=4096),
        # Order sequencing: the state of a p = 2 start-up run carried over to p = 4.
        dict(name="project_32_p2_p4", do="project", n=32, p=2, q=4),
    ]


def draw(rng):
    def logint(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["tgv", "tgv", "tgv", "small", "residual", "passage", "channel", "les", "batch", "train", "project"])
    prec = rng.choice(["mixed", "mixed", "fp64", "vf32"])
    if kind == "tgv":           # up to 8 M points in the fast precisions, 3 M in FP64
        p = rng.randint(2, 7)
        top = (2.5e6 if prec == "fp64" else 8e6) ** (1 / 3) / (p + 1)
        return dict(do="step", flow="tgv", n=logint(5, max(6, top)), p=p, precision=prec, steps=1)
    if kind == "small":
        return dict(do="step", flow="tgv", n=rng.randint(3, 9), p=rng.randint(1, 4), precision=prec, steps=rng.randint(2, 10))
    if kind == "residual":      # the precision with which one residual is looked at by itself
        return dict(do="residual", flow="tgv", n=logint(3, 20), p=rng.randint(1, 5), precision="fp64")
    if kind == "passage":
        return dict(do="step", flow="passage", n=logint(20, 72), p=rng.randint(2, 4), precision=rng.choice(["mixed", "fp64"]), steps=1)
    if kind == "channel":
        return dict(do="step", flow="channel", n=rng.randint(5, 18), p=rng.randint(2, 5), precision=prec, steps=rng.randint(1, 2))
    if kind == "les":
        return dict(do="step", flow="les", n=rng.randint(8, 32), p=rng.randint(2, 3), precision=rng.choice(["fp64", "mixed"]), steps=rng.randint(1, 3))
    if kind == "batch":
        return dict(do="batch", count=rng.randint(4, 16), pick=rng.randint(1, 40), precision=rng.choice(["mixed", "fp64"]), steps=1)
    if kind == "train":
        return dict(do="train", n=logint(300, 16384))
    p = rng.randint(1, 4)
    return dict(do="project", n=rng.randint(8, 36), p=p, q=rng.choice([k for k in range(1, 5) if k != p]))


# ------------------------------------------------------------------------------------ workloads
@functools.lru_cache(maxsize=6)
def _workload(flow, n, p):
    """Mesh description, physics, time step and source of a flow case (host data; no states)."""
    if flow == "passage":
        phys, bcs, _ = inputs.cascade_conditions()
        k = max(1, n // 6)
        desc = inputs.blade_passage_mesh(n_up=k, n_blade=3 * k, n_down=k, ny=n // 2, nz=max(2, n // 5),
                                         n_prism_rows=max(1, n // 14), quadratic=False, bcs=bcs)
        h, lam = 0.3 / max(2, n // 5), 2.5
    elif flow == "channel":
        desc = inputs.hex_box_mesh((n, n, n), lo=(0, 0, 0), hi=(2.0, 1.0, 1.0), periodic=(True, False, True), seed=3,
                                   shuffle=True, rotate=True, perturb=0.1,
                                   wall_tags={3: (inputs.BC_WALL_ISOTHERMAL, (1.0,)), 4: (inputs.BC_WALL_ISOTHERMAL, (1.0,))})
        phys = inputs.Physics(gamma=1.4, R=1.0, mu=1e-3, Pr=0.71, inviscid_flux=1, viscous=2)
        h, lam = 0.6 / n, 2.0
    else:
        rough = flow == "rough"
        desc = inputs.hex_box_mesh((n, n, n), seed=1, shuffle=rough, rotate=rough, perturb=0.1 if rough else 0.0)
        phys = inputs.tgv_physics()
        h, lam = 2 * np.pi / n, 11.5
    return desc, phys, 0.3 * h / ((p + 1) ** 2 * lam), ((0.02, 0.0, 0.0) if flow == "channel" else None)


def _physics(phys, precision):
    return inputs.Physics(**{**phys.__dict__, "precision": PRECISION[precision]})


def _flow_of(case):
    return "rough" if case["do"] == "residual" else case["flow"]


def _modes(x, seed, amplitude, waves):
    """Three velocity components of random-phase Fourier modes at the points x [..., 3]."""
    r = np.random.default_rng(seed)
    out = []
    for _ in range(3):
        v = torch.zeros_like(x[..., 0])
        for _ in range(3):
            k = r.integers(1, 4, size=3) * np.asarray(waves)
            v = v + amplitude * torch.sin(x[..., 0] * k[0] + x[..., 1] * k[1] + x[..., 2] * k[2] + r.uniform(0, 2 * np.pi))
        out.append(v)
    return out


def _conserved(rho, u, p, gamma=1.4):
    return torch.stack([rho] + [rho * c for c in u] + [p / (gamma - 1) + 0.5 * rho * sum(c * c for c in u)], -1)


def _state(flow, x, seed):
    """A flow's state at the points x [..., 3] (a torch FP64 tensor)."""
    X, Y, Z = x[..., 0], x[..., 1], x[..., 2]
    if flow == "passage":
        m = _modes(x, seed, 1e-3, (2 * np.pi, 2 * np.pi / 0.8, 2 * np.pi / 0.3))
        f = 1 + 0.2 * 0.15 ** 2
        T, p = 1 / f, f ** -3.5
        U = 0.15 * math.sqrt(1.4 * T)
        u = [U * math.cos(math.pi / 6) + m[0], U * math.sin(math.pi / 6) + m[1], m[2]]
        return _conserved(torch.full_like(X, p / T), u, torch.full_like(X, p))
    if flow == "channel":
        m = _modes(x, seed, 5e-3, (np.pi, 2 * np.pi, 2 * np.pi))
        return _conserved(torch.ones_like(X), [0.4 * Y * (1 - Y) * 4 + m[0], m[1], m[2]], torch.ones_like(X))
    m = _modes(x, seed, 1e-2, (1, 1, 1))
    p0 = 1 / (1.4 * 0.01)
    p = p0 + (torch.cos(2 * X) + torch.cos(2 * Y)) * (torch.cos(2 * Z) + 2) / 16
    u = [torch.sin(X) * torch.cos(Y) * torch.cos(Z) + m[0], -torch.cos(X) * torch.sin(Y) * torch.cos(Z) + m[1], m[2]]
    return _conserved(p / p0, u, p)


def _vortices(case):
    """Edge counts and orders of the ensemble's members (their seeds pick both, as in the benchmark)."""
    return inputs.vortex_ensemble(case["count"], seed0=case["pick"] * 100)


@functools.lru_cache(maxsize=32)
def _vortex_mesh(n, L):
    return inputs.hex_box_mesh((n, n, n), lo=(-L / 2,) * 3, hi=(L / 2,) * 3)


def _vortex_state(x, seed, k, L):
    c = np.random.default_rng([seed, k]).uniform(-L / 2, L / 2, 2)
    dx, dy = x[..., 0] - c[0], x[..., 1] - c[1]
    dx, dy = dx - L * torch.round(dx / L), dy - L * torch.round(dy / L)
    f = torch.exp(0.5 * (1 - dx * dx - dy * dy))
    U, b = 0.5 * math.sqrt(0.7), 5 / (2 * math.pi)
    T = 1 - 0.4 * 25 / (8 * 1.4 * math.pi ** 2) * f * f
    rho = T ** 2.5
    return _conserved(rho, [U - b * f * dy, U + b * f * dx, torch.zeros_like(rho)], rho * T)


def _vortex_dt(n, p, L):
    return 0.3 * (L / n) / ((p + 1) ** 2 * 2.5)


def _network(seed, device):
    """Weights (rounded to bfloat16's values where the solver does so), input and output scales."""
    r = np.random.default_rng([seed, 7])
    P = np.zeros(fr.N_CLOSURE_PARAMS, dtype=np.float32)
    o = 0
    for a, b in ((11, 64), (64, 64), (64, 64)):
        P[o:o + a * b] = r.standard_normal(a * b) * math.sqrt(2.0 / a)
        P[o + a * b:o + a * b + b] = 0.05 * r.standard_normal(b)
        o += a * b + b
    P[o:o + 64] = 0.1 * r.standard_normal(64)
    scales = np.concatenate([np.zeros(11), np.ones(11), [1e-2]]).astype(np.float32)
    scales[10], scales[21] = 0.1, 0.05
    return P, scales


def _samples(n, seed, device):
    """A minibatch of closure features (velocity gradient, strain, filter width) and targets."""
    g = torch.Generator(device="cpu").manual_seed(int(seed))
    X = torch.randn(n, 11, generator=g)
    S = X[:, :9].reshape(n, 3, 3)
    S = 0.5 * (S + S.transpose(1, 2))
    X[:, 9] = torch.sqrt(2 * (S * S).sum((1, 2)))
    X[:, 10] = 0.05 + 0.1 * torch.rand(n, generator=g)
    y = torch.relu(torch.randn(n, generator=g)) * X[:, 9]
    return X.to(device), y.to(device)


def _moments(n, seed, device):
    g = torch.Generator(device="cpu").manual_seed(int(seed) + 99)
    return (1e-2 * torch.randn(n, generator=g)).to(device), (1e-4 + 1e-3 * torch.rand(n, generator=g)).to(device)


def prepare(case, seed):
    do = case["do"]
    if do == "train":
        P, scales = _network(seed, "cuda")
        tr = fr.MLPTrainer(P, scales, max_batch=case["n"])
        m, v = _moments(P.size, seed, "cuda")
        tr.m.copy_(m)
        tr.v.copy_(v)
        tr.step_count = 10
        return dict(do=do, tr=tr, xy=_samples(case["n"], seed, "cuda"))
    if do == "batch":
        stream = torch.cuda.Stream()
        meshes, dts, Q, out = [], [], [], []
        for k, c in enumerate(_vortices(case)):
            phys = inputs.Physics(gamma=1.4, R=1.0, mu=0.0, viscous=0, precision=PRECISION[case["precision"]])
            m = fr.Mesh(_vortex_mesh(c["n"], c["L"]), phys, c["p"], stream=stream.cuda_stream)
            Q.append(_vortex_state(torch.from_numpy(m.solution_points()).cuda(), seed, k, c["L"]).contiguous())
            out.append(torch.empty_like(Q[-1]))
            dts.append(_vortex_dt(c["n"], c["p"], c["L"]))
            meshes.append(m)
        torch.cuda.synchronize()
        for m, q in zip(meshes, Q):
            m.set_state(q)
        b = fr.Batch(meshes)
        b.tune()
        b.set_dt(dts)
        return dict(do=do, batch=b, meshes=meshes, Q=Q, out=out, steps=case["steps"], stream=stream)
    flow = _flow_of(case) if do != "project" else "tgv"
    desc, phys, dt, accel = _workload(flow, case["n"], case["p"])
    mesh = fr.Mesh(desc, _physics(phys, case.get("precision", "fp64")), case["p"])
    if accel is not None:
        mesh.set_source(accel=accel)
    if flow == "les":
        mesh.set_closure(*_network(seed, "cuda"))
    Q = _state(flow, torch.from_numpy(mesh.solution_points()).cuda(), seed).contiguous()
    s = dict(do=do, mesh=mesh, Q=Q, dt=dt, steps=case.get("steps", 1))
    if do == "project":
        s["to"] = fr.Mesh(desc, phys, case["q"])
        s["out"] = torch.empty(s["to"].shape, dtype=torch.float64, device="cuda")
        mesh.set_state(Q)
    else:
        s["out"] = torch.empty_like(Q)
        s["scheme"] = SCHEME["ssp33" if flow == "channel" else "rk44"]
    return s


def run(s):
    do = s["do"]
    if do == "train":
        loss, grad = s["tr"].loss_grad(*s["xy"])
        s["tr"].adam(2e-3)
        return {"loss": loss, "grad": grad, "params": s["tr"].P, "m": s["tr"].m, "v": s["tr"].v}
    if do == "batch":
        for m, q in zip(s["meshes"], s["Q"]):
            m.set_state(q)
        for _ in range(s["steps"]):
            s["batch"].rk_step()
        return [m.get_state(out=o) for m, o in zip(s["meshes"], s["out"])]
    if do == "project":
        fr.project_state(s["mesh"], s["to"])
        return s["to"].get_state(out=s["out"])
    s["mesh"].set_state(s["Q"])
    if do == "residual":
        return s["mesh"].residual(out=s["out"])
    for k in range(s["steps"]):
        s["mesh"].rk_step(k * s["dt"], s["dt"], s["scheme"])
    return s["mesh"].get_state(out=s["out"])


def work(case):
    """Bytes: the state in and out and the metric terms at the points, once; operations: the
    algorithmic count of every stage (`perfmodel`)."""
    do = case["do"]
    if do == "train":
        n, w = case["n"], fr.N_CLOSURE_PARAMS
        return {"bytes": 4.0 * (12 * n + 8 * w), "flops": 6.0 * n * (11 * 64 + 2 * 64 * 64 + 64)}
    if do == "batch":
        t = {"bytes": 0.0, "flops": 0.0}
        for c in _vortices(case):
            pts = (c["n"] * (c["p"] + 1)) ** 3
            t["bytes"] += 160.0 * pts
            t["flops"] += 4.0 * case["steps"] * pts * sum(perfmodel.flops_per_point(c["p"], False).values())
        return t
    if do == "project":
        a, b = (case["n"] * (case["p"] + 1)) ** 3, (case["n"] * (case["q"] + 1)) ** 3
        return {"bytes": 40.0 * (a + b), "flops": 10.0 * b * 3 * (case["p"] + 1)}
    p, n = case["p"], case["n"]
    desc, _, _, _ = _workload(_flow_of(case), n, p)
    hexes, prisms = len(desc.hex) * (p + 1) ** 3, len(desc.prism) * (p + 1) ** 2 * (p + 2) // 2
    stages = 1 if do == "residual" else case["steps"] * (3 if case["flow"] == "channel" else 4)
    per = [sum(f(p).values()) for f in (perfmodel.flops_per_point, perfmodel.prism_flops_per_point)]
    return {"bytes": 160.0 * (hexes + prisms), "flops": float(stages * (hexes * per[0] + prisms * per[1]))}


# ---------------------------------------------------------------------- the scheme in 64 bits
HEX = np.array([[-1, -1, -1], [1, -1, -1], [1, 1, -1], [-1, 1, -1], [-1, -1, 1], [1, -1, 1], [1, 1, 1], [-1, 1, 1]], float)


def _legvals(x, p):
    return np.polynomial.legendre.legvander(np.asarray(x, float), p)


def _legders(x, p):
    return np.stack([np.polynomial.legendre.legval(x, np.polynomial.legendre.legder(np.eye(p + 1)[k])) for k in range(p + 1)], -1)


class Line:
    def __init__(self, p):
        self.x, self.w = np.polynomial.legendre.leggauss(p + 1)
        Vi = np.linalg.inv(_legvals(self.x, p))
        self.D = _legders(self.x, p) @ Vi
        self.lo, self.hi = (_legvals(s, p)[0] @ Vi for s in ([-1.0], [1.0]))


class Triangle:
    """Nodal basis on the warp-and-blend nodes (Warburton 2006); span of P_i(r) P_j(s), i + j <= p."""
    ALPHA = [0.0, 0.0, 1.4152, 0.1001, 0.2751, 0.9800, 1.0999]

    def __init__(self, p):
        self.p = p
        L1, L3 = np.array([(n / p, m / p) for n in range(p + 1) for m in range(p + 1 - n)]).T
        L2 = 1 - L1 - L3
        even = np.linspace(-1, 1, p + 1)
        inner = np.sort(np.polynomial.legendre.Legendre.basis(p).deriv().roots().real) if p > 1 else []
        shift = np.concatenate([[-1.0], inner, [1.0]]) - even

        def warp(r):
            v = sum(shift[i] * np.prod([(r - even[j]) / (even[i] - even[j]) for j in range(p + 1) if j != i], axis=0) for i in range(p + 1))
            ins = np.abs(r) < 1 - 1e-10
            return np.where(ins, v / np.where(ins, 1 - r * r, 1.0), 0.0)
        al = self.ALPHA[p - 1]
        f = [4 * a * b * warp(c) * (1 + (al * d) ** 2) for a, b, c, d in ((L2, L3, L3 - L2, L1), (L1, L3, L1 - L3, L2), (L1, L2, L2 - L1, L3))]
        X = -L2 + L3 + f[0] - 0.5 * f[1] - 0.5 * f[2]
        Y = (-L2 - L3 + 2 * L1) / math.sqrt(3) + math.sin(2 * math.pi / 3) * f[1] + math.sin(4 * math.pi / 3) * f[2]
        l1, l2, l3 = (math.sqrt(3) * Y + 1) / 3, (-3 * X - math.sqrt(3) * Y + 2) / 6, (3 * X - math.sqrt(3) * Y + 2) / 6
        self.rs = np.stack([-l2 + l3 - l1, -l2 - l3 + l1], 1)
        self.Vi = np.linalg.inv(self.modes(self.rs))
        self.Dr, self.Ds = (self.modes(self.rs, d) @ self.Vi for d in (0, 1))
        a, wa = np.polynomial.legendre.leggauss(p + 3)
        A, S = np.meshgrid(a, a)
        pts = np.stack([(0.5 * (1 + A) * (1 - S) - 1).ravel(), S.ravel()], 1)
        B = self.at(pts)
        self.M = B.T @ (B * (np.outer(wa, wa) * 0.5 * (1 - S)).ravel()[:, None])

    def modes(self, rs, d=None):
        p = self.p
        a, b = _legvals(rs[:, 0], p), _legvals(rs[:, 1], p)
        a, b = (_legders(rs[:, 0], p) if d == 0 else a), (_legders(rs[:, 1], p) if d == 1 else b)
        return np.stack([a[:, i] * b[:, j] for i in range(p + 1) for j in range(p + 1 - i)], 1)

    def at(self, rs):
        return self.modes(np.asarray(rs)) @ self.Vi


def _hex_type(p):
    b, I = Line(p), np.eye(p + 1)
    N = p + 1
    k3 = lambda x, y, z: np.kron(z, np.kron(y, x))          # noqa: E731  first axis fastest
    pts = np.stack([np.tile(b.x, N * N), np.tile(np.repeat(b.x, N), N), np.repeat(b.x, N * N)], 1)
    faces = []
    for f in range(6):
        d, s = f // 2, 2 * (f % 2) - 1
        l = b.hi if s > 0 else b.lo
        ops = [I, I, I]
        ops[d] = l[None, :]
        L = k3(*ops)
        ops[d] = (l / b.w)[:, None]
        fp = np.zeros((N * N, 3))
        t = [a for a in range(3) if a != d]
        fp[:, t[0]], fp[:, t[1]], fp[:, d] = np.tile(b.x, N), np.repeat(b.x, N), s
        faces.append(dict(L=L, C=k3(*ops), N=s * np.eye(3)[d], pts=fp, corners=np.where(HEX[:, d] == s)[0]))
    return dict(D=[k3(b.D, I, I), k3(I, b.D, I), k3(I, I, b.D)], pts=pts, faces=faces, W=np.kron(b.w, np.kron(b.w, b.w)))


def _hex_shape(r):
    N = np.prod(1 + r[:, None, :] * HEX[None], axis=2) / 8
    dN = np.stack([HEX[None, :, a] * np.prod(np.delete(1 + r[:, None, :] * HEX[None], a, axis=2), axis=2) / 8 for a in range(3)], 2)
    return N, dN


def _prism_type(p):
    b, T = Line(p), Triangle(p)
    N, Nt = p + 1, len(T.rs)
    I, It = np.eye(N), np.eye(Nt)
    flat = lambda rs, z: np.concatenate([np.tile(rs, (len(z), 1)), np.repeat(z, len(rs))[:, None]], 1)   # noqa: E731
    faces = []
    for s, l, corners in ((-1, b.lo, [0, 1, 2]), (1, b.hi, [3, 4, 5])):
        faces.append(dict(L=np.kron(l[None], It), C=np.kron((l / b.w)[:, None], It), N=np.array([0.0, 0.0, s]),
                          pts=flat(T.rs, np.array([float(s)])), corners=np.array(corners)))
    o = np.ones(N)
    for rs, nrm, corners in ((np.stack([b.x, -o], 1), (0.0, -1.0, 0.0), [0, 1, 4, 3]), (np.stack([-b.x, b.x], 1), (1.0, 1.0, 0.0), [1, 2, 5, 4]),
                             (np.stack([-o, -b.x], 1), (-1.0, 0.0, 0.0), [2, 0, 3, 5])):
        E = T.at(rs)
        faces.append(dict(L=np.kron(I, E), C=np.kron(I, np.linalg.solve(T.M, E.T * b.w[None])), N=np.array(nrm), pts=flat(rs, b.x), corners=np.array(corners)))
    return dict(D=[np.kron(I, T.Dr), np.kron(I, T.Ds), np.kron(b.D, It)], pts=flat(T.rs, b.x), faces=faces, W=np.kron(b.w, T.M.sum(1)))


def _prism_shape(r):
    lam = np.stack([-(r[:, 0] + r[:, 1]) / 2, (1 + r[:, 0]) / 2, (1 + r[:, 1]) / 2], 1)
    dl = np.array([[-0.5, -0.5], [0.5, 0.0], [0.0, 0.5]])
    lo, hi = ((1 - r[:, 2]) / 2)[:, None], ((1 + r[:, 2]) / 2)[:, None]
    dN = np.stack([np.concatenate([dl[None, :, a] * lo, dl[None, :, a] * hi], 1) for a in (0, 1)] + [np.concatenate([-lam / 2, lam / 2], 1)], 2)
    return np.concatenate([lam * lo, lam * hi], 1), dN


def _cross(a, b):
    return torch.linalg.cross(a, b, dim=-1)


def _prim(q, g):
    u = q[..., 1:4] / q[..., :1]
    return q[..., 0], u, (g - 1) * (q[..., 4] - 0.5 * (q[..., 1:4] * u).sum(-1))


def _inviscid(q, g):
    rho, u, p = _prim(q, g)
    F = u[..., :, None] * q[..., None, :]                     # [..., direction, variable]
    for j in range(3):
        F[..., j, 1 + j] += p
    F[..., 4] += u * p[..., None]
    return F


def _viscous(q, G, ph, mu, kappa):
    rho, u, _ = _prim(q, ph.gamma)
    du = (G[..., 1:4] - u[..., None, :] * G[..., :1]) / rho[..., None, None]        # [..., j, i] = du_i/dx_j
    dT = (ph.gamma - 1) / ph.R * ((G[..., 4] - (q[..., 4] / rho)[..., None] * G[..., 0]) / rho[..., None] - (du * u[..., None, :]).sum(-1))
    tau = mu[..., None, None] * (du + du.transpose(-1, -2))
    div = torch.diagonal(du, dim1=-2, dim2=-1).sum(-1) * mu * (2.0 / 3.0)
    tau = tau - div[..., None, None] * torch.eye(3, dtype=q.dtype, device=q.device)
    return torch.cat([torch.zeros_like(tau[..., :1]), tau, ((tau * u[..., None, :]).sum(-1) + kappa[..., None] * dT)[..., None]], -1)


def _common(kind, a, b, n, g):
    F = 0.5 * ((_inviscid(a, g) + _inviscid(b, g)) * n[..., None]).sum(-2)
    nn = n.norm(dim=-1)
    h = n / nn[..., None]
    (ra, ua, pa), (rb, ub, pb) = _prim(a, g), _prim(b, g)
    if kind == 0:
        lam = torch.maximum((ua * h).sum(-1).abs() + torch.sqrt(g * pa / ra), (ub * h).sum(-1).abs() + torch.sqrt(g * pb / rb))
        return F - 0.5 * (lam * nn)[..., None] * (b - a)
    sa, sb = torch.sqrt(ra)[..., None], torch.sqrt(rb)[..., None]
    u = (sa * ua + sb * ub) / (sa + sb)
    H = ((sa[..., 0] * (a[..., 4] + pa) / ra) + sb[..., 0] * (b[..., 4] + pb) / rb) / (sa + sb)[..., 0]
    r, q2, un, du = (sa * sb)[..., 0], (u * u).sum(-1), (u * h).sum(-1), ub - ua
    c = torch.sqrt((g - 1) * (H - 0.5 * q2))
    dun, dp = (du * h).sum(-1), pb - pa
    out = torch.zeros_like(a)
    for s in (-1.0, 1.0):
        lam, d = un + s * c, 0.1 * c
        lam = torch.where(lam.abs() < d, (lam * lam + d * d) / (2 * d), lam.abs()) * (dp + s * r * c * dun) / (2 * c * c)
        out += lam[..., None] * torch.cat([torch.ones_like(c)[..., None], u + s * c[..., None] * h, (H + s * c * un)[..., None]], -1)
    sh, w = r[..., None] * (du - dun[..., None] * h), (rb - ra - dp / (c * c))[..., None]
    out += un.abs()[..., None] * torch.cat([w, w * u + sh, 0.5 * w * q2[..., None] + (u * sh).sum(-1, keepdim=True)], -1)
    return F - 0.5 * nn[..., None] * out


def _boundary(bc, q, n, ph):
    """Exterior state of the inviscid flux and common solution of the viscous terms."""
    g, R, par = ph.gamma, ph.R, bc.params
    rho, u, p = _prim(q, g)
    if bc.kind == inputs.BC_WALL_ISOTHERMAL:
        ghost, qi = q.clone(), torch.zeros_like(q)
        ghost[..., 1:4] *= -1
        qi[..., 0], qi[..., 4] = rho, rho * R * par[0] / (g - 1)
        return ghost, qi
    h = n / n.norm(dim=-1, keepdim=True)
    un = (u * h).sum(-1)
    out = un + 2 * torch.sqrt(g * p / rho) / (g - 1)
    if bc.kind == inputs.BC_CHAR_OUTFLOW:
        pb = torch.full_like(p, par[0])
        rb = (pb / (p / rho ** g)) ** (1 / g)
        ub = u + (out - 2 * torch.sqrt(g * pb / rb) / (g - 1) - un)[..., None] * h
    else:
        d = torch.tensor(par[2:5], dtype=q.dtype, device=q.device)
        d = d / d.norm()
        a, k = h @ d, 2 / (g - 1)
        A, B, C = a * a + k, -2 * a * out, out * out - k * k * g * R * par[1]
        V = (-B + torch.sqrt(B * B - 4 * A * C)) / (2 * A)
        Tb = par[1] - V * V * (g - 1) / (2 * g * R)
        pb = par[0] * (Tb / par[1]) ** (g / (g - 1))
        rb, ub = pb / (R * Tb), V[..., None] * d
    qi = torch.cat([rb[..., None], rb[..., None] * ub, (pb / (g - 1) + 0.5 * rb * (ub * ub).sum(-1))[..., None]], -1)
    return qi, qi


class Scheme:
    """Flux reconstruction with the DG correction on straight-sided hexahedra and prisms, dense
    operators, all faces of the mesh in one buffer; torch FP64 on the GPU."""

    def __init__(self, desc, phys, p, accel=None, net=None, dev="cuda"):
        self.ph, self.accel, self.net, self.N, self.dev = phys, accel, net, p + 1, dev
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)   # noqa: E731
        xyz = t(desc.xyz)
        nf = (p + 1) ** 2
        self.types, keys, base, corners_all = [], [], 0, []
        for make, shape, conn in ((_hex_type, _hex_shape, desc.hex), (_prism_type, _prism_shape, desc.prism)):
            if len(conn) == 0:
                continue
            T = make(p)
            cn = torch.as_tensor(conn, device=dev)
            V = xyz[cn]

            def geometry(ref):
                n, dn = shape(ref)
                J = [torch.einsum("mv,evi->emi", t(dn[:, :, a]), V) for a in range(3)]
                S = torch.stack([_cross(J[1], J[2]), _cross(J[2], J[0]), _cross(J[0], J[1])], 2)
                return torch.einsum("mv,evi->emi", t(n), V), (J[0] * S[:, :, 0]).sum(-1), S

            k = dict(D=[t(d) for d in T["D"]], W=t(T["W"]), E=len(conn), faces=[])
            k["x"], k["J"], k["S"] = geometry(T["pts"])
            for f in T["faces"]:
                xf, _, Sf = geometry(f["pts"])
                m = len(f["pts"])
                pad = lambda a: torch.cat([a, a[:, :1].expand(-1, nf - m, -1)], 1)       # noqa: E731
                k["faces"].append(dict(L=t(f["L"]), C=t(f["C"]), N=t(f["N"]), m=m, at=base))
                keys.append((pad(xf), pad((t(f["N"])[None, None, :, None] * Sf).sum(2)), np.full(len(conn), m)))
                c = np.full((len(conn), 4), -1, np.int64)
                c[:, :len(f["corners"])] = np.sort(conn[:, f["corners"]], axis=1)
                corners_all.append(c)
                base += len(conn)
            self.types.append(k)
        X, self.n, count = torch.cat([k[0] for k in keys]), torch.cat([k[1] for k in keys]), np.concatenate([k[2] for k in keys])
        corners = np.concatenate(corners_all)
        # Tags of boundary faces by their sorted corner ids, periodic shifts, pairs by shifted centroids.
        bn = np.asarray(desc.bface_nodes)
        bn = np.sort(np.where(bn < 0, np.iinfo(np.int64).max, bn), axis=1)
        bn = np.where(bn == np.iinfo(np.int64).max, -1, bn)
        big = int(corners.max()) + 2
        code = lambda c: ((c[:, 0] * big + c[:, 1]) * big + c[:, 2])                      # noqa: E731
        order = np.argsort(code(bn))
        sortedc = code(bn)[order]
        mine = code(corners)
        pos = np.clip(np.searchsorted(sortedc, mine), 0, max(0, len(sortedc) - 1))
        tag = np.where(sortedc[pos] == mine, np.asarray(desc.bface_tag)[order][pos], 0) if len(sortedc) else np.zeros(base, int)
        shift = np.zeros((base, 3))
        paired = tag == 0
        for q in desc.periodic:
            shift[tag == q.tag_b] = q.t
            paired |= (tag == q.tag_a) | (tag == q.tag_b)
        vert = desc.xyz[np.where(corners < 0, corners[:, :1], corners)]
        cen = np.where((corners >= 0)[..., None], vert, 0).sum(1) / (corners >= 0).sum(1)[:, None] - shift
        scale = np.ptp(desc.xyz, axis=0).max()
        ids = np.where(paired)[0]
        grid = np.round(cen[ids] / scale * 2 ** 20 + 0.371).astype(np.int64)
        o = np.lexsort(grid.T)
        a, b = ids[o[0::2]], ids[o[1::2]]
        if len(ids) % 2 or np.abs(cen[a] - cen[b]).max() > 1e-6 * scale:
            raise ValueError("faces do not pair up")
        partner = np.arange(base)
        partner[a], partner[b] = b, a
        self.partner = torch.as_tensor(partner, device=dev)
        Y = X - t(shift)[:, None]
        self.perm = torch.empty(base, nf, dtype=torch.int64, device=dev)
        step = max(1, 20_000_000 // (nf * nf))
        for i in range(0, base, step):
            A, B = Y[i:i + step], Y[self.partner[i:i + step]]
            d = sum((A[:, :, None, c] - B[:, None, :, c]) ** 2 for c in range(3))
            self.perm[i:i + step] = d.argmin(2)
        self.bcs = [(bc, torch.as_tensor(np.where((tag == bc.tag) & ~paired)[0], device=dev)) for bc in desc.bcs]
        self.edge = torch.as_tensor(~paired, device=dev)
        self.up = (self.n * (torch.arange(nf, device=dev)[None, :] < t(count)[:, None])[..., None]).sum(1) @ t([1.0, math.sqrt(2) / 2, math.sqrt(3) / 4]) > 0
        self.nf = nf

    def points(self):
        return [k["x"] for k in self.types]

    def across(self, a):
        i = self.perm.reshape(self.perm.shape + (1,) * (a.dim() - 2)).expand((-1, -1) + a.shape[2:])
        return a[self.partner].gather(1, i)

    def to_faces(self, parts):
        """Per-type, per-face [E, m, ...] blocks -> one [faces, nf, ...] buffer (padded with point 0)."""
        out = []
        for k, fs in zip(self.types, parts):
            for f, a in zip(k["faces"], fs):
                out.append(a if f["m"] == self.nf else torch.cat([a, a[:, :1].expand((-1, self.nf - f["m"]) + (-1,) * (a.dim() - 2))], 1))
        return torch.cat(out)

    def eddy(self, k, q, G):
        """Eddy viscosity of each element from the mean corrected velocity gradient."""
        P, sc = self.net
        w = k["W"] * k["J"]
        du = (G[..., 1:4] - (q[..., 1:4] / q[..., :1])[..., None, :] * G[..., :1]) / q[..., :1, None]
        g = torch.einsum("em,emji->eij", w, du) / w.sum(1)[:, None, None]
        S = 0.5 * (g + g.transpose(1, 2))
        h = ((k["W"] * k["J"]).sum(1)) ** (1 / 3) / self.N
        x = torch.cat([g.reshape(-1, 9), torch.sqrt(2 * (S * S).sum((1, 2)))[:, None], h[:, None]], 1)
        P = torch.as_tensor(P).to(torch.bfloat16).double().to(x.device)
        sc = torch.as_tensor(sc).double().to(x.device)
        return sc[22] * h * h * _net(P, (x - sc[:11]) / sc[11:22])

    def residual(self, Qs):
        ph, T = self.ph, self.types
        visc = ph.viscous != 0 and ph.mu > 0
        ldg = visc and ph.viscous == 2
        mv = lambda A, q: torch.einsum("mn,en...->em...", A, q)                      # noqa: E731
        Qf = self.to_faces([[mv(f["L"], q) for f in k["faces"]] for k, q in zip(T, Qs)])
        Qo = self.across(Qf)
        qi = torch.where(self.up[:, None, None], Qf, Qo) if ldg else 0.5 * (Qf + Qo)
        gh = Qo.clone()
        for bc, i in self.bcs:
            if len(i):
                gh[i], qi[i] = _boundary(bc, Qf[i], self.n[i], ph)
        F = _common(ph.inviscid_flux, Qf, gh, self.n, ph.gamma)
        kappa = ph.mu * ph.gamma * ph.R / ((ph.gamma - 1) * ph.Pr) if visc else 0.0
        Fh, parts, nus = [], [], []
        for k, q in zip(T, Qs):
            H = _inviscid(q, ph.gamma)
            if visc:
                Ji = k["S"] / k["J"][..., None, None]
                gu = torch.stack([mv(d, q) for d in k["D"]], 2)
                lifts = [mv(f["C"], (qi - Qf)[f["at"]:f["at"] + k["E"], :f["m"]]) for f in k["faces"]]
                gc = gu + sum(l[:, :, None, :] * f["N"][:, None] for l, f in zip(lifts, k["faces"]))
                phys = lambda r: torch.einsum("emdj,emdv->emjv", Ji, r)              # noqa: E731
                G = phys(gc)
                Gu = phys(gu)
                parts.append([mv(f["L"], G) if ldg else mv(f["L"], Gu + ph.br2_eta * phys(l[:, :, None, :] * f["N"][:, None]))
                              for l, f in zip(lifts, k["faces"])])
                nu = self.eddy(k, q, G) if self.net is not None else torch.zeros(k["E"], dtype=q.dtype, device=q.device)
                nus += [nu] * len(k["faces"])
                ev = q[..., 0] * nu[:, None]
                H = H - _viscous(q, G, ph, ph.mu + ev, kappa + ev * ph.gamma * ph.R / ((ph.gamma - 1) * 0.9))
            Fh.append(torch.einsum("emdj,emjv->emdv", k["S"], H))
        if visc:
            g = self.to_faces(parts)
            other = self.across(g)
            inner = self.edge[:, None, None, None]
            g = torch.where(inner, g, torch.where(self.up[:, None, None, None], other, g) if ldg else 0.5 * (g + other))
            nu = torch.cat(nus)
            nu = torch.where(self.edge, nu, 0.5 * (nu + nu[self.partner]))
            ev = qi[..., 0] * nu[:, None]
            F = F - (_viscous(qi, g, ph, ph.mu + ev, kappa + ev * ph.gamma * ph.R / ((ph.gamma - 1) * 0.9)) * self.n[..., None]).sum(-2)
            if ldg:
                o = torch.where(self.edge[:, None, None], qi, Qo)
                F = F + ph.ldg_tau * self.n.norm(dim=-1, keepdim=True) * (Qf - o)
        out = []
        for k, q, h in zip(T, Qs, Fh):
            R = sum(mv(d, h[:, :, i]) for i, d in enumerate(k["D"]))
            for f in k["faces"]:
                R = R + mv(f["C"], F[f["at"]:f["at"] + k["E"], :f["m"]] - mv(f["L"], (h * f["N"][:, None]).sum(2)))
            R = -R / k["J"][..., None]
            if self.accel is not None:
                a = torch.tensor(self.accel, dtype=q.dtype, device=q.device)
                R[..., 1:4] += q[..., :1] * a
                R[..., 4] += q[..., 1:4] @ a
            out.append(R)
        return out

    def step(self, Q, dt, scheme):
        add = lambda x, c, y: [a + c * b for a, b in zip(x, y)]                      # noqa: E731
        if scheme == "ssp33":
            U = Q
            for a, b in ((0.0, 1.0), (0.75, 0.25), (1 / 3, 2 / 3)):
                U = [a * q + b * v for q, v in zip(Q, add(U, dt, self.residual(U)))]
            return U
        acc, U = Q, Q
        for c, w in ((0.5, 1 / 6), (0.5, 1 / 3), (1.0, 1 / 3), (0.0, 1 / 6)):
            R = self.residual(U)
            acc, U = add(acc, w * dt, R), add(Q, c * dt, R)
        return acc


def _net(P, x):
    o = 0
    for a in (11, 64, 64):
        W, b = P[o:o + 64 * a].reshape(64, a), P[o + 64 * a:o + 64 * a + 64]
        x = torch.nn.functional.gelu(x @ W.T + b)
        o += 64 * a + 64
    return torch.nn.functional.softplus(x @ P[o:o + 64] + P[o + 64], threshold=1e9)


def _cat(parts, like_mixed):
    return torch.cat([q.reshape(-1, 5) for q in parts]) if like_mixed else parts[0]


def exact(case, seed):
    do = case["do"]
    if do == "train":
        P0, scales = _network(seed, "cuda")
        sc = torch.as_tensor(scales).double().cuda()
        P = torch.as_tensor(P0).double().cuda().requires_grad_(True)
        X, y = (a.double() for a in _samples(case["n"], seed, "cuda"))
        loss = ((_net(P, (X - sc[:11]) / sc[11:22]) - y) ** 2).mean()
        g, = torch.autograd.grad(loss, P)
        m, v = (a.double() for a in _moments(P0.size, seed, "cuda"))
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        new = P.detach() - 2e-3 * (m / (1 - 0.9 ** 11)) / (torch.sqrt(v / (1 - 0.999 ** 11)) + 1e-8)
        return {"loss": loss.detach().reshape(1), "grad": g, "params": new, "m": m, "v": v}
    if do == "batch":
        out = []
        for k, c in enumerate(_vortices(case)):
            s = Scheme(_vortex_mesh(c["n"], c["L"]), inputs.Physics(gamma=1.4, R=1.0, mu=0.0, viscous=0), c["p"])
            Q = [_vortex_state(x, seed, k, c["L"]) for x in s.points()]
            for _ in range(case["steps"]):
                Q = s.step(Q, _vortex_dt(c["n"], c["p"], c["L"]), "rk44")
            out.append(Q[0])
        return out
    flow = _flow_of(case) if do != "project" else "tgv"
    desc, phys, dt, accel = _workload(flow, case["n"], case["p"])
    s = Scheme(desc, phys, case["p"], accel, _network(seed, "cuda") if flow == "les" else None)
    Q = [_state(flow, x, seed) for x in s.points()]
    if do == "project":
        a, b = Line(case["p"]), Line(case["q"])
        m = min(case["p"], case["q"]) + 1
        L = _legvals(b.x, case["q"])[:, :m] @ np.linalg.inv(_legvals(a.x, case["p"]))[:m]
        return torch.einsum("mn,env->emv", torch.as_tensor(np.kron(L, np.kron(L, L)), device="cuda"), Q[0])
    mixed = len(desc.prism) > 0
    if do == "residual":
        return _cat(s.residual(Q), mixed)
    for _ in range(case["steps"]):
        Q = s.step(Q, dt, "ssp33" if flow == "channel" else "rk44")
    return _cat(Q, mixed)
