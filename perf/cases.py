"""Performance cases: the work that users of the solver have it do, through the public binding.

Four kinds of call, over the meshes of the tests and the benchmark and over drawn boxes:

* ``schur``     the interface operator S_hat x of a linearised handle (one Krylov product);
* ``residual``  the Newton residual F(u) - G of a nodal state;
* ``newton``    one Newton correction: Jacobian, factorisations, preconditioner, Krylov solve
                and interior recovery (``linearize`` then ``krylov_solve``);
* ``step``      one implicit time step from a given state (``set_state``, ``step``, ``get_state``);
* ``mlp``       forward and backward pass of the learned guess's network on host arrays.

States hold a depolarisation front at a seeded place with N(0, 1 mV) noise in v.  The reference
values (``exact``) come from a matrix-free FP64 discretisation in torch, written here from the
equations, with conjugate gradients in place of the domain decomposition.
"""
import math

import numpy as np
import torch

from paper_2101_02959_gb300 import binding

SIGMA_I = (3.0e-3, 3.1525e-4, 3.1525e-5)
SIGMA_E = (2.0e-3, 1.3514e-3, 6.757e-4)
IONIC = dict(G=1.2, eta1=4.4, eta2=0.012, vth=13.0, vp=100.0, chi_cm=1.0)
TAU = 0.05
AMP = 100.0
SHELL = ((2.0, 2.0, 5.0), (2.8, 2.8, 5.8))
# tolerances of accurate time steps with single-precision local solvers: Newton until the
# double-precision residual no longer falls, so that the state is the solution's
TIGHT = dict(snes_rtol=1e-12, snes_atol=1e-16, snes_stol=1e-12)


def _box(kind, name, n, s, h, **more):
    return dict(kind=kind, name=name, nx=n[0], ny=n[1], nz=n[2], sx=s[0], sy=s[1], sz=s[2], h=h, **more)


def listed():
    vep = dict(primal="VE", precision="fp64")
    mix = dict(primal="VE", precision="mixed")
    return [
        # the smallest call: one operator product on 8 subdomains of 125 nodes, all launch latency
        _box("schur", "schur_cube8", (8, 8, 8), (4, 4, 4), 0.05, **vep),
        # the operator product on 256 subdomains, the work of every Krylov iteration
        _box("schur", "schur_slab64", (64, 64, 32), (8, 8, 8), 0.025, **vep),
        # the residual that every Newton and line-search step evaluates, on the weak-scaling slab
        _box("residual", "residual_slab128", (128, 128, 32), (8, 8, 8), 0.025, **mix),
        # one Newton correction of the small cube with vertex constraints (PCG, BDDC)
        _box("newton", "newton_cube8", (8, 8, 8), (4, 4, 4), 0.05, primal="V", precision="fp64", method="bddc",
             krylov="pcg", scaling="deluxe"),
        # ragged blocks with the dual method under GMRES
        _box("newton", "newton_ragged", (10, 9, 7), (4, 4, 4), 0.05, method="fetidp", krylov="gmres",
             scaling="deluxe", **vep),
        # the medium slab, the default solver (double precision, BDDC, PCG)
        _box("newton", "newton_slab32", (32, 32, 16), (8, 8, 8), 0.05, method="bddc", krylov="pcg",
             scaling="deluxe", **vep),
        # large subdomains (the optimality sweep at H/h = 12), the largest factorisation in double precision
        _box("newton", "newton_opt12", (48, 48, 48), (12, 12, 12), 0.8 / 48, method="bddc", krylov="pcg",
             scaling="deluxe", **vep),
        # a whole default time step: double precision, the paper's tolerances, the dual method
        _box("step", "step_slab32_fp64", (32, 32, 16), (8, 8, 8), 0.05, method="fetidp", tc=0, lag=0, **vep),
        # the same slab with single-precision local solvers on the tensor cores, a Jacobian per iterate
        _box("step", "step_slab32_mixed", (32, 32, 16), (8, 8, 8), 0.05, method="bddc", tc=1, lag=0, **mix),
        # uneven subdomains: a masked ellipsoidal wall
        dict(kind="step", name="step_shell_mixed", nx=56, ny=56, nz=58, sx=6, sy=6, sz=6, h=0.1, shell=True,
             method="bddc", tc=1, lag=0, **mix),
        # the largest: 1.1 million unknowns on 1,024 subdomains, one Jacobian per step
        _box("step", "step_slab128_mixed", (128, 128, 32), (8, 8, 8), 0.025, method="bddc", tc=1, lag=1, **mix),
        # training pass of the initial-guess network of the 256-subdomain slab
        _box("mlp", "mlp_slab64", (64, 64, 32), (8, 8, 8), 0.025, **mix),
    ]


def _dense_work(n, s):
    """Sum over the subdomains of (local unknowns)^3, the size of a factorisation."""
    return math.prod(-(-n[d] // s[d]) for d in range(3)) * (2.0 * math.prod(s[d] + 1 for d in range(3))) ** 3


def draw(rng):
    kind = rng.choice(["schur", "residual", "newton", "newton", "step", "step", "mlp"])
    mixed = kind == "mlp" or (kind == "step" and rng.random() < 0.6)
    most = {"schur": 8e11, "residual": 3e12, "newton": 4e12, "step": 2.5e12 if mixed else 1.2e12, "mlp": 8e11}[kind]
    least = 1e5 if kind != "residual" else 1e6
    want = math.exp(rng.uniform(math.log(least), math.log(most)))
    s = [rng.randint(2, 12) for _ in range(3)]
    n = [2 * v - rng.randint(0, v - 1) for v in s]  # two blocks a direction, the last one ragged
    while _dense_work(n, s) > want and max(s) > 2:
        d = s.index(max(s))
        s[d] -= 1
        n[d] = 2 * s[d] - rng.randint(0, s[d] - 1)
    while _dense_work(n, s) < 0.7 * want and math.prod(v + 1 for v in n) < 5e5:
        d = rng.randrange(3)
        if n[d] < 128:
            n[d] += rng.randint(1, s[d])
    case = _box(kind, "", n, s, round(rng.uniform(0.02, 0.05), 4), primal=rng.choice(["VE", "VE", "VEF", "V"]),
                precision="mixed" if mixed else "fp64")
    del case["name"]
    if kind == "newton":
        case.update(method=rng.choice(["bddc", "fetidp"]), krylov=rng.choice(["pcg", "pcg", "gmres"]),
                    scaling=rng.choice(["deluxe", "deluxe", "rho"]))
    elif kind == "step":
        case.update(method=rng.choice(["bddc", "bddc", "fetidp"]), tc=rng.choice([0, 1, 2]) if mixed else 0,
                    lag=rng.choice([0, 1]))
    if mixed or kind == "step":
        case["primal"] = "VE" if case["primal"] == "V" else case["primal"]
    return case


# ---- what a user's program has in hand -------------------------------------------------


def _dims(c):
    return (c["nx"], c["ny"], c["nz"]), (c["sx"], c["sy"], c["sz"])


def _shell_mask(n, h):
    (ai, bi, ci), (ao, bo, co) = SHELL
    x = ((np.arange(n[0]) + 0.5) * h - ao)[None, None, :]
    y = ((np.arange(n[1]) + 0.5) * h - bo)[None, :, None]
    z = ((np.arange(n[2]) + 0.5) * h - co)[:, None, None]
    keep = (z <= 0) & ((x / ai) ** 2 + (y / bi) ** 2 + (z / ci) ** 2 >= 1.0) & \
           ((x / ao) ** 2 + (y / bo) ** 2 + (z / co) ** 2 <= 1.0)
    return np.ascontiguousarray(keep.astype(np.uint8))  # [z][y][x]: x fastest


def _workload(c):
    n, s = _dims(c)
    w = dict(n=n, s=s, l=tuple(c["h"] * v for v in n), primal=c["primal"])
    if c.get("shell"):
        w["mask"] = _shell_mask(n, c["h"]).ravel()
    return w


def _used_nodes(c):
    """Flat grid ids (x fastest) of the nodes of the kept elements, and the element mask."""
    n, _ = _dims(c)
    if not c.get("shell"):
        return torch.arange(math.prod(v + 1 for v in n), device="cuda"), None
    m = torch.from_numpy(_shell_mask(n, c["h"])).cuda().double()
    touched = torch.zeros(n[2] + 1, n[1] + 1, n[0] + 1, dtype=torch.float64, device="cuda")
    for a in range(8):
        touched[(a >> 2) & 1:n[2] + ((a >> 2) & 1), (a >> 1) & 1:n[1] + ((a >> 1) & 1), a & 1:n[0] + (a & 1)] += m
    return torch.nonzero(touched.reshape(-1)).reshape(-1), m


def _stimulus(c):
    """A box at the grid's corner (the apex of the shell), on for the first millisecond."""
    box = (2.45, 3.15, 2.45, 3.15, 0.0, 0.35) if c.get("shell") else (0.0, 0.1, 0.0, 0.1, 0.0, 0.1)
    return dict(amp=AMP, t_on=0.0, t_off=1.0, box=box)


def _coords(c):
    n, _ = _dims(c)
    g = _used_nodes(c)[0]
    return (torch.stack([g % (n[0] + 1), (g // (n[0] + 1)) % (n[1] + 1), g // ((n[0] + 1) * (n[1] + 1))]).double()
            * c["h"])


def _front(c, seed):
    """u_i, u_e, w of a depolarisation front moving away from the stimulated corner."""
    rng = np.random.default_rng([seed, 1])
    x = _coords(c)
    far = float(x.max())
    dist = (x if not c.get("shell") else x[2:]).square().sum(0).sqrt()
    at = far * rng.uniform(0.3, 0.7)
    back = torch.sigmoid((at - dist) / 0.06)
    noise = torch.from_numpy(rng.normal(0.0, 1.0, x.shape[1])).cuda()
    v = 95.0 * back + noise
    w = 0.08 * back * torch.clamp((at - dist) / far, min=0.0)
    ue = -0.3 * (v - v.mean())
    return ue + v, ue, w


def _normal(n, seed, k):
    return torch.from_numpy(np.random.default_rng([seed, k]).standard_normal(n)).cuda()


def _interface(c):
    """Grid ids of the interface nodes of a box (ascending)."""
    n, s = _dims(c)
    cut = [torch.tensor([0 < i < n[d] and i % s[d] == 0 for i in range(n[d] + 1)], device="cuda") for d in range(3)]
    m = cut[2][:, None, None] | cut[1][None, :, None] | cut[0][None, None, :]
    return torch.nonzero(m.reshape(-1)).reshape(-1)


def prepare(case, seed):
    c = case
    stream = torch.cuda.Stream()
    opt = dict(precision=c["precision"], primal=c["primal"], stream=stream.cuda_stream)
    if c["kind"] == "newton":
        # solved to double precision's accuracy, as the solver's own tests do
        opt.update(method=c["method"], krylov=c["krylov"], scaling=c["scaling"], ksp_rtol=1e-12, ksp_atol=0.0)
    elif c["kind"] == "step":
        opt.update(method=c["method"], lag_jacobian=c["lag"], use_tensor_cores=c["tc"],
                   **(TIGHT if c["precision"] == "mixed" else {}))
    elif c["kind"] == "mlp":
        opt.update(learned_guess=1)
    solver = binding.Solver(_workload(c), SIGMA_I, SIGMA_E, IONIC, TAU, **opt)
    st = dict(case=c, solver=solver, stream=stream, stim=_stimulus(c))
    if c["kind"] == "mlp":
        sz = solver.mlp_sizes()
        st.update(zip(("X", "T", "mask"), _mlp_batch(sz, seed)))
        solver.mlp_params(_mlp_weights(sz, seed))
        return st
    st["u"] = _front(c, seed)
    if c["kind"] == "newton":
        st["f"] = _rhs(c, seed)
    elif c["kind"] == "schur":
        st["x"] = _normal(solver.sizes["n_iface"], seed, 2)
    torch.cuda.synchronize()
    if c["kind"] == "schur":
        solver.linearize(*st["u"])
    return st


def run(state):
    c, s = state["case"], state["solver"]
    if c["kind"] == "mlp":
        loss, grad = s.mlp_loss_grad(state["X"], state["T"], state["mask"])
        return {"loss": loss, "grad": grad}
    with torch.cuda.stream(state["stream"]):
        if c["kind"] == "schur":
            return s.schur_apply(state["x"])
        ui, ue, w = state["u"]
        if c["kind"] == "residual":
            return s.residual(state["stim"], TAU, ui, ue, w, ui, ue)
        if c["kind"] == "newton":
            s.linearize(ui, ue, w)
            return s.krylov_solve(state["f"])[0]
        s.set_state(ui, ue, w, 0.0)
        s.step(state["stim"])
        ui1, ue1, w1, _ = s.get_state(like=ui)
        return {"ui": ui1, "ue": ue1, "w": w1}


def _mlp_batch(sz, seed):
    rng = np.random.default_rng([seed, 3])
    X = rng.normal(0.0, 0.3, (sz["batch"], sz["n_in"])).astype(np.float32)
    T = rng.normal(0.0, 0.05, (sz["batch"], sz["n_out"])).astype(np.float32)
    return X, T, np.ones_like(T)


def _mlp_weights(sz, seed):
    rng = np.random.default_rng([seed, 4])
    h, parts = sz["n_hidden"], []
    for rows, cols in ((h, sz["n_in"]), (h, h), (sz["n_out"], h)):
        parts += [rng.uniform(-1, 1, rows * cols) * math.sqrt(6.0 / cols), rng.uniform(-0.05, 0.05, rows)]
    return np.concatenate(parts).astype(np.float32)


def work(case):
    """Bytes: nodal or interface vectors in and out, the stored operator where the call is a
    product with it.  Flops: the banded local factorisations and solves of the method, or the
    products themselves."""
    c = case
    n, s = _dims(c)
    N = math.prod(v + 1 for v in n)
    nsub = math.prod(-(-n[d] // s[d]) for d in range(3))
    if c.get("shell"):
        m = _shell_mask(n, c["h"])
        N, nsub = N * float(m.mean()), nsub * float(m.mean())
    nI = 2.0 * math.prod(v - 1 for v in s)
    nG = 2.0 * math.prod(v + 1 for v in s) - nI
    el = 4 if c["precision"] == "mixed" else 8
    if c["kind"] == "mlp":
        k = nG / 2
        w = 256.0 * (6 * k + 256 + 2 * k)
        return {"bytes": 4.0 * (nsub * (6 + 2 + 2) * k + 2 * w), "flops": 6.0 * nsub * w}
    if c["kind"] == "schur":
        return {"bytes": nsub * nG * (nG + 1) / 2 * el, "flops": 2.0 * nsub * nG * nG}
    if c["kind"] == "residual":
        return {"bytes": N * (54 * 8 + 8 + 7 * 8), "flops": N * (108.0 + 30.0)}
    band = 2.0 * (min(s) + 1) * (sorted(s)[1] + 1)
    jac = nsub * (nI * band ** 2 + (nI + nG) * band ** 2 + 2.0 * nI * band * nG)
    solve = 15.0 * nsub * 8.0 * (nI + nG) * band
    k = 1.0 if c["kind"] == "newton" else (2.0 if c["precision"] == "fp64" else 6.0)
    jacs = 1.0 if c.get("lag") else k
    return {"bytes": N * 8.0 * 10 + jacs * nsub * (nI + nG) * band * el, "flops": jacs * jac + k * solve}


# ---- reference values: the equations in FP64, matrix-free -------------------------------


class _Fem:
    """Q1 stiffness and lumped mass of a box grid (elements outside the mask dropped)."""

    def __init__(self, c):
        self.n, _ = _dims(c)
        self.nodes, self.mask = _used_nodes(c)
        self.shape = (self.n[2] + 1, self.n[1] + 1, self.n[0] + 1)
        h = c["h"]
        z = (torch.arange(self.n[2], dtype=torch.float64) + 0.5) / self.n[2]
        ang = torch.deg2rad(-60.0 + 120.0 * (1.0 - z))
        zero = torch.zeros_like(ang)
        al = torch.stack([ang.cos(), ang.sin(), zero], 1)
        at = torch.stack([-ang.sin(), ang.cos(), zero], 1)
        an = torch.tensor([0.0, 0.0, 1.0], dtype=torch.float64).expand(self.n[2], 3)
        # gradients of the eight shape functions at the 2 x 2 x 2 Gauss points
        g = [0.5 - 0.5 / math.sqrt(3.0), 0.5 + 0.5 / math.sqrt(3.0)]
        B = torch.zeros(8, 8, 3, dtype=torch.float64)
        for q in range(8):
            xi = [g[(q >> d) & 1] for d in range(3)]
            for a in range(8):
                l = [xi[d] if (a >> d) & 1 else 1.0 - xi[d] for d in range(3)]
                sg = [1.0 if (a >> d) & 1 else -1.0 for d in range(3)]
                for d in range(3):
                    B[q, a, d] = sg[d] / h * math.prod(l[e] for e in range(3) if e != d)
        self.K = []
        for sig in (SIGMA_I, SIGMA_E):
            D = sum(sk * v[:, :, None] * v[:, None, :] for sk, v in zip(sig, (al, at, an)))
            self.K.append((torch.einsum("qap,zpr,qbr->zab", B, D, B) * h ** 3 / 8.0).cuda())
        one = torch.ones(self.n[2], self.n[1], self.n[0], dtype=torch.float64, device="cuda")
        one = one if self.mask is None else one * self.mask
        self.M = self._gather([one * h ** 3 / 8.0] * 8)
        self.diag = [self._gather([one * k[:, a, a][:, None, None] for a in range(8)]) for k in self.K]

    def _corner(self, a):
        x, y, z = a & 1, (a >> 1) & 1, (a >> 2) & 1
        return (slice(z, self.n[2] + z), slice(y, self.n[1] + y), slice(x, self.n[0] + x))

    def _gather(self, per_corner):
        out = torch.zeros(self.shape, dtype=torch.float64, device="cuda")
        for a in range(8):
            out[self._corner(a)] += per_corner[a]
        return out.reshape(-1)[self.nodes]

    def stiff(self, f, u):
        """A_f u (f = 0 intra-, 1 extracellular) for a vector over the used nodes."""
        grid = torch.zeros(math.prod(self.shape), dtype=torch.float64, device="cuda")
        grid[self.nodes] = u
        grid = grid.reshape(self.shape)
        U = torch.stack([grid[self._corner(a)].reshape(self.n[2], -1) for a in range(8)], 2)
        Y = torch.bmm(U, self.K[f])  # symmetric element matrices
        Y = Y.reshape(self.n[2], self.n[1], self.n[0], 8)
        if self.mask is not None:
            Y = Y * self.mask[..., None]
        return self._gather([Y[..., a] for a in range(8)])


def _iion(v, w):
    p = IONIC
    return p["G"] * v * (1 - v / p["vth"]) * (1 - v / p["vp"]) + p["eta1"] * v * w


def _diion(v, w):
    a, b = 1 / IONIC["vth"], 1 / IONIC["vp"]
    return IONIC["G"] * (1 - 2 * (a + b) * v + 3 * a * b * v * v) + IONIC["eta1"] * w


def _residual(c, fem, ui, ue, w, uin, uen):
    """F(u) - G at the end of the first step (the stimulus is on)."""
    x, b = _coords(c), _stimulus(c)["box"]
    on = torch.ones(x.shape[1], dtype=torch.bool, device="cuda")
    for d in range(3):
        on &= (x[d] >= b[2 * d] - 1e-9) & (x[d] <= b[2 * d + 1] + 1e-9)
    v = ui - ue
    q = IONIC["chi_cm"] * fem.M * (v - (uin - uen)) + TAU * fem.M * (_iion(v, w) - AMP * on)
    return torch.stack([q + TAU * fem.stiff(0, ui), TAU * fem.stiff(1, ue) - q])


class _Jacobian:
    def __init__(self, fem, ui, ue, w):
        self.fem = fem
        self.kc = fem.M * (IONIC["chi_cm"] + TAU * _diion(ui - ue, w))
        a, b = self.kc + TAU * fem.diag[0], self.kc + TAU * fem.diag[1]
        det = a * b - self.kc ** 2
        self.inv = (b / det, self.kc / det, a / det)  # of the nodal 2 x 2 blocks

    def __call__(self, s):
        d = self.kc * (s[0] - s[1])
        return torch.stack([TAU * self.fem.stiff(0, s[0]) + d, TAU * self.fem.stiff(1, s[1]) - d])

    def solve(self, f, free=None, rtol=1e-14, most=8000):
        """Conjugate gradients on the free nodes (all: the constant mode projected out of f)."""
        keep = torch.ones_like(f) if free is None else free.double().expand_as(f)
        r = f * keep
        if free is None:
            r = r - r.mean()
        x = torch.zeros_like(f)
        a, b, d = self.inv
        z = torch.stack([a * r[0] + b * r[1], b * r[0] + d * r[1]])
        p, rz = z.clone(), (r * z).sum()
        first = float(rz)
        for it in range(most):
            q = self(p) * keep
            al = rz / (p * q).sum()
            x += al * p
            r -= al * q
            z = torch.stack([a * r[0] + b * r[1], b * r[0] + d * r[1]])
            new = (r * z).sum()
            p = z + (new / rz) * p
            rz = new
            if it % 25 == 24 and float(rz) <= rtol ** 2 * first:
                break
        return x


def _rhs(c, seed):
    """Right-hand side of a Newton correction: minus the residual of the seeded state after a
    step from a state one increment behind it."""
    fem = _Fem(c)
    ui, ue, w = _front(c, seed)
    dv = 0.5 * _normal(ui.numel(), seed, 5) + 2.0 * torch.sigmoid((ui - ue - 50.0) / 20.0)
    r = _residual(c, fem, ui, ue, w, ui - 0.7 * dv, ue + 0.3 * dv)
    r = r - r.mean()
    return (-r).reshape(-1).contiguous()


def exact(case, seed):
    c = case
    if c["kind"] == "mlp":
        return _exact_mlp(c, seed)
    fem = _Fem(c)
    ui, ue, w = _front(c, seed)
    n, s = _dims(c)
    gauge = s[0] + (n[0] + 1) * (s[1] + (n[1] + 1) * s[2])  # the lowest vertex of a box
    if c["kind"] == "residual":
        return _residual(c, fem, ui, ue, w, ui, ue).reshape(-1)
    if c["kind"] == "newton":
        d = _Jacobian(fem, ui, ue, w).solve(_rhs(c, seed).reshape(2, -1))
        return (d - d[1, gauge]).reshape(-1)
    if c["kind"] == "schur":
        J, g = _Jacobian(fem, ui, ue, w), _interface(c)
        x = torch.zeros(2, ui.numel(), dtype=torch.float64, device="cuda")
        x[:, g] = _normal(2 * g.numel(), seed, 2).reshape(-1, 2).T
        inner = torch.ones(ui.numel(), dtype=torch.bool, device="cuda")
        inner[g] = False
        y = J(x + J.solve(-J(x), free=inner))
        y[1, gauge] = 0.0
        return y[:, g].T.reshape(-1).contiguous()
    te = TAU * IONIC["eta2"]
    wn = (w + te * (ui - ue) / IONIC["vp"]) / (1 + te)
    a, b = ui.clone(), ue.clone()
    r = _residual(c, fem, a, b, wn, ui, ue)
    first = float(r.norm())
    for _ in range(12):
        d = _Jacobian(fem, a, b, wn).solve(-r, rtol=1e-11)
        a, b = a + d[0], b + d[1]
        r = _residual(c, fem, a, b, wn, ui, ue)
        if float(r.norm()) < 1e-13 * first or float(d.norm()) < 1e-13 * float(a.norm() + b.norm()):
            break
    shift = (fem.M * b).sum() / fem.M.sum()
    return {"ui": a - shift, "ue": b - shift, "w": wn}


def _exact_mlp(c, seed):
    """Loss and gradient of the network in FP64 (its bfloat16 roundings left out)."""
    n, s = _dims(c)
    most = max(2 * (math.prod(min(s[d], n[d]) + 1 for d in range(3)) - _inner(n, s)), 2)
    nsub = math.prod(-(-n[d] // s[d]) for d in range(3))
    sz = dict(batch=nsub, n_hidden=256, n_in=3 * most, n_out=most)
    X, T, _ = (torch.from_numpy(v).cuda().double() for v in _mlp_batch(sz, seed))
    flat = torch.from_numpy(_mlp_weights(sz, seed)).cuda().double().requires_grad_(True)
    h, at, layers = 256, 0, []
    for rows, cols in ((h, sz["n_in"]), (h, h), (sz["n_out"], h)):
        W = flat[at:at + rows * cols].reshape(rows, cols)
        layers.append((W, flat[at + rows * cols:at + rows * cols + rows]))
        at += rows * cols + rows
    Y = X
    for k, (W, bias) in enumerate(layers):
        Y = Y @ W.T + bias
        Y = torch.relu(Y) if k < 2 else Y
    loss = (Y - T).square().mean()
    loss.backward()
    return {"loss": loss.detach(), "grad": flat.grad}


def _inner(n, s):
    """Fewest nodes of a subdomain that no other subdomain shares (over the blocks that hold
    the most interface nodes, the middle ones where a direction has three or more)."""
    best = None
    blocks = [-(-n[d] // s[d]) for d in range(3)]
    for i in range(min(blocks[0], 3)):
        for j in range(min(blocks[1], 3)):
            for k in range(min(blocks[2], 3)):
                own, whole = 1, 1
                for d, b in enumerate((i, j, k)):
                    b = blocks[d] - 1 if b == min(blocks[d], 3) - 1 else b
                    lo, hi = b * s[d], min((b + 1) * s[d], n[d])
                    own *= hi - lo + 1 - (lo > 0) - (hi < n[d])
                    whole *= hi - lo + 1
                if best is None or whole - own > best[0]:
                    best = (whole - own, whole)
    return math.prod(min(s[d], n[d]) + 1 for d in range(3)) - best[0]
