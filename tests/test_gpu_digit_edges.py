"""FP32 digit products at the edges of their panels (64), tiles (128 x 64), digit blocks (32) and groups
(64 columns), in both tensor-core arithmetics; and the Krylov row loops of large interfaces.
"""
import numpy as np
import pytest

import synth
from oracle import ionic
from oracle.bidomain import Problem
from oracle.dd import DDSolver

pytestmark = pytest.mark.gpu


def _problem(s, primal):
    w = dict(n=tuple(2 * v for v in s), l=tuple(0.1 * v for v in s), s=s, primal=primal, name="edges")
    prob = Problem(w, synth.SIGMA_I, synth.SIGMA_E, synth.IONIC, synth.TAU, synth.stimulus(w))
    ui, ue, wv = synth.initial_state(prob.N, 5)
    wn = ionic.gating_step(ui - ue, wv, prob.tau, prob.p)
    dd = DDSolver(prob)
    dd.setup(prob.p["chi_cm"] + prob.tau * ionic.di_ion_dv(ui - ue, wn, prob.p))
    x = synth.random_vector(prob.dofs.n_iface, 6)
    x[dd.g_iface] = 0.0
    return w, dd, (ui, ue, wn), x


def _solver(w, **opt):
    from paper_2101_02959_gb300 import binding, build
    build.build()
    return binding.Solver(w, synth.SIGMA_I, synth.SIGMA_E, synth.IONIC, synth.TAU, **opt)


# interior unknowns per subdomain: 2, 62, 64, 66, 126 .. 130, 250, 686
@pytest.mark.parametrize("s", [(1, 1, 1), (31, 1, 1), (4, 4, 2), (11, 3, 1), (9, 7, 1), (4, 4, 4), (13, 5, 1),
                               (5, 5, 5), (7, 7, 7)])
@pytest.mark.parametrize("tc", [1, 2])
def test_schur_operator(s, tc):
    """Bar 2e-5, the mixed operators': FP32 roundoff (6e-8) times the condition of the interior blocks
    (48 to 1,430 here), of which a Schur complement of backward-stable updates shows a part."""
    w, dd, state, x = _problem(s, "V")
    ref = dd.schur_apply(x)
    sol = _solver(w, precision="mixed", use_tensor_cores=tc)
    for _ in range(2):  # a second Jacobian finds the first one's workspace
        sol.linearize(*state)
        y = sol.schur_apply(x)
        assert np.linalg.norm(y - ref) < 2e-5 * np.linalg.norm(ref)
        assert np.max(np.abs(y - ref)) < 2e-5 * np.max(np.abs(ref))
    sol.close()


# largest class orders on both sides of 48 (the first product on the tensor cores), 64 and 128
@pytest.mark.parametrize("s", [(4, 4, 4), (4, 6, 2), (5, 5, 5), (8, 4, 1), (7, 7, 7), (9, 7, 1), (13, 5, 1)])
@pytest.mark.parametrize("tc", [1, 2])
def test_deluxe_preconditioner(s, tc):
    """Bar 16 u cond(K_IDelta,IDelta), u = 2^-24 (2e-3 to 1.5e-2 here): the forward error of the local
    solves, with a growth of order ten through panels and class products."""
    w, dd, state, r = _problem(s, "VE")
    ref = dd.bddc_apply(r)
    n = [L["nI"] + len(L["dual"]) for L in dd.loc]
    bar = 16.0 * 2.0 ** -24 * max(np.linalg.cond(L["Kb"][:k, :k]) for L, k in zip(dd.loc, n))
    sol = _solver(w, precision="mixed", use_tensor_cores=tc)
    sol.linearize(*state)
    z = sol.bddc_apply(r)
    sol.close()
    assert np.linalg.norm(z - ref) < bar * np.linalg.norm(ref)
    assert np.max(np.abs(z - ref)) < bar * np.max(np.abs(ref))


# 9.8e4 interface unknowns (512 threads a block) and 3.2e5 (1,024)
@pytest.mark.parametrize("n", [(64, 64, 40), (128, 128, 32)])
def test_large_interfaces_under_both_krylov_methods(n):
    """PCG runs the row loops fused with its dots, GMRES the plain ones: the interface parts of the two
    solutions, through the operator.  Both stop at 1e-10 of the preconditioned right-hand side; with a
    condition number below 4 and 25 iterations the difference stays below 1e-10 x 4 x 25 = 1e-8 in the
    operator's norm, 1e-6 with the FP32 rounding of the condensed right-hand side's recovery (6e-8)."""
    w = dict(n=n, l=tuple(0.025 * v for v in n), s=(8, 8, 8), primal="VE", name="large")
    out = []
    for krylov in ("pcg", "gmres"):
        s = _solver(w, precision="mixed", use_tensor_cores=1, krylov=krylov, ksp_rtol=1e-10, ksp_atol=0.0)
        ui, ue, wv = synth.initial_state(s.N, 5)
        s.linearize(ui, ue, wv)
        f = -s.residual(None, synth.TAU, ui, ue, wv, ui - 1.0, ue)
        sol, st = s.krylov_solve(f)
        assert st["cond"] < 4.0
        nodes = s.index_set("IFACE_NODES")
        u = np.empty(2 * len(nodes))
        u[0::2], u[1::2] = sol[:s.N][nodes], sol[s.N:][nodes]
        out.append((s.schur_apply(u), st["its"]))
        s.close()
    (a, ka), (b, kb) = out
    assert len(a) > 77824 and abs(ka - kb) <= 3
    assert np.linalg.norm(a - b) < 1e-6 * np.linalg.norm(a)
