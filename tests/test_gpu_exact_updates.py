"""FP64 factorisation on the tensor cores (exact digit products): the Schur operator against the
oracle at block sizes on both sides of the panel (64), tile (64 x 128) and group (128) edges.

Bar 1e-11: the operator's rounding error is the unit roundoff (1.1e-16) times cond(K_II)
(below 1e3 at these sizes) times a growth of order ten through the panels, about 1e-12.
"""
import numpy as np
import pytest

import synth
from oracle import ionic
from oracle.bidomain import Problem
from oracle.dd import DDSolver

pytestmark = pytest.mark.gpu

# interior unknowns per subdomain: 2, 62, 64, 66 (a panel), 126 .. 130 (a tile, a group), 250, 686
BLOCKS = [(1, 1, 1), (31, 1, 1), (4, 4, 2), (11, 3, 1), (9, 7, 1), (4, 4, 4), (13, 5, 1), (5, 5, 5), (7, 7, 7)]


@pytest.mark.parametrize("s", BLOCKS)
def test_schur_operator_at_tile_edges(s):
    from paper_2101_02959_gb300 import binding, build
    build.build()
    w = dict(n=tuple(2 * v for v in s), l=tuple(0.1 * v for v in s), s=s, primal="V", name="edges")
    prob = Problem(w, synth.SIGMA_I, synth.SIGMA_E, synth.IONIC, synth.TAU, synth.stimulus(w))
    ui, ue, wv = synth.initial_state(prob.N, 5)
    wn = ionic.gating_step(ui - ue, wv, prob.tau, prob.p)
    dd = DDSolver(prob)
    dd.setup(prob.p["chi_cm"] + prob.tau * ionic.di_ion_dv(ui - ue, wn, prob.p))
    x = synth.random_vector(prob.dofs.n_iface, 6)
    x[dd.g_iface] = 0.0
    ref = dd.schur_apply(x)
    sol = binding.Solver(w, synth.SIGMA_I, synth.SIGMA_E, synth.IONIC, synth.TAU, precision="fp64")
    for _ in range(2):  # a second Jacobian reuses the workspace
        sol.linearize(ui, ue, wn)
        y = sol.schur_apply(x)
        assert np.linalg.norm(y - ref) < 1e-11 * np.linalg.norm(ref)
        assert np.max(np.abs(y - ref)) < 1e-11 * np.max(np.abs(ref))
    sol.close()


# largest face blocks of order 46, 48 (the first product on the tensor cores), 50, 64, 98, 126
@pytest.mark.parametrize("s", [(1, 23, 2), (4, 6, 2), (5, 5, 5), (8, 4, 1), (7, 7, 7), (9, 7, 1)])
def test_deluxe_products_at_tile_edges(s):
    """M^-1 r in FP64 against the oracle: the deluxe operators are products of order n on the tensor
    cores from n = 48 on.  Bar 1e-9, the operators' bar of the parity tests (the coarse solve and the
    local inverses amplify rounding by their condition numbers)."""
    from paper_2101_02959_gb300 import binding, build
    build.build()
    w = dict(n=tuple(2 * v for v in s), l=tuple(0.1 * v for v in s), s=s, primal="V", name="edges")
    prob = Problem(w, synth.SIGMA_I, synth.SIGMA_E, synth.IONIC, synth.TAU, synth.stimulus(w))
    ui, ue, wv = synth.initial_state(prob.N, 5)
    wn = ionic.gating_step(ui - ue, wv, prob.tau, prob.p)
    dd = DDSolver(prob)
    dd.setup(prob.p["chi_cm"] + prob.tau * ionic.di_ion_dv(ui - ue, wn, prob.p))
    r = synth.random_vector(prob.dofs.n_iface, 6)
    r[dd.g_iface] = 0.0
    ref = dd.bddc_apply(r)
    sol = binding.Solver(w, synth.SIGMA_I, synth.SIGMA_E, synth.IONIC, synth.TAU, precision="fp64")
    sol.linearize(ui, ue, wn)
    z = sol.bddc_apply(r)
    sol.close()
    assert np.linalg.norm(z - ref) < 1e-9 * np.linalg.norm(ref)
    assert np.max(np.abs(z - ref)) < 1e-9 * np.max(np.abs(ref))
