"""FP32 symmetric operator products at the edges of their 32 x 32 tiles and of the split over CTAs.

Bar 2e-5, the mixed operators' bar of the parity tests: FP32 roundoff (6e-8) times the condition
of the interior blocks (below 1e3 here) with a factor of a few for the sums.
"""
import numpy as np
import pytest

import synth
from oracle import ionic
from oracle.bidomain import Problem
from oracle.dd import DDSolver

pytestmark = pytest.mark.gpu


# interface unknowns per subdomain on both sides of one, two and several tiles; 8 subdomains (split
# over many CTAs) and 256 (a few CTAs a matrix)
@pytest.mark.parametrize("subs,s", [((2, 2, 2), (1, 1, 1)), ((2, 2, 2), (2, 2, 1)), ((2, 2, 2), (2, 2, 2)),
                                    ((2, 2, 2), (3, 2, 2)), ((2, 2, 2), (5, 5, 5)), ((2, 2, 2), (9, 7, 1)),
                                    ((2, 1, 1), (4, 4, 4)), ((8, 8, 4), (2, 2, 2)), ((2, 2, 2), (7, 7, 7))])
def test_mixed_schur_operator_at_tile_edges(subs, s):
    from paper_2101_02959_gb300 import binding, build
    build.build()
    n = tuple(a * b for a, b in zip(subs, s))
    w = dict(n=n, l=tuple(0.1 * v for v in s), s=s, primal="V", name="edges")
    prob = Problem(w, synth.SIGMA_I, synth.SIGMA_E, synth.IONIC, synth.TAU, synth.stimulus(w))
    ui, ue, wv = synth.initial_state(prob.N, 5)
    wn = ionic.gating_step(ui - ue, wv, prob.tau, prob.p)
    dd = DDSolver(prob)
    dd.setup(prob.p["chi_cm"] + prob.tau * ionic.di_ion_dv(ui - ue, wn, prob.p))
    x = synth.random_vector(prob.dofs.n_iface, 6)
    x[dd.g_iface] = 0.0
    ref = dd.schur_apply(x)
    sol = binding.Solver(w, synth.SIGMA_I, synth.SIGMA_E, synth.IONIC, synth.TAU, precision="mixed")
    sol.linearize(ui, ue, wn)
    for _ in range(2):  # the counters of the split are back at their start
        y = sol.schur_apply(x)
        assert np.linalg.norm(y - ref) < 2e-5 * np.linalg.norm(ref)
        assert np.max(np.abs(y - ref)) < 2e-5 * np.max(np.abs(ref))
    sol.close()
