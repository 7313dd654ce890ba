"""Preconditioner of two subdomains that share one small face: a single deluxe class whose panel is
narrower than 32 columns, so that the class workspace holds one matrix of less than a full panel.

Bars: FP64 1e-9, the operators' bar of the parity tests.  FP32: the forward error of the local solves,
16 u cond(K_IDelta,IDelta) with u = 2^-24 and a growth of order ten through panels and class products.
"""
import numpy as np
import pytest

import synth
from oracle import ionic
from oracle.bidomain import Problem
from oracle.dd import DDSolver

pytestmark = pytest.mark.gpu


# class orders 6, 16, 22, 30 (one digit block of 32 columns) and 38, 48
@pytest.mark.parametrize("s", [(2, 1, 1), (2, 2, 2), (3, 3, 2), (2, 3, 3), (2, 4, 3), (4, 4, 4)])
@pytest.mark.parametrize("precision,tc", [("fp64", 0), ("mixed", 0), ("mixed", 1), ("mixed", 2)])
def test_one_small_class(s, precision, tc):
    from paper_2101_02959_gb300 import binding, build
    build.build()
    w = dict(n=(2 * s[0], s[1], s[2]), l=(0.2 * s[0], 0.1 * s[1], 0.1 * s[2]), s=s, primal="V", name="pair")
    prob = Problem(w, synth.SIGMA_I, synth.SIGMA_E, synth.IONIC, synth.TAU, synth.stimulus(w))
    ui, ue, wv = synth.initial_state(prob.N, 5)
    wn = ionic.gating_step(ui - ue, wv, prob.tau, prob.p)
    dd = DDSolver(prob, keep_fetidp=True)
    dd.setup(prob.p["chi_cm"] + prob.tau * ionic.di_ion_dv(ui - ue, wn, prob.p))
    r = synth.random_vector(prob.dofs.n_iface, 6)
    r[dd.g_iface] = 0.0
    ref = dd.bddc_apply(r)
    bar = 1e-9
    if precision == "mixed":
        n = [L["nI"] + len(L["dual"]) for L in dd.loc]
        bar = 16.0 * 2.0 ** -24 * max(np.linalg.cond(L["Kb"][:k, :k]) for L, k in zip(dd.loc, n))
    sol = binding.Solver(w, synth.SIGMA_I, synth.SIGMA_E, synth.IONIC, synth.TAU, precision=precision,
                         use_tensor_cores=tc)
    for _ in range(2):  # a second Jacobian finds the workspace of the first
        sol.linearize(ui, ue, wn)
        z = sol.bddc_apply(r)
        assert np.linalg.norm(z - ref) < bar * np.linalg.norm(ref)
        assert np.max(np.abs(z - ref)) < bar * np.max(np.abs(ref))
    sol.close()
