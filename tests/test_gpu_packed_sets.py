"""Packed copies of the FP64 operators: only the methods that read a set pack it."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def test_bddc_handles_pack_no_fetidp_operator():
    """A BDDC handle's Jacobian packs S_Gamma and S_DeltaDelta^-1, a FETI-DP handle's S_DeltaDelta too
    (one launch more); the FETI-DP preconditioner is the same on both (bar: the operators', 1e-9)."""
    from paper_2101_02959_gb300 import binding, build
    build.build()
    w = synth.workload("cube8ve")
    launches, out = {}, {}
    for method in ("bddc", "fetidp"):
        s = binding.Solver(w, synth.SIGMA_I, synth.SIGMA_E, synth.IONIC, synth.TAU, method=method)
        ui, ue, wv = synth.initial_state(s.N, 5)
        s.linearize(ui, ue, wv)
        before = binding.launch_count()
        s.linearize(ui, ue, wv)
        launches[method] = binding.launch_count() - before
        out[method] = s.fetidp_apply(synth.random_vector(s.sizes["n_lambda"], 7))
        s.close()
    assert launches["fetidp"] == launches["bddc"] + 1
    assert np.linalg.norm(out["bddc"] - out["fetidp"]) < 1e-9 * np.linalg.norm(out["fetidp"])
