"""Profiled kernel classes add up: the times of the factorisation's launches are those of launches one
after another, so their sum fits into the region that holds them."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tc", [("fp64", 0), ("mixed", 1), ("mixed", 2)])
def test_factorisation_classes_fit_into_the_jacobian(precision, tc):
    """2,310 coarse unknowns: the coarse matrix's panels run beside its updates, the deluxe classes beside
    the local factorisation, unless the classes are timed.  Either way the Jacobian is the same."""
    from paper_2101_02959_gb300 import binding, build
    build.build()
    w = synth.workload("coarse2k")
    s = binding.Solver(w, synth.SIGMA_I, synth.SIGMA_E, synth.IONIC, synth.TAU, precision=precision, use_tensor_cores=tc)
    ui, ue, wv = synth.initial_state(s.N, 5)
    r = synth.random_vector(s.sizes["n_iface"], 6)
    s.linearize(ui, ue, wv)
    ref = s.bddc_apply(r)
    s.profile(1)
    s.linearize(ui, ue, wv)
    classes = s.profile_read("panel")["ms"] + s.profile_read("rankk")["ms"]
    region = s.profile_read("linearize")["ms"]
    s.profile(0)
    assert 0.0 < classes <= region
    assert np.array_equal(s.bddc_apply(r), ref)
    s.close()
