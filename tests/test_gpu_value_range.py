"""Operators at the ends of the number range: scaling the data by a power of two scales the result by
one and changes nothing else, as long as the numbers stay normal.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _solver(w, scale=1.0, **opt):
    """The cube's problem with every entry of its matrices times `scale`."""
    from paper_2101_02959_gb300 import binding, build
    build.build()
    ionic = dict(synth.IONIC, **{k: synth.IONIC[k] * scale for k in ("G", "eta1", "chi_cm")})
    return binding.Solver(w, tuple(v * scale for v in synth.SIGMA_I), tuple(v * scale for v in synth.SIGMA_E), ionic,
                          synth.TAU, **opt)


def test_operator_of_small_and_large_vectors():
    """FP64: the products' fixed-point segments keep all their bits down to the smallest vectors whose
    result is normal (entries of S_hat are 1e-8 .. 1e-3 here).  Bar 1e-13: 32 x 434 terms of 2^-53 a row
    sum, and nothing that depends on the scale; the first results that round to subnormals lie below
    2^-990."""
    w = synth.workload("cube8ve")
    s = _solver(w, precision="fp64")
    ui, ue, wv = synth.initial_state(s.N, 5)
    s.linearize(ui, ue, wv)
    x = synth.random_vector(s.sizes["n_iface"], 6)
    ref = s.schur_apply(x)
    for k in (-970, -950, -930, -900, -500, 500, 900, 1000):
        y = np.ldexp(s.schur_apply(np.ldexp(x, k)), -k)
        assert np.linalg.norm(y - ref) < 1e-13 * np.linalg.norm(ref), k
    assert not s.schur_apply(np.zeros_like(x)).any()
    s.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_infinite_and_nan_entries(precision, bad):
    """One entry that is no finite number: the rows that one subdomain alone couples to it follow the
    sign of their entry of S_hat, rows of subdomains that do not hold it stay as they are."""
    from conftest import oracle_problem
    prob = oracle_problem("cube8ve")
    part, dofs = prob.part, prob.dofs
    s = _solver(synth.workload("cube8ve"), precision=precision)
    ui, ue, wv = synth.initial_state(s.N, 5)
    s.linearize(ui, ue, wv)
    face = next(c for c in range(part.n_cls) if len(part.cls_subs[c]) == 2)
    g = 2 * dofs.gnode_to_iface[part.cls_nodes[face][0]]
    e = np.zeros(s.sizes["n_iface"])
    e[g] = 1.0
    col = s.schur_apply(e)
    x = synth.random_vector(e.size, 6)
    x[g] = 0.0
    rest = s.schur_apply(x)
    x[g] = bad
    y = s.schur_apply(x)
    gauge = 2 * dofs.gnode_to_iface[part.gauge_node] + 1
    seen = 0
    for c in range(part.n_cls):
        shared = len(set(part.cls_subs[c]) & set(part.cls_subs[face]))
        rows = np.concatenate([[2 * dofs.gnode_to_iface[n], 2 * dofs.gnode_to_iface[n] + 1] for n in part.cls_nodes[c]])
        rows = rows[rows != gauge]
        if shared == 0:
            assert np.array_equal(y[rows], rest[rows])
        elif shared == 1:
            seen += len(rows)
            assert (col[rows] != 0.0).all()
            assert np.array_equal(y[rows], col[rows] * bad, equal_nan=True)
    assert seen > 100
    s.close()


@pytest.mark.parametrize("precision,tc", [("fp64", 0), ("mixed", 0), ("mixed", 1), ("mixed", 2)])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_state_that_is_no_finite_number_is_refused(precision, tc, bad):
    """A Jacobian at a state with an infinity or a NaN, at the one interior vertex (whose rows only the
    coarse matrix factorises) and inside a subdomain."""
    from paper_2101_02959_gb300 import binding
    s = _solver(synth.workload("cube8ve"), precision=precision, use_tensor_cores=tc)
    ui, ue, wv = synth.initial_state(s.N, 5)
    for node in (s.N // 2, 2 * 81 + 2 * 9 + 2):
        u = ui.copy()
        u[node] = bad
        with pytest.raises(binding.BidomainError) as err:
            s.linearize(u, ue, wv)
        assert err.value.code == -2  # BD_ERR_NOT_SPD
    s.linearize(ui, ue, wv)  # the handle goes on
    s.close()


@pytest.mark.parametrize("tc", [0, 1, 2])
def test_mixed_operators_of_small_and_large_matrices(tc):
    """All matrices times a power of two (entries of K are 2^-45 .. 2^-17 before).  Bars: the operator
    1e-6, the preconditioners 1e-5.  At the ends of the range the smallest couplings turn subnormal, at
    2^-23 or less of their row's largest entry, one FP32 rounding (6e-8) in the operator, times a
    condition of 1e2 in the preconditioners."""
    out = {}
    for k in (0, -90, -80, -60, 60, 100, 124, 130):
        s = _solver(synth.workload("cube8ve"), 2.0 ** k, precision="mixed", use_tensor_cores=tc)
        ui, ue, wv = synth.initial_state(s.N, 5)
        s.linearize(ui, ue, wv)
        x = synth.random_vector(s.sizes["n_iface"], 6)
        lam = synth.random_vector(s.sizes["n_lambda"], 7)
        out[k] = (np.ldexp(s.schur_apply(x), -k), np.ldexp(s.bddc_apply(x), k), np.ldexp(s.fetidp_apply(lam), -k))
        s.close()
    for k, got in out.items():
        for y, ref, bar in zip(got, out[0], (1e-6, 1e-5, 1e-5)):
            assert np.linalg.norm(y - ref) < bar * np.linalg.norm(ref), k


@pytest.mark.parametrize("tc", [0, 1, 2])
def test_mixed_pivots_in_the_last_binades(tc):
    """Pivots of the local and coarse matrices between 2^126 and the end of FP32's range (bars as above:
    the inverses' smallest entries are subnormal)."""
    out = []
    for k in (0, 138):
        s = _solver(synth.workload("cube8ve"), 2.0 ** k, precision="mixed", use_tensor_cores=tc)
        ui, ue, wv = synth.initial_state(s.N, 5)
        s.linearize(ui, ue, wv)
        x = synth.random_vector(s.sizes["n_iface"], 6)
        out.append((np.ldexp(s.schur_apply(x), -k), np.ldexp(s.bddc_apply(x), k)))
        s.close()
    for ref, y, bar in zip(*out, (1e-6, 1e-5)):
        assert np.linalg.norm(y - ref) < bar * np.linalg.norm(ref)


@pytest.mark.parametrize("contrast", [1e2, 1e4, 1e6, 1e8, 1e-6])
def test_operator_of_media_of_different_scale(contrast):
    """FP64 with the extracellular conductivities times a contrast: tiles hold rows of both media, whose
    entries differ by that factor.  The vector is scaled so that both media give terms of the same size;
    bar 1e-12 for the rows of each medium by itself: 2^-53 times a condition of 1e3 of the scaled
    matrices and a growth of ten.  (Entries cut to a common number of bits per tile lost 1e-17 x contrast
    in the smaller medium's rows: 2e-10 at 1e8.)"""
    from oracle import ionic
    from oracle.bidomain import Problem
    from oracle.dd import DDSolver
    from paper_2101_02959_gb300 import binding, build
    build.build()
    w = synth.workload("cube8ve")
    se = tuple(v * contrast for v in synth.SIGMA_E)
    prob = Problem(w, synth.SIGMA_I, se, synth.IONIC, synth.TAU, synth.stimulus(w))
    ui, ue, wv = synth.initial_state(prob.N, 5)
    dd = DDSolver(prob)
    dd.setup(prob.p["chi_cm"] + prob.tau * ionic.di_ion_dv(ui - ue, wv, prob.p))
    x = synth.random_vector(prob.dofs.n_iface, 6)
    x[1::2] /= max(contrast, 1.0) ** 0.5
    x[dd.g_iface] = 0.0
    ref = dd.schur_apply(x)
    s = binding.Solver(w, synth.SIGMA_I, se, synth.IONIC, synth.TAU, precision="fp64")
    s.linearize(ui, ue, wv)
    y = s.schur_apply(x)
    s.close()
    for rows in (slice(0, None, 2), slice(1, None, 2)):
        assert np.linalg.norm((y - ref)[rows]) < 1e-12 * np.linalg.norm(ref[rows])


@pytest.mark.parametrize("precision,tc", [("fp64", 0), ("mixed", 0), ("mixed", 1), ("mixed", 2)])
@pytest.mark.parametrize("s", [(4, 4, 4), (7, 7, 7)])
@pytest.mark.parametrize("contrast", [1e6, 1e8])
def test_preconditioner_of_media_of_different_scale(contrast, s, precision, tc):
    """The panel solves and deluxe products of media of different scale, for the rows of each medium.  Bar
    16 u cond(D K_IDelta,IDelta D), D the square roots of the diagonal's inverse: the local solves'
    forward error does not depend on the scaling, with a growth of order ten."""
    from oracle import ionic
    from oracle.bidomain import Problem
    from oracle.dd import DDSolver
    from paper_2101_02959_gb300 import binding, build
    build.build()
    w = dict(n=tuple(2 * v for v in s), l=tuple(0.1 * v for v in s), s=s, primal="VE", name="edges")
    se = tuple(v * contrast for v in synth.SIGMA_E)
    prob = Problem(w, synth.SIGMA_I, se, synth.IONIC, synth.TAU, synth.stimulus(w))
    ui, ue, wv = synth.initial_state(prob.N, 5)
    dd = DDSolver(prob)
    dd.setup(prob.p["chi_cm"] + prob.tau * ionic.di_ion_dv(ui - ue, wv, prob.p))
    r = synth.random_vector(prob.dofs.n_iface, 8)
    r[1::2] *= contrast ** 0.5
    r[dd.g_iface] = 0.0
    ref = dd.bddc_apply(r)
    cond = 0.0
    for L in dd.loc:
        n = L["nI"] + len(L["dual"])
        K = L["Kb"][:n, :n]
        d = 1.0 / np.sqrt(np.diag(K))
        cond = max(cond, np.linalg.cond(K * d[:, None] * d))
    bar = 16.0 * 2.0 ** (-53 if precision == "fp64" else -24) * cond
    sol = binding.Solver(w, synth.SIGMA_I, se, synth.IONIC, synth.TAU, precision=precision, use_tensor_cores=tc)
    sol.linearize(ui, ue, wv)
    z = sol.bddc_apply(r)
    sol.close()
    for rows in (slice(0, None, 2), slice(1, None, 2)):
        assert np.linalg.norm((z - ref)[rows]) < bar * np.linalg.norm(ref[rows])
