"""Results of calls with device tensors while torch's current stream, another one than the handle's, is
busy: the result holds when the call returns, whatever is still queued on the current stream."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("own", [True, False])
def test_results_while_the_current_stream_is_busy(own):
    torch = pytest.importorskip("torch")
    from paper_2101_02959_gb300 import binding, build
    build.build()
    w = synth.workload("cube8ve")
    stream = None if own else torch.cuda.Stream()
    s = binding.Solver(w, synth.SIGMA_I, synth.SIGMA_E, synth.IONIC, synth.TAU,
                       stream=None if own else stream.cuda_stream)
    if not own:
        assert s._lib.bidomain_stream(s._h) == stream.cuda_stream
    ui, ue, wv = (torch.from_numpy(a).cuda() for a in synth.initial_state(s.N, 5))
    x = torch.from_numpy(synth.random_vector(s.sizes["n_iface"], 6)).cuda()
    lam = torch.from_numpy(synth.random_vector(s.sizes["n_lambda"], 7)).cuda()
    torch.cuda.synchronize()
    s.linearize(ui, ue, wv)
    s.set_state(ui, ue, wv, 0.0)
    f = s.residual(None, synth.TAU, ui, ue, wv, ui - 1.0, ue)
    f = f - f.mean()
    torch.cuda.synchronize()
    calls = {
        "schur": lambda: s.schur_apply(x), "bddc": lambda: s.bddc_apply(x), "feti": lambda: s.fetidp_apply(lam),
        "operator": lambda: s.fetidp_operator(lam), "gating": lambda: s.gating(ui, ue, wv),
        "residual": lambda: s.residual(None, synth.TAU, ui, ue, wv, ui, ue), "solve": lambda: s.krylov_solve(f)[0],
        "state": lambda: s.get_state(like=ui)[1],
    }
    side = torch.cuda.Stream()
    for name, call in calls.items():
        ref = call().cpu()
        with torch.cuda.stream(side):
            junk = torch.full((ref.numel(),), 7.0, dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            torch.cuda._sleep(int(4e8))  # about 0.2 s
            junk.add_(1.0)
            del junk  # its memory is free for the current stream's next tensor, but still to be written
            y = call()
            assert not side.query(), name
        torch.cuda.synchronize()
        assert np.array_equal(y.cpu().numpy(), ref.numpy()), name
    s.close()
