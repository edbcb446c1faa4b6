"""The stream form's SC^2 path (the GEMM above n_pad = 2048) against the
synchronous call's (chosen on the device), around the sizes where the rules
change, on sparse and dense graphs: every stage's integers and the result equal."""
import numpy as np
import pytest

import paper_2507_01439_gb300 as trg
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,tau,path", [(2048, 0.1, 1), (2049, 0.05, 2), (5000, 0.1, 2), (5120, 0.4, 2), (5121, 0.1, 2)])
def test_stream_form_equals_synchronous(n, tau, path):
    import torch
    p = synth.make_problem("indoor", n, 0.05, 600 + n)
    prm = trg.default_params(tau, 500, p.theta)
    which = (trg.BUF_ROWSCORE, trg.BUF_PIVOTS, trg.BUF_CLIQUES, trg.BUF_INLIERS)
    iu = np.triu_indices(n, 1)
    with trg.TurboReg(max_n=n) as c:
        r = c.register(p.x, p.y, prm)
        ref = [c.buffer(w) for w in which] + [c.buffer(trg.BUF_SC2)[:n, :n][iu]]
        slots = trg.ResultSlots(1)
        x, y = torch.from_numpy(p.x).cuda(), torch.from_numpy(p.y).cuda()
        c.register_async(x, y, prm, slots, 0)
        c.synchronize()
        assert c.sc2_path() == path
        got = [c.buffer(w) for w in which] + [c.buffer(trg.BUF_SC2)[:n, :n][iu]]
    for a, b in zip(ref, got):
        assert np.array_equal(a, b)
    q = slots.result(0)
    assert (q.status, q.hypothesis, q.inlier_count, q.clique) == (r.status, r.hypothesis, r.inlier_count, r.clique)
    assert np.array_equal(q.R, r.R) and np.array_equal(q.t, r.t)
