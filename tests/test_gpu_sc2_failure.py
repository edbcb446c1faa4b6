"""An SC^2 GEMM one of whose workers gives up on a bounded wait
(TURBOREG_FLAG_DEBUG_STALL_SC2; no GPU fault): the weights and their histogram
are then incomplete and mixed with an earlier registration's, so every problem
of the call reports the timeout and nothing is selected from them; the next
call is unaffected."""
import numpy as np
import pytest

import paper_2507_01439_gb300 as trg
import synth

pytestmark = pytest.mark.gpu


def _same(a, b):
    return (a.status == b.status and a.hypothesis == b.hypothesis and a.inlier_count == b.inlier_count
            and np.array_equal(a.R, b.R) and np.array_equal(a.t, b.t) and a.n_pivots == b.n_pivots)


@pytest.mark.parametrize("extra", [0, trg.FLAG_SC2_SINGLE_CTA, trg.FLAG_NO_GRAPH])
def test_one_problem(extra):
    dense = synth.make_problem("indoor", 3000, 0.8, 1)     # large weights left behind
    p = synth.make_problem("indoor", 2700, 0.05, 2)
    prm = trg.default_params(p.tau, 500, p.theta, flags=trg.FLAG_SC2_GEMM | extra)
    stall = trg.default_params(p.tau, 500, p.theta, flags=trg.FLAG_SC2_GEMM | extra | trg.FLAG_DEBUG_STALL_SC2)
    with trg.TurboReg(max_n=3000) as c:
        ref = c.register(p.x, p.y, prm)
        c.register(dense.x, dense.y, prm)
        bad = c.register(p.x, p.y, stall)
        after = c.register(p.x, p.y, prm)
    assert ref.status == trg.OK and _same(ref, after)
    assert bad.status == trg.ERR_TIMEOUT and bad.n_pivots == 0 and bad.hypothesis == -1


def test_batch():
    probs = [synth.make_problem("indoor", n, 0.3, 60 + b) for b, n in enumerate([700, 300, 1500, 900] * 40)]
    offs = np.cumsum([0] + [q.n for q in probs]).astype(np.int64)
    xs, ys = np.concatenate([q.x for q in probs]), np.concatenate([q.y for q in probs])
    prm = trg.default_params(0.1, 200, 0.1)
    stall = trg.default_params(0.1, 200, 0.1, flags=trg.FLAG_DEBUG_STALL_SC2)
    with trg.TurboReg(max_n=1500, max_batch=len(probs)) as c:
        ref = c.register_batched(xs, ys, offs, prm)
        bad = c.register_batched(xs, ys, offs, stall)
        after = c.register_batched(xs, ys, offs, prm)
    assert all(r.status == trg.OK for r in ref)
    assert all(r.status == trg.ERR_TIMEOUT and r.n_pivots == 0 and r.hypothesis == -1 for r in bad)
    assert all(_same(a, b) for a, b in zip(ref, after))
