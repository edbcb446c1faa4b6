"""The SC^2 GEMM at the sizes where its shared-memory plan changes.  One
problem, pair MMAs: each CTA's bins beside five ring stages up to N = 7423, the
bins split over the pair up to 14846, each CTA's beside four stages up to 15615,
split again from there, beside three stages from 31231.  Single CTAs: three
stages up to 11519, then two.  Whole numbers throughout: equal to the
CUDA-core form."""
import numpy as np
import pytest

import paper_2507_01439_gb300 as trg
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,flag", [(n, trg.FLAG_SC2_GEMM) for n in (14846, 14847, 15615, 15616, 31230, 31231)] +
                                   [(n, trg.FLAG_SC2_SINGLE_CTA) for n in (11519, 11520)])
def test_gemm_equals_bitset_where_the_plan_changes(n, flag):
    p = synth.make_problem("indoor", n, 0.03, 7000 + n)
    got = []
    with trg.TurboReg(max_n=n) as c:
        for fl in (trg.FLAG_SC2_BITSET, flag):
            r = c.register(p.x, p.y, trg.default_params(p.tau, 1000, p.theta, flags=fl))
            got.append((r, [c.buffer(w) for w in (trg.BUF_ROWSCORE, trg.BUF_PIVOTS, trg.BUF_CLIQUES)]))
    (a, x), (b, y) = got
    assert a.status == trg.OK
    assert (a.hypothesis, a.n_pivots, a.inlier_count) == (b.hypothesis, b.n_pivots, b.inlier_count)
    assert np.array_equal(a.R, b.R) and np.array_equal(a.t, b.t)
    for u, v in zip(x, y):
        assert np.array_equal(u, v)
