"""A batch in which every cluster of the SC^2 GEMM leaves several problems
behind: the histogram bins a CTA still holds belong to its last problem and to
no other, whatever the other CTA of its cluster is doing at that moment.  The
inliers come first, so that the rows of one CTA hold most of the edges and the
two CTAs of a cluster run apart.  Integers throughout: a batch's pivots,
hypotheses and inlier numbers equal single calls', on every repetition."""
import numpy as np
import pytest

import paper_2507_01439_gb300 as trg
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [0, trg.FLAG_SC2_SINGLE_CTA])
@pytest.mark.parametrize("n_lo,n_hi,num,tau", [(100, 256, 256, 0.5), (130, 400, 256, 0.3), (257, 900, 96, 0.5)])
def test_dense_small_problems_equal_single_calls(n_lo, n_hi, num, tau, flags):
    rng = np.random.default_rng(n_hi)
    probs = []
    for b in range(num):
        # sorted by quality: from nearly all inliers to few
        p = synth.make_problem("indoor", int(rng.integers(n_lo, n_hi + 1)), 0.95 - 0.8 * b / num, 500 + b)
        order = np.argsort(~p.inlier, kind="stable")
        probs.append((np.ascontiguousarray(p.x[order]), np.ascontiguousarray(p.y[order])))
    offs = np.cumsum([0] + [len(x) for x, _ in probs]).astype(np.int64)
    xs, ys = (np.concatenate([p[k] for p in probs]) for k in (0, 1))
    prm = trg.default_params(tau, 150, 0.1, flags=flags)
    with trg.TurboReg(max_n=n_hi, max_batch=num) as c:
        one = [c.register(x, y, prm) for x, y in probs]
        for _ in range(8):
            out = c.register_batched(xs, ys, offs, prm)
            for a, b in zip(one, out):
                assert (a.status, a.hypothesis, a.n_pivots, a.n_valid, a.inlier_count, a.clique) == \
                    (b.status, b.hypothesis, b.n_pivots, b.n_valid, b.inlier_count, b.clique)
                assert np.array_equal(a.R, b.R) and np.array_equal(a.t, b.t)
