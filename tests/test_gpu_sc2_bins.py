"""Where the SC^2 GEMM keeps its histogram bins: in each CTA beside five ring
stages (N <= 7423), split over the CTA pair for one larger problem, in each CTA
beside fewer stages in a batch (N <= 31999), and in global memory above that or
with single CTAs above N = 23807.  Integers throughout: everything equal."""
import numpy as np
import pytest

import paper_2507_01439_gb300 as trg
import synth

pytestmark = pytest.mark.gpu

BUFS = (trg.BUF_ROWSCORE, trg.BUF_PIVOTS, trg.BUF_CLIQUES)


def _same(a, b):
    assert (a[0].status, a[0].hypothesis, a[0].n_pivots, a[0].inlier_count) == \
        (b[0].status, b[0].hypothesis, b[0].n_pivots, b[0].inlier_count)
    assert np.array_equal(a[0].R, b[0].R) and np.array_equal(a[0].t, b[0].t)
    for x, y in zip(a[1], b[1]):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("n,flags", [
    (7423, (trg.FLAG_SC2_GEMM, trg.FLAG_SC2_BITSET)), (7424, (trg.FLAG_SC2_GEMM, trg.FLAG_SC2_BITSET)),
    (23807, (trg.FLAG_SC2_GEMM, trg.FLAG_SC2_SINGLE_CTA)), (23808, (trg.FLAG_SC2_GEMM, trg.FLAG_SC2_SINGLE_CTA))])
def test_one_problem(n, flags):
    p = synth.make_problem("indoor", n, 0.03, 8000 + n)
    got = []
    with trg.TurboReg(max_n=n) as c:
        for fl in flags:
            r = c.register(p.x, p.y, trg.default_params(p.tau, 1000, p.theta, flags=fl))
            got.append((r, [c.buffer(w) for w in BUFS]))
    assert got[0][0].status == 0
    _same(got[0], got[1])


@pytest.mark.parametrize("n", [7424, 31999, 32000])
def test_batch(n):
    p, q = synth.make_problem("indoor", n, 0.03, 8000 + n), synth.make_problem("indoor", 3000, 0.05, 3)
    prm = trg.default_params(p.tau, 1000, p.theta)
    with trg.TurboReg(max_n=n, max_batch=2) as c:
        r = c.register(p.x, p.y, prm)
        one = (r, [c.buffer(w) for w in BUFS])
        out = c.register_batched(np.concatenate([p.x, q.x]), np.concatenate([p.y, q.y]),
                                 np.array([0, n, n + 3000], dtype=np.int64), prm)
        _same(one, (out[0], [c.buffer(w) for w in BUFS]))
        r2 = c.register(q.x, q.y, prm)
        assert (out[1].hypothesis, out[1].inlier_count) == (r2.hypothesis, r2.inlier_count)
        assert np.array_equal(out[1].R, r2.R)
