"""A batch's own kernels (warp-wide count and emit passes, sorted pivots, the
separate Kabsch) against one problem's, for every K2 form, at sizes around a
row group (16 rows), a warp's sweep and a block's keys: pivots, cliques and
every hypothesis equal bit for bit."""
import numpy as np
import pytest

import paper_2507_01439_gb300 as trg
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k1,k2,tau,graph", [
    (40, 7, 1, 0.1, trg.GRAPH_O2), (129, 64, 2, 0.3, trg.GRAPH_O2), (257, 65, 3, 0.5, trg.GRAPH_SC2),
    (1025, 2049, 4, 0.1, trg.GRAPH_O2), (2049, 1000, 2, 0.1, trg.GRAPH_SC2), (3000, 8192, 5, 0.2, trg.GRAPH_O2),
    (600, 300, 2, 9.0, trg.GRAPH_O2),            # complete graph: every edge ties, every row is active
])
def test_batch_equals_single(n, k1, k2, tau, graph):
    p = synth.make_problem("indoor", n, 0.1, 9000 + n)
    other = synth.make_problem("cube", 333, 0.1, 5)
    prm = trg.default_params(tau, k1, p.theta, k2=k2, graph_mode=graph)
    which = (trg.BUF_PIVOTS, trg.BUF_CLIQUES, trg.BUF_RT, trg.BUF_INLIERS)
    with trg.TurboReg(max_n=max(n, 333), max_batch=3) as c:
        r = c.register(p.x, p.y, prm)
        one = [c.buffer(w) for w in which]
        offs = np.cumsum([0, n, 333, n]).astype(np.int64)
        out = c.register_batched(np.concatenate([p.x, other.x, p.x]), np.concatenate([p.y, other.y, p.y]), offs, prm)
        many = [c.buffer(w) for w in which]
    for a, b in zip(one, many):
        assert a.shape == b.shape and np.array_equal(a.view(np.uint32), b.view(np.uint32))
    for b in (0, 2):
        assert (out[b].status, out[b].hypothesis, out[b].n_pivots, out[b].n_valid, out[b].inlier_count, out[b].clique) == \
            (r.status, r.hypothesis, r.n_pivots, r.n_valid, r.inlier_count, r.clique)
        assert np.array_equal(out[b].R, r.R) and np.array_equal(out[b].t, r.t)
