"""Weight histogram and row maxima of the pivot selection at the edges of its
row-pair groups (16 rows), 8-weight chunks and 256-chunk windows (at n = 2035 a
pair of rows holds one chunk more than a window), and, for the learned weights,
where a block takes several groups (n > 8192).  All results are whole numbers:
equal, not close."""
import numpy as np
import pytest

import paper_2507_01439_gb300 as trg
import synth
from test_zz_no_alloc import _noalloc, _packed_w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,wmax", [(3, 1), (15, 13), (16, 14), (17, 15), (31, 5), (33, 31), (257, 255), (2033, 90),
                                    (2035, 300), (4085, 60), (8179, 60), (8191, 60), (8192, 8190)])
def test_caller_weights(n, wmax):
    import oracle
    k1 = min(8192, 3 * n)
    W, S = _packed_w(n, (n + 7) // 8 * 8, wmax, n, density=0.6 if n < 1000 else 0.02)
    opi, opj, opw = oracle.pivots(S, k1)
    rc, m, got = _noalloc(W, n, k1)
    assert rc == trg.OK and m == len(opi)
    assert np.array_equal(got[:m, :3], np.stack([opi, opj, opw], 1))


@pytest.mark.parametrize("n", [8192, 8300])
def test_learned_weights_above_8192(n):
    from paper_2507_01439_gb300.train_proposal import load_model
    p = synth.make_problem("indoor", n, 0.05, 77)
    with trg.TurboReg(max_n=n) as ctx:
        ctx.set_proposal_model(load_model())
        res = ctx.register(p.x, p.y, trg.default_params(p.tau, 500, p.theta, proposal=trg.PROPOSAL_LEARNED))
        assert res.status == 0 and res.used_fallback == 0
        prob = ctx.buffer(trg.BUF_PROB)[:n].astype(np.float32)
        W = ctx.buffer(trg.BUF_SC2)[:n, :n]
        piv = ctx.buffer(trg.BUF_PIVOTS)
    lin = np.flatnonzero(np.triu(W, 1))          # floor(W p_i p_j) in the library's FP32 order
    i, j = np.divmod(lin, n)
    w = ((W[i, j].astype(np.float32) * prob[i]).astype(np.float32) * prob[j]).astype(np.float32).astype(np.int64)
    keep = np.flatnonzero(w > 0)
    order = keep[np.lexsort((lin[keep], -w[keep]))][:500]
    assert np.array_equal(piv[:, :3], np.stack([i[order], j[order], w[order]], 1))
