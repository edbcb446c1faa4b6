"""The emit pass of the pivot selection on both sides of the size at which one
problem changes from a warp to a block per active row (a row is one sweep of a
warp up to n = 1024): the allocation-free selection against a sort, and the
registration's pivots against the same.  Whole numbers throughout."""
import numpy as np
import pytest

import paper_2507_01439_gb300 as trg
import synth

pytestmark = pytest.mark.gpu

SIZES = [1016, 1023, 1024, 1025, 1032, 2047, 2048, 2049]


def _top(w, k1):
    """The k1 heaviest edges above the diagonal, heavier first, then lower (i, j)."""
    n = w.shape[0]
    i, j = np.triu_indices(n, 1)
    x = w[i, j].astype(np.int64)
    i, j, x = i[x > 0], j[x > 0], x[x > 0]
    o = np.lexsort((j, i, -x))[:k1]
    return np.stack([i[o], j[o], x[o], np.zeros_like(i[o])], 1)


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("few", [False, True])
def test_selection(n, few):
    import torch
    rng = np.random.default_rng(n)
    w = rng.integers(0, 40, (n, n)) * (rng.random((n, n)) < 0.3)   # heavy ties
    if few:                                                        # a handful of full rows
        w[rng.random(n) < 0.98] = 0
    ld = (n + 7) // 8 * 8
    wd = torch.zeros(n, ld, dtype=torch.int32, device="cuda")
    wd[:, :n] = torch.from_numpy(w.astype(np.int32)).cuda()
    wd = wd.to(torch.uint16)
    for k1 in (1, 700, 8192):
        piv = torch.zeros(k1, 4, dtype=torch.int32, device="cuda")
        cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
        assert trg.turboreg_select_pivots_noalloc(wd, n, ld, k1, piv, cnt) == trg.OK
        want = _top(w, k1)
        assert int(cnt) == len(want)
        assert np.array_equal(piv.cpu().numpy()[:len(want)], want)


@pytest.mark.parametrize("n", SIZES)
def test_registration(n):
    p = synth.make_problem("indoor", n, 0.1, n)
    with trg.TurboReg(max_n=n) as c:
        c.register(p.x, p.y, trg.default_params(p.tau, 1500, p.theta))
        w = np.triu(c.buffer(trg.BUF_SC2)[:n, :n], 1)
        assert np.array_equal(c.buffer(trg.BUF_PIVOTS), _top(w, 1500))
