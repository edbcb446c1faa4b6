"""SC^2 forms against one another at the edges of the GEMM's block order and
of its shared-memory plan: N around the multiples of 256 and 2048 (one block,
a panel of eight column blocks, the first block of the next panel) and on
both sides of the N at which the histogram takes a ring stage away (8575,
16767, 24959).  Integers throughout: everything must be equal."""
import numpy as np
import pytest

import paper_2507_01439_gb300 as trg
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [256, 257, 2048, 2049, 4097, 8575, 8576, 16767, 16768, 24959, 24960])
def test_gemm_forms_equal_bitset(n):
    p = synth.make_problem("indoor", n, 0.03, 4000 + n)
    got = []
    with trg.TurboReg(max_n=n) as c:
        for fl in (trg.FLAG_SC2_BITSET, trg.FLAG_SC2_GEMM, trg.FLAG_SC2_SINGLE_CTA):
            r = c.register(p.x, p.y, trg.default_params(p.tau, 1000, p.theta, flags=fl))
            got.append((r, c.buffer(trg.BUF_ROWSCORE), c.buffer(trg.BUF_PIVOTS), c.buffer(trg.BUF_CLIQUES)))
    ref = got[0]
    assert ref[0].status == 0
    for r, rows, piv, cl in got[1:]:
        assert np.array_equal(rows, ref[1]) and np.array_equal(piv, ref[2]) and np.array_equal(cl, ref[3])
        assert r.hypothesis == ref[0].hypothesis and r.inlier_count == ref[0].inlier_count
        assert np.array_equal(r.R, ref[0].R) and np.array_equal(r.t, ref[0].t)


@pytest.mark.parametrize("flags", [0, trg.FLAG_SC2_SINGLE_CTA])
def test_gemm_batch_in_chunks_equals_single_calls(flags):
    # enough blocks that every worker takes several of them in a row: a chunk
    # then ends inside, at the end of and past a problem
    sizes = [2600, 300, 2048, 2049, 1100, 3000, 256, 700] * 8
    probs = [synth.make_problem("indoor", n, 0.05, 700 + b) for b, n in enumerate(sizes)]
    offs = np.cumsum([0] + sizes).astype(np.int64)
    prm = trg.default_params(0.1, 200, 0.1, flags=flags)
    with trg.TurboReg(max_n=3000, max_batch=len(sizes)) as c:
        out = c.register_batched(np.concatenate([p.x for p in probs]), np.concatenate([p.y for p in probs]), offs, prm)
        for b in (0, 1, 2, 3, 5, 6, 31, 62, 63):
            r = c.register(probs[b].x, probs[b].y, prm)
            assert (r.status, r.hypothesis, r.n_pivots, r.inlier_count) == \
                (out[b].status, out[b].hypothesis, out[b].n_pivots, out[b].inlier_count)
            assert np.array_equal(r.R, out[b].R) and np.array_equal(r.t, out[b].t)
