"""Batches on both sides of the lines at which their passes change form, against
single calls: equal bit for bit, for mixed K2, graph and scoring too."""
import numpy as np
import pytest

import paper_2507_01439_gb300 as trg
import synth

pytestmark = pytest.mark.gpu


def _check(sizes, params, model=None):
    probs = [synth.make_problem("indoor", n, 0.05 + 0.02 * (b % 12), 3000 + 31 * b) for b, n in enumerate(sizes)]
    offs = np.cumsum([0] + list(sizes)).astype(np.int64)
    xs, ys = (np.concatenate([getattr(p, k) for p in probs]) for k in "xy")
    which = (trg.BUF_PIVOTS, trg.BUF_CLIQUES, trg.BUF_RT, trg.BUF_INLIERS)
    with trg.TurboReg(max_n=max(sizes), max_batch=len(sizes)) as c:
        if model is not None:
            c.set_proposal_model(model)
        one = [c.register(p.x, p.y, q) for p, q in zip(probs, params)]
        c.register(probs[0].x, probs[0].y, params[0])
        first = [c.buffer(w) for w in which]
        out = c.register_batched(xs, ys, offs, params)
        many = [c.buffer(w) for w in which]
    for a, b in zip(first, many):
        assert a.shape == b.shape and np.array_equal(a.view(np.uint32), b.view(np.uint32))
    for a, b in zip(one, out):
        assert (a.status, a.hypothesis, a.n_pivots, a.n_valid, a.inlier_count, a.clique, a.score) == \
            (b.status, b.hypothesis, b.n_pivots, b.n_valid, b.inlier_count, b.clique, b.score)
        assert np.array_equal(a.R, b.R) and np.array_equal(a.t, b.t)


def _sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


# the clique search's blocks (eight pivots each): 8 per SM with 13 problems and more, 16 with five, 26 with fewer
@pytest.mark.parametrize("num,per_sm", [(2, 26), (4, 26), (5, 16), (12, 16), (13, 8), (64, 8)])
@pytest.mark.parametrize("more", [0, 1])
def test_clique_search_forms(num, per_sm, more):
    k1 = 8 * (per_sm * _sms() // num + more)
    k1 = min(k1, trg.TURBOREG_K1_MAX)
    _check([900 + 7 * b for b in range(num)], [trg.default_params(0.1, k1, 0.1) for _ in range(num)])


@pytest.mark.parametrize("num", [3, 20])
def test_mixed_parameters(num):
    prm = [trg.default_params(0.1 + 0.05 * (b % 3), 50 + 400 * (b % 4), 0.1, k2=1 + b % 5,
                              graph_mode=trg.GRAPH_SC2 if b % 2 else trg.GRAPH_O2, scoring=b % 3) for b in range(num)]
    _check([150 + 97 * b for b in range(num)], prm)


# the count pass: a block per group up to 16 problems, then a warp
@pytest.mark.parametrize("num", [16, 17])
@pytest.mark.parametrize("k1", [10, 3000])
def test_count_forms(num, k1):
    _check([200 + 61 * b for b in range(num)], [trg.default_params(0.1, k1, 0.1) for _ in range(num)])


# the emit pass: up to four problems of more than 2048 matches a block per active row, else a warp
@pytest.mark.parametrize("sizes", [[2048, 2047], [2049, 40], [2500, 300, 2049, 1000], [2500, 300, 2049, 1000, 64]])
@pytest.mark.parametrize("k1", [10, 3000])
def test_emit_forms(sizes, k1):
    _check(sizes, [trg.default_params(0.1 if n > 500 else 9.0, k1, 0.1) for n in sizes])   # 9.0: complete graphs, all ties


# verification: from 16 blocks per SM on (128 hypotheses x 256 matches each, then x 512) another register budget
@pytest.mark.parametrize("num,k1", [(8, 1152), (19, 1000), (20, 1024), (40, 1024)])
@pytest.mark.parametrize("scoring", [trg.SCORE_IN, trg.SCORE_MAE, trg.SCORE_MSE])
def test_verification_forms(num, k1, scoring):
    _check([2040 + b for b in range(num)], [trg.default_params(0.1, k1, 0.1, scoring=scoring) for _ in range(num)])


# the learned proposal's weights through every form of the count and emit passes
@pytest.mark.parametrize("sizes", [[2100, 60, 3000], [300, 900, 2049, 70, 1500], [150 + 90 * b for b in range(18)]])
@pytest.mark.parametrize("k1", [20, 2000])
def test_learned_forms(sizes, k1):
    from paper_2507_01439_gb300.train_proposal import load_model
    prm = [trg.default_params(0.1, k1, 0.1, proposal=trg.PROPOSAL_LEARNED, learned_min_inliers=1) for _ in sizes]
    _check(sizes, prm, load_model())
