"""A clique's R, t and kappa are the same bits wherever it is solved: in one
problem's clique search, in a large batch's solve kernel and by the
clique-Kabsch entry point, for well- and ill-conditioned cliques."""
import numpy as np
import pytest

import paper_2507_01439_gb300 as trg
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k2", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("thin", [1.0, 1e-2, 1e-4])
def test_every_kernel_solves_a_clique_to_the_same_bits(k2, thin):
    p = synth.make_problem("indoor", 900, 0.4, 70 + k2)
    rng = np.random.default_rng(k2)
    x = p.x.copy()
    x[:, 1:] *= np.float32(thin)     # a thin cloud: nearly collinear cliques
    y = (x @ p.R_gt.T + p.t_gt + rng.normal(size=x.shape) * 1e-3).astype(np.float32)
    fill = [synth.make_problem("indoor", 300, 0.2, 900 + b) for b in range(63)]
    prm, pf = trg.default_params(p.tau, 500, p.theta, k2=k2), trg.default_params(0.1, 300, 0.1, k2=k2)
    with trg.TurboReg(max_n=900, max_batch=64) as c:
        one = c.register(x, y, prm)
        cl, rt = c.buffer(trg.BUF_CLIQUES), c.buffer(trg.BUF_RT)
        offs = np.cumsum([0, 900] + [q.n for q in fill]).astype(np.int64)
        out = c.register_batched(np.concatenate([x] + [q.x for q in fill]), np.concatenate([y] + [q.y for q in fill]),
                                 offs, [prm] + [pf] * 63)
        many = c.buffer(trg.BUF_RT)
        ok = cl[:, 3] == 1
        entry, valid = c.kabsch_cliques(x, y, cl[ok][:, :3], prm)
    flags = rt[:, 13].view(np.int32)
    v = flags & 1 == 1
    assert v.sum() > 100 and (thin == 1.0 or (flags & 2 != 0).any())
    assert np.array_equal(rt.view(np.uint32), many.view(np.uint32))
    assert np.array_equal(valid, v[ok])
    assert np.array_equal(entry[valid].view(np.uint32), np.ascontiguousarray(rt[v][:, :12]).view(np.uint32))
    assert one.hypothesis == out[0].hypothesis and np.array_equal(one.R, out[0].R) and np.array_equal(one.t, out[0].t)
