"""A bounded wait that gives up inside a training pass, injected without a GPU
fault (turboreg_mlp_debug_stall: every block waits 20 ms for a barrier on which
nothing arrives).  The wait expires long before the pass adds to the gradient,
while the clearing of the gradient and of the error bits may still be running."""
import numpy as np
import pytest

import paper_2507_01439_gb300 as trg

pytestmark = pytest.mark.gpu


def _batch(m):
    import torch
    rng = np.random.default_rng(m)
    feat = rng.normal(size=(m, 8)).astype(np.float32)
    label = (rng.random(m) < 0.5).astype(np.float32)
    return torch.from_numpy(feat).cuda(), torch.from_numpy(label).cuda()


@pytest.mark.parametrize("m", [100, 5000])
def test_gradient_reports_an_expired_wait_and_recovers(m):
    feat, label = _batch(m)
    t = trg.MLPTrainer(max_samples=m, seed=5)
    ref, loss = t.grad(feat, label)
    for _ in range(3):
        assert t._lib.turboreg_mlp_debug_stall(t.handle, 1) == trg.OK
        with pytest.raises(RuntimeError, match="timed out"):
            t.grad(feat, label)
        g, l = t.grad(feat, label)   # the next pass is unaffected
        # the blocks' sums are added in any order: FP32 rounding of at most 152 of them
        np.testing.assert_allclose(g, ref, rtol=1e-4, atol=1e-6)
        assert abs(l - loss) <= 1e-5
    t.close()


def test_step_reports_an_expired_wait_and_leaves_the_weights(m=3000):
    feat, label = _batch(m)
    t = trg.MLPTrainer(max_samples=m, seed=5)
    t.train_step(feat, label, 1e-3, want_loss=True)
    w, (mom, vel, step) = t.get_params(), t.get_state()
    stall = t._lib.turboreg_mlp_debug_stall
    assert stall(t.handle, 1) == trg.OK
    with pytest.raises(RuntimeError, match="timed out"):
        t.train_step(feat, label, 1e-3, want_loss=True)
    assert stall(t.handle, 2) == trg.OK          # two steps that nobody waits for, then a good one
    for _ in range(3):
        t.train_step(feat, label, 1e-3)
    with pytest.raises(RuntimeError, match="timed out"):
        t.get_params()                           # reported once, by the next call that waits
    m2, v2, step2 = t.get_state()
    assert step2 == step + 1                     # only the good step counts
    g, _ = t.grad(feat, label)
    assert np.isfinite(g).all() and not np.array_equal(t.get_params(), w)
    # stalled steps alone change nothing
    w, (mom, vel, step) = t.get_params(), t.get_state()
    assert stall(t.handle, 1) == trg.OK
    with pytest.raises(RuntimeError, match="timed out"):
        t.train_step(feat, label, 1e-3, want_loss=True)
    assert np.array_equal(t.get_params(), w)
    got = t.get_state()
    assert np.array_equal(got[0], mom) and np.array_equal(got[1], vel) and got[2] == step
    t.close()
