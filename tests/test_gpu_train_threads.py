"""Several host threads reading one trainer: parameters and gradients arrive
whole in each caller's own memory."""
import threading

import numpy as np
import pytest

import paper_2507_01439_gb300 as trg

pytestmark = pytest.mark.gpu


def test_parameters_and_gradients_read_by_several_threads():
    import torch
    rng = np.random.default_rng(1)
    feat = torch.from_numpy(rng.normal(size=(300, 8)).astype(np.float32)).cuda()
    label = torch.from_numpy((rng.random(300) < 0.5).astype(np.float32)).cuda()
    t = trg.MLPTrainer(max_samples=300, seed=7)
    w = t.get_params()
    g, _ = t.grad(feat, label)
    assert np.abs(w - g).max() > 0.1   # a gradient in the place of parameters shows
    bad = []

    def read():
        for _ in range(1000):
            if not np.array_equal(t.get_params(), w):
                bad.append("parameters")

    def grad():
        for _ in range(1000):
            # the blocks' sums are added in any order: FP32 rounding of three of them
            if not np.allclose(t.grad(feat, label)[0], g, rtol=1e-4, atol=1e-6):
                bad.append("gradient")

    th = [threading.Thread(target=f) for f in (read, read, grad)]
    for x in th:
        x.start()
    for x in th:
        x.join()
    t.close()
    assert not bad, (len(bad), bad[:3])
