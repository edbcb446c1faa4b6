"""The fused training kernel at the edges of its 128-sample tiles and of its
one-CTA-per-SM grid: loss and gradient against the FP64 oracle.

Tolerance, per layer and relative in the 2-norm: dz3, dz2 and the operands of
the next product are each rounded to BF16 once (2^-9 per element), three
roundings in a chain to the first layer, so at most 3 * 2^-9 = 5.9e-3; FP32
accumulation adds less than 1e-5.  1e-2 leaves the rest for a ReLU whose input
the two sides round to different signs."""
import numpy as np
import pytest

import oracle.mlp as omlp
import paper_2507_01439_gb300 as trg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 31, 127, 128, 129, 300, 152 * 128, 152 * 128 + 1])
def test_gradient_at_tile_edges(m):
    import torch
    rng = np.random.default_rng(1000 + m)
    f = rng.normal(size=(m, 8)).astype(np.float32)
    lab = (rng.random(m) < 0.5).astype(np.float32)
    t = trg.MLPTrainer(max_samples=m, seed=11)
    th = t.get_params()
    th[trg.TURBOREG_MLP_PARAMS - 65:] += 0.1       # W4 and b4 away from their initial values
    t.set_params(th)
    # features at an address that is only 4-byte aligned
    buf = torch.empty(8 * m + 1, device="cuda")
    buf[1:] = torch.from_numpy(f.ravel()).cuda()
    g, loss = t.grad(buf[1:].view(m, 8), torch.from_numpy(lab).cuda())
    gw, lw = omlp.grad(th.astype(np.float64), f, lab, bf16_round=True)
    assert abs(loss - lw) < 1e-3 * max(1.0, abs(lw))
    o = 0
    for name, shape in omlp.SIZES:
        k = int(np.prod(shape))
        a, b = g[o:o + k].astype(np.float64), gw[o:o + k]
        rel = np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-12)
        assert rel <= 1e-2, (name, rel)
        o += k
    t.close()
