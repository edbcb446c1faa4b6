"""The training kernel's grid in a process that creates a trainer and no
registration context: one block per SM of the device it runs on, and the
gradient right on both sides of the count at which a block takes a second
tile of 128 samples (tolerance as for the tiles' edges: three roundings of an
operand to BF16, 2^-9 each, in a chain to the first layer, and room for a ReLU
whose input the two sides round to different signs)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import numpy as np
import torch
import oracle.mlp as omlp
import paper_2507_01439_gb300 as trg
sms = torch.cuda.get_device_properties(0).multi_processor_count
t = trg.MLPTrainer(max_samples=(sms + 1) * 128, seed=11)
for m, want in ((128, 1), (129, 2), (sms * 128, sms), (sms * 128 + 1, sms)):
    assert t._lib.turboreg_mlp_debug_blocks(t.handle, m) == want, (m, want)
for m in (sms * 128, sms * 128 + 1):
    rng = np.random.default_rng(m)
    f, lab = rng.normal(size=(m, 8)).astype(np.float32), (rng.random(m) < 0.5).astype(np.float32)
    g, loss = t.grad(torch.from_numpy(f).cuda(), torch.from_numpy(lab).cuda())
    gw, lw = omlp.grad(t.get_params().astype(np.float64), f, lab, bf16_round=True)
    assert abs(loss - lw) < 1e-3 * max(1.0, abs(lw))
    o = 0
    for name, shape in omlp.SIZES:
        k = int(np.prod(shape))
        rel = np.linalg.norm(g[o:o + k] - gw[o:o + k]) / max(np.linalg.norm(gw[o:o + k]), 1e-12)
        assert rel <= 1e-2, (name, rel)
        o += k
print("grid ok")
"""


def test_one_block_per_sm_without_a_context():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "grid ok" in r.stdout, (r.returncode, r.stderr[-800:])
