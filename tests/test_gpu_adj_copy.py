"""Reading the GEMM's adjacency back (TURBOREG_BUF_ADJ_FP8): equal to the
bitset for every byte count asked for, and without host memory of its own: in a
process that can allocate no more, the call still answers."""
import os
import subprocess
import sys

import numpy as np
import pytest

import paper_2507_01439_gb300 as trg
import synth

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import ctypes, resource
import numpy as np
import paper_2507_01439_gb300 as trg
import synth
n = 8192
p = synth.make_problem("indoor", n, 0.05, 1)
c = trg.TurboReg(max_n=n)
assert c.register(p.x, p.y, trg.default_params(p.tau, 100, p.theta, flags=trg.FLAG_SC2_GEMM)).status == trg.OK
dst = np.ones(n * n, dtype=np.uint8)
copy = lambda which: c._lib.turboreg_debug_copy(c.handle, which, ctypes.c_void_p(dst.ctypes.data), dst.nbytes)
assert copy(trg.BUF_SC2) == n * n          # the runtime's own staging memory is in place from here on
used = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
hard = resource.getrlimit(resource.RLIMIT_AS)[1]
resource.setrlimit(resource.RLIMIT_AS, (used + (8 << 20), hard))
got = copy(trg.BUF_ADJ_FP8)
resource.setrlimit(resource.RLIMIT_AS, (hard, hard))
assert got == n * n, got
assert set(np.unique(dst).tolist()) == {0, 0x38}
print("answered")
"""


def test_bytes_equal_the_bitset_for_any_length():
    import ctypes
    p = synth.make_problem("indoor", 300, 0.3, 2)
    with trg.TurboReg(max_n=300) as c:
        c.register(p.x, p.y, trg.default_params(0.5, 100, p.theta, flags=trg.FLAG_SC2_GEMM))
        bits = c.buffer(trg.BUF_ADJ_BITS)
        want = (np.unpackbits(bits.view(np.uint8), axis=1, bitorder="little") * 0x38).ravel()
        assert np.array_equal(c.buffer(trg.BUF_ADJ_FP8).ravel(), want) and want.any()
        for count in (0, 1, 2, 3, 511, 512, 5001, want.size - 1, want.size, want.size + 7):
            dst = np.full(want.size + 16, 0xAA, dtype=np.uint8)
            got = c._lib.turboreg_debug_copy(c.handle, trg.BUF_ADJ_FP8, ctypes.c_void_p(dst.ctypes.data), count)
            k = min(count, want.size)
            assert got == k and np.array_equal(dst[:k], want[:k]) and (dst[k:] == 0xAA).all()


def test_answers_without_host_memory():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "answered" in r.stdout, (r.returncode, r.stderr[-500:])
