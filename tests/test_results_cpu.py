"""Results of a batched call converted a field at a time equal the ones
converted one by one (values, types, shapes)."""
import numpy as np

import paper_2507_01439_gb300 as trg


def test_list_from_c_equals_from_c():
    rng = np.random.default_rng(3)
    out = (trg.turboreg_result * 7)()
    for r in out:
        r.R[:] = rng.normal(size=9).tolist()
        r.t[:] = rng.normal(size=3).tolist()
        r.clique[:] = rng.integers(-1, 99, 3).tolist()
        r.score = float(rng.normal())
        for f in ("inlier_count", "hypothesis", "n_pivots", "n_valid", "used_fp64", "used_fallback", "status"):
            setattr(r, f, int(rng.integers(-1, 1 << 20)))
    got = trg.Result.list_from_c(out)
    assert len(got) == 7
    for a, b in zip(got, map(trg.Result.from_c, out)):
        for f in ("R", "t"):
            x, y = getattr(a, f), getattr(b, f)
            assert x.dtype == y.dtype == np.float32 and x.shape == y.shape and np.array_equal(x, y)
            assert x.flags.writeable and y.flags.writeable
        for f in ("clique", "inlier_count", "hypothesis", "n_pivots", "n_valid", "used_fp64", "used_fallback", "status",
                  "score"):
            assert getattr(a, f) == getattr(b, f) and type(getattr(a, f)) is type(getattr(b, f)), f
