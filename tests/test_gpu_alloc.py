"""The allocator's device search against the oracle's sequential bisections,
field for field, on inputs that stress its shortcuts: equal and nearly equal
block means (the high-word search), values whose sums round (the sequential
sums), zeros and subnormals, one row and many, and every probe count."""
import os
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
sys.path.insert(0, os.path.join(ROOT, "oracle"))

import oracle as O  # noqa: E402
from paper_2609_38477_gb300 import workloads as W  # noqa: E402

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _factors(kind, rng):
    one = lambda C: np.ones(C, np.float32)
    ln = lambda n, s: np.exp(rng.normal(0, s, n)).astype(np.float32)
    if kind == "equal":
        return [(40, 256, one(256), None), (300, 128, one(128), one(300)), (33, 64, one(64), ln(33, 1.0))]
    if kind == "nearly_equal":  # within 2^-20 of one another: one high word for all
        return [(64, 512, (1.0 + 1e-7 * rng.integers(0, 4, 512)).astype(np.float32), ln(64, 0.5)),
                (1, 800, (1.0 + 1e-7 * rng.integers(0, 9, 800)).astype(np.float32), None)]
    if kind == "rounding_sums":  # 2^-100 to 2^60: partial sums round, so order matters
        a = np.ldexp(rng.uniform(1, 2, 640), rng.integers(-100, 60, 640)).astype(np.float32)
        r = np.ldexp(rng.uniform(1, 2, 257), rng.integers(-40, 30, 257)).astype(np.float32)
        return [(257, 640, a, r), (5, 640, a[::-1].copy(), None)]
    if kind == "zeros":
        a = ln(320, 1.0)
        a[:200] = 0.0
        b = ln(320, 1.0)
        b[:50] = 1e-42
        return [(70, 320, a, ln(70, 0.5)), (70, 320, b, None)]
    if kind == "long_row":
        return [(3, 65536, ln(65536, 1.0), ln(3, 0.5)), (1, 8, ln(8, 1.0), None)]
    return [(R, 96, ln(96, 0.7), ln(R, 0.5)) for R in (1, 255, 256, 257, int(kind))]


# The numbers are the rows of the largest tensor: 31, 15, 7, 3 and 1 probes.
@pytest.mark.parametrize("kind", ["equal", "nearly_equal", "rounding_sums", "zeros", "long_row", "900", "2400", "6000",
                                  "12000", "40000"])
def test_search_matches_oracle(kind):
    from paper_2609_38477_gb300 import build

    build.build()
    from paper_2609_38477_gb300 import seedq as Q

    rungs, _, slopes = O.hull_rungs(W.DAMAGE_TABLES["llama2_7b"](), 4.0)
    fs = _factors(kind, np.random.default_rng(sum(map(ord, kind))))
    ts = [O.Tensor(R, C, a, rho) for R, C, a, rho in fs]
    for rbar, floor_f in ((3.9, 0.06), (4.4, 0.0)):
        try:
            s, T, bits = O.allocate(ts, rungs, slopes, rbar, floor_f)
        except RuntimeError:
            with pytest.raises(Q.SeedQError) as e:
                Q.allocate(fs, rungs, slopes, rbar, floor_f)
            assert e.value.status == 3
            continue
        got = Q.allocate(fs, rungs, slopes, rbar, floor_f)
        assert list(got[0]) == list(s.theta) and got[1] == s.j_tie and got[2] == s.q
        assert list(got[3]) == list(T) and list(got[4]) == list(bits)
