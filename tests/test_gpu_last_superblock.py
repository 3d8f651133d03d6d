"""The tensor-core batch products where the last superblock of 128 rows is not
full: about the time of the whole one (a CTA passes over its columns at nearly
the same pace), not the time of the columns that one CTA would get if its rows
alone counted."""
import os
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

RUNGS = [(8, 2), (10, 3), (12, 3), (16, 3), (14, 4), (16, 5), (16, 6)]
THETA = [0.3, 0.5, 0.8, 1.2, 2.0, 3.5]
C = 5008


def _time(R, n):
    from paper_2609_38477_gb300 import build

    build.build()
    from paper_2609_38477_gb300 import seedq as Q

    a = np.exp(np.random.default_rng(1).normal(0, 1, C)).astype(np.float32)
    L = Q.Layer(R, C, a, None, RUNGS, THETA, -1, 0.1, 0, max_batch=16)
    nbytes = Q.stream_bytes_required(L.stream_bits)
    buf = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    L.synth_stream(3, buf, nbytes)
    L.bind_stream(buf, L.stream_bits, nbytes)
    x = torch.randn((n, C), device="cuda").to(torch.bfloat16)
    y = torch.empty((n, R), device="cuda")
    best = 1e9
    for _ in range(8):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(20):
            L.gemm_small_batch(x, n, y)
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    L.release()
    return best


@pytest.mark.parametrize("n", [8, 16])
@pytest.mark.parametrize("rows", [8, 32, 70])
def test_time_next_to_a_whole_superblock(rows, n):
    assert _time(39 * 128 + rows, n) < 1.25 * _time(40 * 128, n)
