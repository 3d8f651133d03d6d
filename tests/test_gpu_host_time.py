"""Host time of a product call: the cut of a launch into ranges looks at every
row group of a tensor once, so even 4008 of them cost less than the launch."""
import os
import sys
import time

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

RUNGS = [(8, 2), (10, 3), (12, 3), (16, 3), (14, 4), (16, 5), (16, 6)]
THETA = [0.3, 0.5, 0.8, 1.2, 2.0, 3.5]


def _call_time(R, C, n):
    from paper_2609_38477_gb300 import build

    build.build()
    from paper_2609_38477_gb300 import seedq as Q

    a = np.exp(np.random.default_rng(1).normal(0, 1, C)).astype(np.float32)
    L = Q.Layer(R, C, a, None, RUNGS, THETA, -1, 0.1, 0, max_batch=4)
    nbytes = Q.stream_bytes_required(L.stream_bits)
    buf = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    L.synth_stream(3, buf, nbytes)
    L.bind_stream(buf, L.stream_bits, nbytes)
    x = torch.randn((n, C), device="cuda").to(torch.bfloat16)
    y = torch.empty((n, R), device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    best = 1e9
    for _ in range(15):
        torch.cuda.synchronize()
        t = time.perf_counter()
        for _ in range(100):
            L.gemm_small_batch(x, n, y, stream)
        best = min(best, (time.perf_counter() - t) / 100 * 1e6)
    torch.cuda.synchronize()
    L.release()
    return best


@pytest.mark.parametrize("n", [1, 4])
def test_many_row_groups(n):
    few, many = _call_time(64, 128, n), _call_time(128256, 128, n)
    print(f"n = {n}: {few:.1f} us at 2 row groups, {many:.1f} at 4008")
    assert many < 1.9 * few
