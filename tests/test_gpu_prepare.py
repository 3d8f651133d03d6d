"""What preparing a layer for the tensor-core batches adds on the host: the
work profile of a tensor without a row factor repeats from group to group, so
max_batch 16 costs little more than max_batch 1."""
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


def test_profile_of_equal_groups():
    from paper_2609_38477_gb300 import build

    build.build()
    from paper_2609_38477_gb300 import seedq as Q

    R, C = 128256, 4096
    a = np.exp(np.random.default_rng(1).normal(0, 1, C)).astype(np.float32)

    def prepare(max_batch):
        t = time.perf_counter()
        L = Q.Layer(R, C, a, None, RUNGS, THETA, -1, 0.1, 0, max_batch=max_batch)
        t = time.perf_counter() - t
        L.release()
        return t

    times = {b: [] for b in (1, 16)}
    for _ in range(12):
        for b in times:
            times[b].append(prepare(b))
    assert min(times[16]) < 1.25 * min(times[1]), {b: min(v) for b, v in times.items()}
