"""The tensor-core batch products on small tensors: how a launch is cut (at
least a few columns per CTA, cuts moved to the ends of superblocks) against
the oracle's weights in fp64, at sizes around those rules, and its time next to
the four-column products, whose kernel pays no such cuts."""
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

RUNGS = [(8, 2), (10, 3), (12, 3), (16, 3), (14, 4), (16, 5), (16, 6)]
THETA = [0.3, 0.5, 0.8, 1.2, 2.0, 3.5]
# tests/test_gpu_gemm.py derives it; the partial sums of a cut superblock carry
# their rounding errors along, so more CTAs per superblock do not add to it.
TOL = 2e-5


def _layer(R, C, spread, seed=1):
    from paper_2609_38477_gb300 import build

    build.build()
    from paper_2609_38477_gb300 import seedq as Q

    rng = np.random.default_rng(seed)
    a = np.exp(rng.normal(0, 1, C)).astype(np.float32)
    rho = np.exp(rng.normal(0, spread, R)).astype(np.float32) if spread else None
    L = Q.Layer(R, C, a, rho, RUNGS, THETA, -1, 0.1, 0, max_batch=16)
    nbytes = Q.stream_bytes_required(L.stream_bits)
    buf = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    L.synth_stream(seed, buf, nbytes)
    L.bind_stream(buf, L.stream_bits, nbytes)
    return L, a, rho


@pytest.mark.parametrize("R,C,spread", [(128, 8, 0), (128, 88, 0), (300, 96, 0.5), (256, 1216, 0), (200, 1224, 0.7),
                                        (5 * 128, 2432, 0), (13 * 128 + 1, 1040, 0.5), (20 * 128, 400, 0.3)])
def test_products_at_the_cuts(R, C, spread):
    L, a, rho = _layer(R, C, spread, R + C)
    Wm = O.Tensor(R, C, a, rho).synth_rows(O.Sched(RUNGS, THETA, -1, 0.1), 0, R + C, 0, R).astype(np.float64)
    for n in (8, 11):
        b = W.to_bf16_bits(np.random.default_rng(n).normal(0, 1, (n, C)).astype(np.float32).ravel()).reshape(n, C)
        x = W.bf16_bits_to_f32(b).astype(np.float64)
        y = torch.full((n, R), 7.0, device="cuda")
        L.gemm_small_batch(torch.from_numpy(b.view(np.int16)).cuda(), n, y)
        y = y.cpu().numpy().astype(np.float64)
        assert np.all(np.abs(y - x @ Wm.T) <= TOL * (np.abs(x) @ np.abs(Wm).T))
    assert L.device_error() == 0
    L.release()


@pytest.mark.parametrize("R,C", [(128, 1040), (256, 5008), (640, 5008), (1024, 1040)])
def test_time_next_to_four_columns(R, C):
    L, _, _ = _layer(R, C, 0)

    def time(n):
        x = torch.randn((n, C), device="cuda").to(torch.bfloat16)
        y = torch.empty((n, R), device="cuda")
        best = 1e9
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(40):
                L.gemm_small_batch(x, n, y)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b) / 40 * 1e3)
        return best

    t4, t8 = time(4), time(8)
    print(f"{R} x {C}: {t4:.1f} us at four columns, {t8:.1f} at eight")
    assert t8 < 1.5 * t4
    L.release()
