"""The seed search among other calls is not slower than evaluating every seed,
where the screening has little to save: few seeds, few blocks, and weights too
small or too large for any exponent, which leave every seed in the race.  (The
exhaustive kernels run when no memory is left, see test_gpu_encode_routes.)"""
import os
import sys
import time

import pytest

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))

from test_gpu_encode_routes import _buffers, _lib, no_memory_left  # noqa: E402

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _both(S, k, n, scale):
    Q = _lib()
    w = torch.randn((n, 8), device="cuda") * scale
    out = _buffers(n)

    def call_time():
        Q.encode_blocks(S, k, w, n, *out)
        best = 1e9
        for _ in range(5):
            torch.cuda.synchronize()
            t = time.perf_counter()
            for _ in range(30):
                Q.encode_blocks(S, k, w, n, *out)
            torch.cuda.synchronize()
            best = min(best, (time.perf_counter() - t) / 30 * 1e6)
        return best

    fast = call_time()
    with no_memory_left():
        every = call_time()
    print(f"({S}, {k}) x {n}, {scale}: {fast:.0f} us, every seed {every:.0f}")
    return fast, every


@pytest.mark.parametrize("S,k,n", [(8, 2, 100), (8, 3, 2000), (8, 4, 20), (8, 4, 1000), (8, 5, 300), (8, 6, 100),
                                   (10, 2, 1), (10, 3, 20), (12, 2, 100)])
def test_weights_of_a_model(S, k, n):
    fast, every = _both(S, k, n, 0.02)
    assert fast < 1.2 * every


@pytest.mark.parametrize("scale", [1e-4, 1e6])
@pytest.mark.parametrize("S,k,n", [(8, 4, 4000), (8, 6, 2048), (10, 4, 1000), (12, 3, 300)])
def test_weights_out_of_range(S, k, n, scale):
    fast, every = _both(S, k, n, scale)
    assert fast < 1.75 * every
