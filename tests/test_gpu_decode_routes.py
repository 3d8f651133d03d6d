"""Full decode: the whole-row kernel at sizes that it takes (rows of two buffers
and of one, several tiles per CTA so that its buffers and stages come round
again, a last tile that is not full, single rows), against the oracle's rows and
the direct kernel (taken for an output 4 bytes past a 16-byte boundary), bit for
bit; and that a call is not slower than the direct kernel where the rows are
few or short."""
import os
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
sys.path.insert(0, os.path.join(ROOT, "oracle"))

import oracle as O  # noqa: E402

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

RUNGS = [(8, 2), (8, 3), (10, 3), (12, 3), (14, 4), (16, 5), (16, 6)]
THETA = [0.2, 0.4, 0.7, 1.1, 1.9, 3.5]


def _layer(R, C, n_out):
    from paper_2609_38477_gb300 import build

    build.build()
    from paper_2609_38477_gb300 import seedq as Q

    rng = np.random.default_rng(R * 100003 + C)
    a = np.exp(rng.normal(0, 1, C)).astype(np.float32)
    rho = np.exp(rng.normal(0, 0.7, R)).astype(np.float32)
    cols = vals = dev = None
    if n_out:
        cols = rng.choice(C, n_out, replace=False).astype(np.int32)
        vals = rng.normal(0, 8, (R, n_out)).astype(np.float16)
        dev = torch.from_numpy(vals.view(np.int16)).cuda()
    layer = Q.Layer(R, C, a, rho, RUNGS, THETA, -1, 0.1, 0, cols, dev, max_batch=1)
    nbytes = Q.stream_bytes_required(layer.stream_bits)
    buf = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    layer.synth_stream(77, buf, nbytes)
    layer.bind_stream(buf, layer.stream_bits, nbytes)
    return layer, a, rho, cols, vals


# Two buffers up to 15384 columns, one up to 22400; 4104 columns give tiles of
# five rows, so 6003 rows are eight tiles for most CTAs and a last one of three.
@pytest.mark.parametrize("R,C,n_out", [(700, 20000, 3), (610, 15392, 0), (157, 22400, 1), (500, 15384, 2),
                                       (6003, 4104, 4), (5003, 520, 2), (4099, 1000, 16), (20003, 264, 1)])
def test_whole_rows(R, C, n_out):
    layer, a, rho, cols, vals = _layer(R, C, n_out)
    W = torch.full((R, C), 7.0, device="cuda")
    layer.decode_weights(W)
    odd = torch.full((R * C + 1,), 7.0, device="cuda")
    layer.decode_weights(odd[1:])
    assert torch.equal(W.view(torch.int32).flatten(), odd[1:].view(torch.int32))
    r0 = R // 7
    part = torch.full((R - r0, C), 7.0, device="cuda")
    layer.decode_rows(r0, R - r0, part)
    assert torch.equal(part, W[r0:])
    s = O.Sched(RUNGS, THETA, -1, 0.1)
    T = O.Tensor(R, C, a, rho)
    for first in {0, R // 2, max(0, R - 150)}:
        n = min(150, R - first)
        ref = T.synth_rows(s, 0, 77, first, n).copy()
        if n_out:
            ref[:, cols] = vals[first:first + n].astype(np.float32)
        assert np.array_equal(W[first:first + n].cpu().numpy(), ref)
    assert layer.device_error() == 0
    layer.release()


@pytest.mark.parametrize("R,C,n_out", [(1, 16000, 0), (8, 22400, 0), (33, 11008, 4), (4096, 64, 0), (8192, 128, 2),
                                       (2048, 512, 0), (400, 11008, 0)])
def test_not_slower_than_the_direct_kernel(R, C, n_out):
    layer = _layer(R, C, n_out)[0]
    flat = torch.empty(R * C + 1, device="cuda")

    def time(W):
        layer.decode_weights(W)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            for _ in range(20):
                layer.decode_weights(W)
        best = 1e9
        for _ in range(9):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            g.replay()
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b) / 20 * 1e3)
        return best

    whole, direct = time(flat[:-1]), time(flat[1:])
    print(f"{R} x {C}, {n_out} outliers: {whole:.1f} us, direct kernel {direct:.1f}")
    assert whole < 1.1 * direct + 0.2
    layer.release()
