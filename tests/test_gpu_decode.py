"""Full decode: the whole-row kernel against the oracle's rows and against the
direct kernel (an output that is not 16-byte aligned takes it), bit for bit, at
the edges of its tiles."""
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


# Rows of one block, of fewer and more blocks than the CTA has threads, of two
# buffers and of one, and (C = 65536) too long for shared memory.
@pytest.mark.parametrize("R,C,n_out", [(1, 8, 0), (70, 8, 2), (37, 64, 4), (650, 1000, 0), (33, 4096, 4),
                                       (5, 4104, 16), (9, 13000, 3), (3, 40000, 0), (2, 65536, 1)])
def test_rows_match_oracle_and_direct_kernel(R, C, n_out):
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
    W = torch.full((R, C), 7.0, device="cuda")
    layer.decode_weights(W)
    odd = torch.full((R * C + 1,), 7.0, device="cuda")
    layer.decode_weights(odd[1:])  # 4 bytes past a 16-byte boundary
    part = torch.full((R, C), 7.0, device="cuda")
    r0 = R // 3
    layer.decode_rows(r0, R - r0, part)
    torch.cuda.synchronize()
    Wh = W.cpu().numpy()
    assert np.array_equal(Wh.view(np.uint32), odd[1:].cpu().numpy().reshape(R, C).view(np.uint32))
    assert np.array_equal(Wh[r0:], part.cpu().numpy()[:R - r0])
    s = O.Sched(RUNGS, THETA, -1, 0.1)
    ref = O.Tensor(R, C, a, rho).synth_rows(s, 0, 77, 0, R)
    if n_out:
        ref = ref.copy()
        ref[:, cols] = vals.astype(np.float32)
    assert np.array_equal(Wh, ref)
    assert layer.device_error() == 0
    layer.release()
