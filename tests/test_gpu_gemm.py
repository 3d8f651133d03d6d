"""The tensor-core batch products (n = 5 to 16) against fp64 products of the
oracle's weights, at the edges of their tiles: rows around 8, 16, 32 and 128,
columns that are not whole steps, stages or windows, rows whose rungs differ,
outlier columns, several tensors a launch and layer sets; and activations that
are infinite or NaN, which must reach exactly the outputs fp32 products and
sums would give them.

Tolerance, from the arithmetic: products are exact; a sum of four block columns
takes 8 tensor-core additions that may truncate (2^-23 each), then there are at
most 6 rounding additions per stage, one per stage, three parts and one per CTA
(2^-24 each): below 2e-5 of the sum of magnitudes for any row here."""
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
TOL = 2e-5


def _tensor(R, C, spread, n_out, seed):
    from paper_2609_38477_gb300 import build

    build.build()
    from paper_2609_38477_gb300 import seedq as Q

    rng = np.random.default_rng(seed)
    a = np.exp(rng.normal(0, 1, C)).astype(np.float32)
    rho = np.exp(rng.normal(0, spread, R)).astype(np.float32) if spread else None
    cols = vals = dev = None
    if n_out:
        cols = rng.choice(C, n_out, replace=False).astype(np.int32)
        vals = rng.normal(0, 8, (R, n_out)).astype(np.float16)
        dev = torch.from_numpy(vals.view(np.int16)).cuda()
    L = Q.Layer(R, C, a, rho, RUNGS, THETA, -1, 0.1, 0, cols, dev, max_batch=16)
    nbytes = Q.stream_bytes_required(L.stream_bits)
    buf = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    L.synth_stream(seed + 5, buf, nbytes)
    L.bind_stream(buf, L.stream_bits, nbytes)
    Wm = O.Tensor(R, C, a, rho).synth_rows(O.Sched(RUNGS, THETA, -1, 0.1), 0, seed + 5, 0, R).astype(np.float64)
    if n_out:
        Wm[:, cols] = vals.astype(np.float64)
    return Q, L, Wm


def _x(rng, n, C):
    b = W.to_bf16_bits(rng.normal(0, 1, (n, C)).astype(np.float32).ravel()).reshape(n, C)
    return torch.from_numpy(b.view(np.int16)).cuda(), W.bf16_bits_to_f32(b).astype(np.float64)


def _check(y, Wm, x):
    assert np.all(np.abs(y.astype(np.float64) - x @ Wm.T) <= TOL * (np.abs(x) @ np.abs(Wm).T))


@pytest.mark.parametrize("R,C,n,spread,n_out", [
    (1, 8, 5, 0, 0), (7, 24, 16, 0.5, 2), (31, 40, 8, 0.5, 0), (33, 200, 6, 2.0, 0), (129, 584, 16, 0.7, 4),
    (160, 1016, 7, 0, 0), (500, 2072, 13, 0.5, 4), (513, 1160, 8, 1.5, 0), (96, 11008, 9, 0.5, 0),
    (3000, 136, 16, 0.5, 0)])
def test_batch_products(R, C, n, spread, n_out):
    Q, L, Wm = _tensor(R, C, spread, n_out, R + C)
    xd, x = _x(np.random.default_rng(n), n, C)
    y = torch.full((n, R), 7.0, device="cuda")
    again = torch.full((n, R), 7.0, device="cuda")
    L.gemm_small_batch(xd, n, y)
    L.gemm_small_batch(xd, n, again)
    torch.cuda.synchronize()
    _check(y.cpu().numpy(), Wm, x)
    assert torch.equal(y, again) and L.device_error() == 0
    L.release()


@pytest.mark.parametrize("n", [5, 16])
def test_several_tensors_and_sets(n):
    """One launch over three tensors and the same through a layer set."""
    ts = [_tensor(*s) for s in ((200, 520, 0.5, 0, 3), (130, 1032, 0, 3, 4), (40, 64, 1.0, 0, 5))]
    Q = ts[0][0]
    rng = np.random.default_rng(n)
    xs = [_x(rng, n, t[2].shape[1]) for t in ts]
    ys = [torch.zeros((n, t[2].shape[0]), device="cuda") for t in ts]
    Q.gemm_multi([t[1] for t in ts], [x[0] for x in xs], n, ys)
    S = Q.LayerSet([t[1] for t in ts])
    Y = torch.zeros(n * sum(t[2].shape[0] for t in ts), device="cuda")
    S.gemm(torch.cat([x[0].flatten() for x in xs]), n, Y)
    torch.cuda.synchronize()
    for i, (t, x, y) in enumerate(zip(ts, xs, ys)):
        _check(y.cpu().numpy(), t[2], x[1])
        part = Y[n * int(S.row_offsets[i]):n * int(S.row_offsets[i + 1])].view(n, -1)
        assert torch.equal(part, y)
    S.release()


@pytest.mark.parametrize("n", [6, 16])
def test_infinities_and_nans(n):
    R, C = 300, 520
    Q, L, Wm = _tensor(R, C, 1.0, 2, 11)
    xd, _ = _x(np.random.default_rng(n), n, C)
    bits = xd.cpu().numpy().view(np.uint16).copy()
    bits[0, 17] = 0x7F80                        # one infinity
    bits[1, 5], bits[1, 400] = 0x7F80, 0xFF80   # two of opposite sign
    bits[2, 100] = 0x7FC0                       # a NaN
    xd = torch.from_numpy(bits.view(np.int16)).cuda()
    y = torch.zeros((n, R), device="cuda")
    L.gemm_small_batch(xd, n, y)
    torch.cuda.synchronize()
    y = y.cpu().numpy()
    x = W.bf16_bits_to_f32(bits).astype(np.float64)
    with np.errstate(invalid="ignore"):
        ref = np.stack([(x[b] * Wm).sum(1) for b in range(n)])
    for b in range(3):
        assert np.array_equal(np.isnan(y[b]), np.isnan(ref[b]))
        ok = ~np.isnan(ref[b])
        assert np.array_equal(y[b][ok], ref[b][ok])  # infinities, sign and all
    _check(y[3:], Wm, x[3:])
    L.release()
