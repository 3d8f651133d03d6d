"""Activations that are not finite in the tensor-core batch products: the same
infinities and NaNs as the rows' own products give (many infinities of one
sign, weights that are zero, outlier columns, columns past the first chunk,
superblocks cut between CTAs, tensors of several rungs and of one), and at no
more than a small multiple of a finite call's time."""
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


def _layer(R, C, rungs, theta, n_out, seed, weights=True):
    from paper_2609_38477_gb300 import build

    build.build()
    from paper_2609_38477_gb300 import seedq as Q

    rng = np.random.default_rng(seed)
    a = np.exp(rng.normal(0, 1, C)).astype(np.float32)
    rho = np.exp(rng.normal(0, 0.7, R)).astype(np.float32)
    cols = vals = dev = None
    if n_out:
        cols = rng.choice(C, n_out, replace=False).astype(np.int32)
        vals = rng.normal(0, 8, (R, n_out)).astype(np.float16)
        dev = torch.from_numpy(vals.view(np.int16)).cuda()
    L = Q.Layer(R, C, a, rho, rungs, theta, -1, 0.1, 0, cols, dev, max_batch=16)
    nbytes = Q.stream_bytes_required(L.stream_bits)
    buf = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    L.synth_stream(seed, buf, nbytes)
    L.bind_stream(buf, L.stream_bits, nbytes)
    Wm = None
    if weights:
        Wm = O.Tensor(R, C, a, rho).synth_rows(O.Sched(rungs, theta, -1, 0.1), 0, seed, 0, R).astype(np.float64)
        if n_out:
            Wm[:, cols] = vals.astype(np.float64)
    return L, Wm, cols


@pytest.mark.parametrize("R,C,n,J,n_out", [(1, 8, 5, 7, 0), (129, 584, 16, 7, 4), (300, 3080, 8, 7, 3),
                                           (200, 6152, 13, 1, 0), (513, 1160, 9, 7, 16)])
def test_outputs_follow_the_rows_products(R, C, n, J, n_out):
    L, Wm, cols = _layer(R, C, RUNGS[-J:], THETA[:J - 1], n_out, R + C)
    rng = np.random.default_rng(n)
    x = rng.normal(0, 1, (n, C)).astype(np.float32)
    x[0] = np.inf                                     # every column
    x[1] = np.where(rng.random(C) < 0.5, np.inf, -np.inf)
    x[2, C - 1] = np.nan                              # (a NaN and infinities)
    x[2, : C // 2] = np.inf
    x[3, C - 1] = -np.inf
    # The sign of one row's weights: that row's products are all plus infinity.
    x[4] = np.where(Wm[R // 2] > 0, np.inf, -np.inf)
    if n > 5 and n_out:
        x[5, cols[0]] = np.inf                        # in a stored column alone
    bits = W.to_bf16_bits(np.nan_to_num(x, nan=0.0, posinf=0.0, neginf=0.0).ravel()).reshape(n, C)
    bits[np.isposinf(x)], bits[np.isneginf(x)], bits[np.isnan(x)] = 0x7F80, 0xFF80, 0x7FC1
    xd = torch.from_numpy(bits.view(np.int16)).cuda()
    y = torch.zeros((n, R), device="cuda")
    L.gemm_small_batch(xd, n, y)
    torch.cuda.synchronize()
    y = y.cpu().numpy()
    xb = W.bf16_bits_to_f32(bits).astype(np.float64)
    with np.errstate(invalid="ignore"):
        ref = np.stack([(xb[b] * Wm).sum(1) for b in range(n)])
    bad = ~np.isfinite(ref)
    assert bad[:5].all()
    assert np.array_equal(np.isnan(y), np.isnan(ref))
    assert np.array_equal(y[np.isinf(ref)], ref[np.isinf(ref)])
    ok = ~bad
    # (The bound of tests/test_gpu_gemm.py.)
    mag = np.abs(np.where(np.isfinite(xb), xb, 0.0)) @ np.abs(Wm).T
    assert np.all(np.abs(y - np.where(ok, ref, 0.0))[ok] <= 2e-5 * mag[ok])
    assert L.device_error() == 0
    L.release()


@pytest.mark.parametrize("n", [5, 16])
@pytest.mark.parametrize("bad", ["one nan", "one infinity", "all nan", "all infinite"])
def test_time_of_a_call(n, bad):
    """4096 x 4096: at most five times a finite call (the infinities of an
    entry cost a look at its activations and a few weights a row)."""
    L, _, _ = _layer(4096, 4096, RUNGS, THETA, 0, 9, weights=False)
    fin = torch.randn((n, 4096), device="cuda").to(torch.bfloat16)
    x = fin.clone()
    if bad.startswith("one"):
        x[1, 100] = float(bad[4:7])
    elif bad == "all nan":
        x[:] = float("nan")
    else:
        x[:] = float("inf")
    y = torch.empty((n, 4096), device="cuda")

    def time(v):
        best = 1e9
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(4):
                L.gemm_small_batch(v, n, y)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        return best

    assert time(x) < 5 * time(fin)
    L.release()


@pytest.mark.parametrize("n", [7, 16])
def test_several_tensors_and_sets(n):
    """One launch over three tensors and a layer set of them, whole and cut
    superblocks: the outputs of each tensor's own call, NaN for NaN."""
    from paper_2609_38477_gb300 import seedq as Q

    ts = [_layer(R, C, RUNGS, THETA, n_out, seed, weights=False) for R, C, n_out, seed in
          ((300, 520, 2, 3), (4100, 64, 0, 4), (40, 2056, 0, 5))]
    xs = []
    for i, (L, _, _) in enumerate(ts):
        x = torch.randn((n, L.cols), generator=torch.Generator(device="cuda").manual_seed(i), device="cuda").to(torch.bfloat16)
        x[1, 7], x[2, :9], x[4, L.cols - 1], x[n - 1, 3] = float("inf"), float("-inf"), float("nan"), float("-inf")
        xs.append(x)
    own = []
    for (L, _, _), x in zip(ts, xs):
        y = torch.zeros((n, L.rows), device="cuda")
        L.gemm_small_batch(x, n, y)
        own.append(y)
    multi = [torch.zeros_like(y) for y in own]
    Q.gemm_multi([t[0] for t in ts], xs, n, multi)
    S = Q.LayerSet([t[0] for t in ts])
    Y = torch.zeros(n * sum(t[0].rows for t in ts), device="cuda")
    S.gemm(torch.cat([x.flatten() for x in xs]), n, Y)
    torch.cuda.synchronize()
    for i, y in enumerate(own):
        # (Each within the bound of tests/test_gpu_gemm.py of the exact product.)
        Wm = torch.empty((ts[i][0].rows, ts[i][0].cols), device="cuda")
        ts[i][0].decode_weights(Wm)
        mag = torch.nan_to_num(xs[i].double(), 0.0, 0.0, 0.0).abs() @ Wm.double().abs().T
        part = Y[n * int(S.row_offsets[i]):n * int(S.row_offsets[i + 1])].view(n, -1)
        for other in (multi[i], part):
            bad = ~torch.isfinite(y)
            assert bad[[1, 2, 4, n - 1]].all() and not bad[[0, 3]].any()
            assert torch.equal(torch.isnan(y), torch.isnan(other))
            assert torch.equal(y[torch.isinf(y)], other[torch.isinf(y)])
            assert ((y - other).double().abs() <= 4e-5 * mag)[~bad].all()
    S.release()
