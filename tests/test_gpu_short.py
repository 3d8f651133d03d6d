"""Rounds too short to give every warp a whole stage (n = 1 to 4): the stage
width follows the round.  Sizes around the widths at which it changes (one
column, two, 12 warps of two or three, the line to the full-width kernel),
ragged rows, outlier columns, several tensors and layer sets, against fp64
products of the oracle's weights.

Tolerance, from the arithmetic: a row of C/8 blocks takes C/8 additions of
block sums (each of at most 9 rounded steps) over stages, warps and CTAs, so
(C/8 + 9 + 14) 2^-24 of the sum of magnitudes bounds it: below 2e-4 for every
row here; sums of rounding errors of both signs stay far below the bound."""
import os
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))

from test_gpu_gemm import _tensor, _x  # noqa: E402

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _check(y, Wm, x):
    tol = (Wm.shape[1] / 8 + 23) * 2.0 ** -24
    assert np.all(np.abs(y.astype(np.float64) - x @ Wm.T) <= tol * (np.abs(x) @ np.abs(Wm).T))


@pytest.mark.parametrize("n", [1, 2, 3, 4])
@pytest.mark.parametrize("R,C,spread,n_out", [
    (1, 8, 0, 0), (32, 16, 0, 0), (33, 1016, 0.5, 2), (64, 11008, 0.5, 0), (1024, 1024, 0.5, 4),
    (1000, 1096, 1.0, 0), (4096, 512, 0.5, 0), (1216, 5176, 0.7, 0), (1216, 5184, 0, 0), (1216, 2008, 0.5, 0), (1216, 2016, 0, 2),
    (1216, 1432, 0.5, 0), (1216, 1440, 0.5, 0)])
def test_short_rounds(R, C, spread, n_out, n):
    _, L, Wm = _tensor(R, C, spread, n_out, R + C)
    xd, x = _x(np.random.default_rng(n), n, C)
    y = torch.full((n, R), 7.0, device="cuda")
    again = torch.full((n, R), 7.0, device="cuda")
    L.gemm_small_batch(xd, n, y)
    L.gemm_small_batch(xd, n, again)
    torch.cuda.synchronize()
    _check(y.cpu().numpy(), Wm, x)
    assert torch.equal(y, again) and L.device_error() == 0
    L.release()


@pytest.mark.parametrize("n", [1, 4])
def test_several_tensors_and_sets(n):
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
