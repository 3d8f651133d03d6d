"""Blocks built from every seed of a width in turn (as tests/test_gpu_screen.py
builds them): the fields the search returns reproduce the block exactly, and a
sample of those that are not the planted seed's, and of those that are, equals
the oracle's search, so that a smaller seed with zero error is not missed."""
import os
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
sys.path.insert(0, os.path.join(ROOT, "oracle"))
sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))

import oracle as O  # noqa: E402
from test_gpu_screen import _encode  # noqa: E402

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,k", [(8, 2), (8, 6), (10, 3), (12, 2), (12, 3), (12, 4), (12, 5), (12, 6), (16, 4)])
def test_fields_of_planted_blocks(S, k):
    rng = np.random.default_rng(7 * S + k)
    taps = O.find_taps(S)
    seeds = np.arange(1, 1 << S) if S < 16 else np.arange(1, 1 << S, 13)
    # Small mantissas among them, which many seeds reproduce.
    t = [rng.integers(-8, 8, k) if i % 2 else rng.integers(-1, 2, k) for i in range(len(seeds))]
    w = np.stack([O.reconstruct_block(S, k, taps, int(s), -6, v.tolist()) for s, v in zip(seeds, t)])
    gs, gE, gt, gerr = _encode(S, k, w)
    zero = gerr == 0.0
    plain = zero & (gs <= seeds)
    assert plain.mean() > 0.9
    for b in np.nonzero(zero)[0]:
        back = O.reconstruct_block(S, k, taps, int(gs[b]), int(gE[b]), gt[b, :k].tolist())
        assert np.array_equal(back.astype(np.float32), w[b].astype(np.float32)), int(seeds[b])
    take = 12 if S < 16 else 3
    for kind in (plain & (gs == seeds), plain & (gs < seeds)):
        at = np.nonzero(kind)[0]
        for b in rng.permutation(at)[:take]:
            seed, E, v, err = O.encode_block(S, k, taps, w[b].astype(np.float32).astype(np.float64))
            assert (int(gs[b]), int(gE[b]), list(gt[b, :k]), gerr[b]) == (seed, E, list(v), err), int(seeds[b])
