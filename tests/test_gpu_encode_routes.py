"""The two routes of the seed search give the same bits: the screened search,
and the exhaustive kernels, which a call takes for which the device has no
memory left.  That is brought about by a memory pool of this process's own,
small and full, in the place of the device's default one."""
import contextlib
import ctypes as C
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

OUT_OF_MEMORY = 2


class _Props(C.Structure):  # CUmemPoolProps
    _fields_ = [("alloc_type", C.c_int), ("handle_types", C.c_int), ("location_type", C.c_int),
                ("location_id", C.c_int), ("security", C.c_void_p), ("max_size", C.c_size_t),
                ("usage", C.c_ushort), ("reserved", C.c_ubyte * 54)]


@contextlib.contextmanager
def no_memory_left():
    """The current device's stream-ordered allocations come from a full pool."""
    cu = C.CDLL("libcuda.so.1")

    def call(name, *args):
        r = getattr(cu, name)(*args)
        assert r == 0, (name, r)

    torch.cuda.synchronize()
    device, pool, default = torch.cuda.current_device(), C.c_void_p(), C.c_void_p()
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    call("cuDeviceGetDefaultMemPool", C.byref(default), device)
    props = _Props(alloc_type=1, location_type=1, location_id=device, max_size=32 << 20)
    call("cuMemPoolCreate", C.byref(pool), C.byref(props))
    held = []
    try:
        for size in (4 << 20, 64 << 10, 512):
            for _ in range(4096):
                p = C.c_uint64()
                r = cu.cuMemAllocFromPoolAsync(C.byref(p), C.c_size_t(size), pool, stream)
                if r:
                    assert r == OUT_OF_MEMORY
                    break
                held.append(p)
            else:
                raise AssertionError("the pool has no limit")
        call("cuDeviceSetMemPool", device, pool)
        yield
    finally:
        cu.cuDeviceSetMemPool(device, default)
        for p in held:
            cu.cuMemFreeAsync(p, stream)
        torch.cuda.synchronize()
        cu.cuMemPoolDestroy(pool)


def _lib():
    from paper_2609_38477_gb300 import build

    build.build()
    from paper_2609_38477_gb300 import seedq as Q

    return Q


def _buffers(n):
    return (torch.full((n,), 7, dtype=torch.int32, device="cuda"), torch.full((n,), 7, dtype=torch.int8, device="cuda"),
            torch.full((n, 6), 7, dtype=torch.int8, device="cuda"), torch.full((n,), 7.0, dtype=torch.float64, device="cuda"))


def _same(a, b):
    return all(torch.equal(x, y) for x, y in zip(a[:3], b[:3])) and torch.equal(a[3].view(torch.int64), b[3].view(torch.int64))


def _time(f):
    best = 1e9
    f()
    for _ in range(7):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        f()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3)
    return best


@pytest.mark.parametrize("S,n", [(8, 40), (10, 70), (12, 130), (14, 9), (16, 3)])
@pytest.mark.parametrize("k", [2, 3, 4, 5, 6])
def test_lists_of_blocks(S, k, n):
    """Both routes bit for bit, the scales of weights mixed; the first blocks also
    against the oracle."""
    Q = _lib()
    rng = np.random.default_rng(S * 10 + k)
    w = rng.normal(0, 1, (n, 8)) * 10.0 ** rng.uniform(-3, 1, (n, 1))
    w[0] *= 1e-5
    w[1] *= 1e5
    w = w.astype(np.float32)
    wd = torch.from_numpy(w).cuda()
    screened, every = _buffers(n), _buffers(n)
    Q.encode_blocks(S, k, wd, n, *screened)
    with no_memory_left():
        Q.encode_blocks(S, k, wd, n, *every)
        torch.cuda.synchronize()
    assert _same(screened, every)
    if S <= 12:
        taps = O.find_taps(S)
        for b in range(min(n, 6)):
            seed, E, t, err = O.encode_block(S, k, taps, w[b].astype(np.float64))
            assert (int(every[0][b]), int(every[1][b]), every[2][b, :k].tolist(), float(every[3][b])) == (seed, E, list(t), err)


@pytest.mark.parametrize("R,C_,n_out", [(5, 104, 2), (9, 256, 0)])
def test_layer_of_mixed_rungs(R, C_, n_out):
    Q = _lib()
    rng = np.random.default_rng(R)
    a = np.exp(rng.normal(0, 1, C_)).astype(np.float32)
    rho = np.exp(rng.normal(0, 0.7, R)).astype(np.float32)
    cols = vals = None
    if n_out:
        cols = rng.choice(C_, n_out, replace=False).astype(np.int32)
        vals = torch.zeros((R, n_out), dtype=torch.int16, device="cuda")
    L = Q.Layer(R, C_, a, rho, [(8, 2), (10, 3), (12, 3), (14, 4), (12, 5), (12, 6)], [0.3, 0.6, 0.9, 1.4, 2.5], -1, 0.1, 0,
                cols, vals, max_batch=1)
    W = torch.from_numpy(rng.normal(0, 0.02, (R, C_)).astype(np.float32)).cuda()
    n = R * C_ // 8
    screened, every = _buffers(n), _buffers(n)
    L.encode(W, *screened)
    with no_memory_left():
        L.encode(W, *every)
        torch.cuda.synchronize()
    assert len(set(L.rung_map().flatten().tolist())) > 3
    assert _same(screened, every)
    L.release()


def test_the_exhaustive_route_is_taken():
    """(By its time: at (12, 6) it takes more than ten times as long.)"""
    Q = _lib()
    w = torch.randn((200, 8), device="cuda") * 0.02
    out = _buffers(200)
    call = lambda: Q.encode_blocks(12, 6, w, 200, *out)
    fast = _time(call)
    with no_memory_left():
        slow = _time(call)
    assert slow > 4 * fast
