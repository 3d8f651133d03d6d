"""The work a user of this framework has it do, as cases that can be timed.

Every case goes through the public binding (paper_2609_38477_gb300.seedq):

* products  y = W_hat x over compressed tensors, batch 1 to 16: one tensor,
  the seven tensors of a decoder layer in one call, a whole model as a layer
  set;
* decoding  the full weight matrix of a tensor;
* encoding  the exhaustive seed search over a list of blocks or a prepared
  layer, and the packing of the stream;
* importance and outlier columns of a whole FP16 checkpoint, and the rung
  allocation over a set of tensors.

`listed()` holds the cases, `draw(rng)` gives more of the same ranges,
`prepare` makes what a program has in hand before the call, `run` is the call,
`work` is what it cannot do without and `exact` is its result in 64 bits from
plain numpy and torch.
"""
from __future__ import annotations

import numpy as np
import torch

from paper_2609_38477_gb300 import seedq as Q
from paper_2609_38477_gb300 import workload_gpu as G
from paper_2609_38477_gb300 import workloads as W

# Rung schedules as a model file carries them, with thresholds in units of the
# mean importance: the stored schedules of the Llama-2-7B-shaped layer set at
# 4.0 and at 3.0 bits per weight.  At 3.0 the floor coincides with the lowest
# threshold, so many blocks are tied there and the tie pass splits them.
SCHEDULES = {
    "4bpw": dict(
        rungs=[(8, 3), (10, 3), (12, 3), (14, 3), (16, 3), (14, 4), (16, 5), (16, 6)],
        theta=[0.017282761534617958, 0.06184954960515235, 0.2088509158644461, 0.4343936203262455,
               0.9773856457340522, 2.1565541344583607, 6.6520575291750434],
        q=0.10838851810261675, j_tie=-1),
    "3bpw": dict(
        rungs=[(8, 2), (10, 2), (12, 2), (14, 2), (16, 2), (16, 3), (14, 4)],
        theta=[0.08663793571142325, 0.310049831546792, 1.0469630206776868, 2.1776014484660657,
               6.67927977915152, 9.799206518097295],
        q=0.08663793571142325, j_tie=0),
}
# Slopes of the damage hull behind the 4.0 bits-per-weight schedule (allocation).
SLOPES_4BPW = [5.1576, 1.4412, 0.4268, 0.2052, 0.0912, 0.04133333333333333, 0.0134]

# Feedback taps of the stream format (bit i: o_{t+S} takes o_{t+i}).
TAPS = {8: 0x1D, 10: 0x09, 12: 0x53, 14: 0x2B, 16: 0x2D}


def listed():
    return [
        # One small linear layer for one token: the call's own latency.
        dict(name="linear_1k_b1", kind="product", shapes="1024x1024", sched="4bpw", n=1, rho=False,
             outliers=0),
        # An odd-sized projection with stored outlier columns, three sequences.
        dict(name="linear_ragged_b3", kind="product", shapes="1997x2072", sched="3bpw", n=3, rho=True,
             outliers=4),
        # One decoder layer of a 7B model for one token: the token loop of a chat.
        dict(name="layer_7b_b1", kind="product", shapes="llama:4096,4096,11008", sched="4bpw", n=1,
             rho=False, outliers=0),
        # The same layer at the low rate, four sequences decoded together.
        dict(name="layer_7b_3bpw_b4", kind="product", shapes="llama:4096,4096,11008", sched="3bpw", n=4,
             rho=True, outliers=0),
        # The same layer at the full decode batch.
        dict(name="layer_7b_b16", kind="product", shapes="llama:4096,4096,11008", sched="4bpw", n=16,
             rho=False, outliers=0),
        # Layers of an 8B model and its vocabulary head behind one launch, one token.
        dict(name="set_8b_b1", kind="set", dims="4096,1024,14336,128256", layers=4, sched="4bpw", n=1,
             rho=False),
        # Two layers of a 70B model behind one launch, eight sequences.
        dict(name="set_70b_3bpw_b8", kind="set", dims="8192,1024,28672,0", layers=2, sched="3bpw", n=8,
             rho=True),
        # A tensor decoded in full, to hand it to a program that wants plain weights.
        dict(name="decode_7b_down", kind="decode", R=4096, C=11008, sched="4bpw", rho=True, outliers=4),
        # Compression of a model: the seed search of a list of blocks at one rung.
        dict(name="encode_blocks_16_3", kind="encode_blocks", S=16, k=3, blocks=32768),
        # Compression of a layer: every block at its planned rung, then the stream.
        dict(name="encode_layer", kind="encode_layer", R=256, C=1024, sched="4bpw", rho=True, outliers=4),
        # Before compression: importance and outlier columns of a 7B checkpoint.
        dict(name="importance_7b", kind="importance", layers=32, d=4096, heads=32, kv=32, hd=128, ff=11008,
             vocab=32000),
        # Before compression: the rung schedule of a layer's tensors.
        dict(name="allocate_7b", kind="allocate", dims="4096,4096,11008", layers=1),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["product", "product", "layer", "layer", "set", "decode", "encode_blocks",
                       "encode_layer", "importance", "allocate"])
    sched = rng.choice(["4bpw", "3bpw"])
    if kind == "product":
        R, C = _log(rng, 33, 11008), 8 * _log(rng, 16, 1376)
        return dict(kind="product", shapes=f"{R}x{C}", sched=sched, n=rng.randint(1, 16),
                    rho=rng.random() < 0.5, outliers=rng.choice([0, 0, 4]))
    if kind == "layer":
        d = 128 * rng.randint(8, 32)
        return dict(kind="product", shapes=f"llama:{d},{rng.choice([d, d // 4])},{8 * rng.randint(d // 4, 11008 // 8)}",
                    sched=sched, n=rng.choice([1, 1, 2, 4, 7, 8, 13, 16]), rho=rng.random() < 0.5,
                    outliers=0)
    if kind == "set":
        d = 256 * rng.randint(4, 16)
        return dict(kind="set", dims=f"{d},{d // 4},{8 * rng.randint(d // 4, 11008 // 8)},{rng.randint(1000, 32000)}",
                    layers=rng.randint(1, 4), sched=sched, n=rng.choice([1, 1, 2, 3, 4, 8, 16]),
                    rho=rng.random() < 0.5)
    if kind == "decode":
        return dict(kind="decode", R=_log(rng, 33, 4096), C=8 * _log(rng, 16, 1376), sched=sched,
                    rho=rng.random() < 0.5, outliers=rng.choice([0, 4]))
    if kind == "encode_blocks":
        S, k = rng.choice([8, 10, 12, 14, 16]), rng.randint(2, 6)
        return dict(kind="encode_blocks", S=S, k=k, blocks=_log(rng, 5, 6000 if S == 16 else 12000))
    if kind == "encode_layer":
        return dict(kind="encode_layer", R=_log(rng, 5, 64), C=8 * _log(rng, 16, 256), sched=sched,
                    rho=rng.random() < 0.5, outliers=rng.choice([0, 4]))
    if kind == "importance":
        kv, rep, hd = rng.choice([2, 4, 8]), rng.choice([1, 2, 4]), rng.choice([64, 128])
        return dict(kind="importance", layers=rng.randint(1, 8), d=32 * rng.randint(8, 128),
                    heads=kv * rep, kv=kv, hd=hd, ff=32 * rng.randint(16, 344), vocab=rng.randint(300, 32000))
    d = 128 * rng.randint(4, 32)
    return dict(kind="allocate", dims=f"{d},{d // 4},{8 * rng.randint(d // 4, 11008 // 8)}", layers=1)


# ------------------------------------------------------------------ inputs

def _tensors(case):
    """(rows, cols, input group, row factor) of each tensor of a product."""
    rho = bool(case["rho"])
    if case["kind"] == "set":
        d, kv, ff, vocab = (int(v) for v in case["dims"].split(","))
        out = []
        for l in range(case["layers"]):
            out += _layer(d, kv, ff, rho, f"l{l}.")
        return out + ([(vocab, d, "head", False)] if vocab else [])
    s = case["shapes"]
    if s.startswith("llama:"):
        return _layer(*(int(v) for v in s[6:].split(",")), rho, "")
    R, C = (int(v) for v in s.split("x"))
    return [(R, C, "in", rho)]


def _layer(d, kv, ff, rho, p):
    return [(d, d, p + "attn", rho), (kv, d, p + "attn", rho), (kv, d, p + "attn", rho),
            (d, d, p + "o", True), (ff, d, p + "mlp", rho), (ff, d, p + "mlp", rho),
            (d, ff, p + "down", True)]


def _rng(seed, *parts):
    words = [seed & 0xFFFFFFFF, seed >> 32]
    for p in parts:
        words += list(p.encode()) if isinstance(p, str) else [p]
    return np.random.default_rng(words)


def _input_factor(seed, group, C):
    """Input-side importance: squared norm gains, four channels at 100x the mean."""
    r = _rng(seed, "a", group)
    a = np.exp(0.5 * r.standard_normal(C)) ** 2
    a[r.choice(C, 4, replace=False)] = 100.0 * a.mean()
    return a.astype(np.float32)


def _row_factor(seed, i, R):
    return np.exp(0.5 * _rng(seed, "rho", i).standard_normal(R)).astype(np.float32)


def _outliers(seed, i, R, C, count):
    """Columns kept in FP16 and their values (rows x count, binary16 bits)."""
    r = _rng(seed, "out", i)
    cols = np.sort(r.choice(C, count, replace=False)).astype(np.int32)
    vals = (8.0 * r.standard_normal((R, count))).astype(np.float16)
    return cols, vals


def _key(seed, i):
    return int(_rng(seed, "payload", i).integers(1, 1 << 62))


def _activations(seed, group, n, C):
    """n activation vectors of C channels, normal, rounded to bfloat16."""
    g = torch.Generator(device="cuda").manual_seed(int(_rng(seed, "x", group).integers(1, 1 << 62)))
    return torch.randn((n, C), generator=g, device="cuda").to(torch.bfloat16)


class _Plan:
    """The decoder's schedule of one tensor from its factors, in numpy and torch."""

    def __init__(self, R, a, rho, sched):
        nb = a.size // 8
        self.perm = np.argsort(a, kind="stable")
        blocks = a.astype(np.float64)[self.perm].reshape(nb, 8)
        s = np.zeros(nb)
        for i in range(8):
            s = s + blocks[:, i]
        abar = s / 8.0
        self.abar = abar / (np.cumsum(abar)[-1] / nb)
        self.rho = None
        if rho is not None:
            r = rho.astype(np.float64)
            self.rho = r / (np.cumsum(r)[-1] / r.size)
        self.sched = sched
        self.tie_count = 0
        if sched["j_tie"] >= 0:  # half of the tied blocks take the lower rung
            v, tied = sched["theta"][sched["j_tie"]], 0
            for r0 in range(0, R, 4096):
                tied += int((self._imp(r0, min(R, r0 + 4096)) == v).sum())
            self.tie_count = tied // 2

    def _imp(self, r0, r1):
        """Floored importance of the blocks of rows [r0, r1), on the GPU."""
        ab = torch.from_numpy(self.abar).cuda()
        rr = (torch.ones(r1 - r0, dtype=torch.float64, device="cuda") if self.rho is None
              else torch.from_numpy(self.rho[r0:r1]).cuda())
        return torch.clamp(ab[None, :] * rr[:, None], min=self.sched["q"])

    def rungs(self, r0, r1, done):
        """Rung of every block of rows [r0, r1) on the GPU; `done` tied blocks precede."""
        imp = self._imp(r0, r1)
        rung = torch.zeros(imp.shape, dtype=torch.int64, device="cuda")
        for th in self.sched["theta"]:
            rung += imp >= th
        jt = self.sched["j_tie"]
        if jt >= 0:
            tied = imp == self.sched["theta"][jt]
            order = torch.cumsum(tied.flatten().to(torch.int64), 0).view(tied.shape) + done
            rung -= (tied & (order <= self.tie_count)).to(torch.int64)
            done += int(tied.sum())
        return rung, done


def _factors(case, seed, i, t):
    R, C, group, has_rho = t
    return _input_factor(seed, group, C), (_row_factor(seed, i, R) if has_rho else None)


def _prepare_layer(case, seed, i, t, max_batch):
    R, C, group, _ = t
    a, rho = _factors(case, seed, i, t)
    sched = SCHEDULES[case["sched"]]
    plan = _Plan(R, a, rho, sched)
    if not plan.tie_count:
        sched = dict(sched, j_tie=-1)
    count = case.get("outliers", 0)
    cols = vals = None
    if count:
        cols, v = _outliers(seed, i, R, C, count)
        vals = torch.from_numpy(v.view(np.int16)).cuda()
    return Q.Layer(R, C, a, rho, sched["rungs"], sched["theta"], sched["j_tie"], sched["q"], plan.tie_count,
                   cols, vals, max_batch=max_batch)


def _with_stream(layer, key):
    nbytes = Q.stream_bytes_required(layer.stream_bits)
    buf = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    layer.synth_stream(key, buf, nbytes)
    layer.bind_stream(buf, layer.stream_bits, nbytes)
    return layer


def _spec(case, seed):
    return W.ModelSpec("case", case["layers"], case["d"], case["heads"], case["kv"], case["hd"], case["ff"],
                       case["vocab"], seed & 0x7FFFFFFF, "")


def _allocation_tensors(case):
    d, kv, ff = (int(v) for v in case["dims"].split(","))
    out = []
    for l in range(case["layers"]):
        out += _layer(d, kv, ff, False, f"l{l}.")
    return out


def _encoder_weights(seed, shape):
    g = torch.Generator(device="cuda").manual_seed(int(_rng(seed, "w").integers(1, 1 << 62)))
    return torch.randn(shape, generator=g, device="cuda") * 0.02


def prepare(case, seed):
    kind, st = case["kind"], {"case": case}
    if kind in ("product", "set"):
        n, ts = case["n"], _tensors(case)
        st["layers"] = [_with_stream(_prepare_layer(case, seed, i, t, n), _key(seed, i))
                        for i, t in enumerate(ts)]
        xs = {t[2]: _activations(seed, t[2], n, t[1]) for t in ts}
        if kind == "set":
            st["set"] = Q.LayerSet(st["layers"])
            st["x"] = torch.cat([xs[t[2]].flatten() for t in ts])
            st["y"] = torch.empty(n * sum(t[0] for t in ts), dtype=torch.float32, device="cuda")
        else:
            st["x"] = [xs[t[2]] for t in ts]
            st["y"] = [torch.empty((n, t[0]), dtype=torch.float32, device="cuda") for t in ts]
    elif kind == "decode":
        t = (case["R"], case["C"], "in", case["rho"])
        st["layer"] = _with_stream(_prepare_layer(case, seed, 0, t, 1), _key(seed, 0))
        st["W"] = torch.empty((case["R"], case["C"]), dtype=torch.float32, device="cuda")
    elif kind in ("encode_blocks", "encode_layer"):
        if kind == "encode_blocks":
            nblk = case["blocks"]
            st["W"] = _encoder_weights(seed, (nblk, 8))
        else:
            nblk = case["R"] * (case["C"] // 8)
            st["W"] = _encoder_weights(seed, (case["R"], case["C"]))
            t = (case["R"], case["C"], "in", case["rho"])
            st["layer"] = _prepare_layer(case, seed, 0, t, 1)
            # Room for the stream at the highest rate (44 bits a block), whatever the plan spends.
            st["stream"] = torch.empty(Q.stream_bytes_required(44 * nblk), dtype=torch.uint8, device="cuda")
        st["seed"] = torch.empty(nblk, dtype=torch.int32, device="cuda")
        st["E"] = torch.empty(nblk, dtype=torch.int8, device="cuda")
        st["t"] = torch.empty((nblk, 6), dtype=torch.int8, device="cuda")
        st["err"] = torch.empty(nblk, dtype=torch.float64, device="cuda")
    elif kind == "importance":
        spec = _spec(case, seed)
        st["model"] = G.synth_model_device(spec)
        st["out"] = G.importance_buffers(spec)
    else:
        st["factors"] = [(t[0], t[1], *_factors(case, seed, i, t))
                         for i, t in enumerate(_allocation_tensors(case))]
    return st


# -------------------------------------------------------------------- calls

def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "product":
        n = case["n"]
        if len(st["layers"]) > 1:
            Q.gemm_multi(st["layers"], st["x"], n, st["y"])
        elif n == 1:
            st["layers"][0].gemv(st["x"][0], st["y"][0])
        else:
            st["layers"][0].gemm_small_batch(st["x"][0], n, st["y"][0])
        return st["y"]
    if kind == "set":
        st["set"].gemm(st["x"], case["n"], st["y"])
        return st["y"]
    if kind == "decode":
        st["layer"].decode_weights(st["W"])
        return st["W"]
    if kind == "encode_blocks":
        Q.encode_blocks(case["S"], case["k"], st["W"], case["blocks"], st["seed"], st["E"], st["t"], st["err"])
        return {k: st[k] for k in ("seed", "E", "t", "err")}
    if kind == "encode_layer":
        st["layer"].encode(st["W"], st["seed"], st["E"], st["t"], st["err"])
        st["layer"].pack_stream(st["seed"], st["E"], st["t"], st["stream"], st["stream"].numel())
        return {k: st[k] for k in ("seed", "E", "t", "err", "stream")}
    if kind == "importance":
        columns = G.run_importance(st["model"], st["out"])
        return dict(st["out"], outliers=np.asarray(columns, np.int64))
    sched = SCHEDULES["4bpw"]
    theta, j_tie, q, ties, bits = Q.allocate(st["factors"], sched["rungs"], SLOPES_4BPW, 4.0, 0.06)
    return {"theta": theta, "j_tie": j_tie, "q": q, "ties": ties, "bits": bits.astype(np.int64)}


# --------------------------------------------------------------------- work

def _mean_k(sched):
    """Coefficients per block the schedule spends on average, to a tenth."""
    return 3.3 if sched == "4bpw" else 2.1


def work(case):
    kind = case["kind"]
    if kind in ("product", "set"):
        ts, n = _tensors(case), case["n"]
        w = sum(t[0] * t[1] for t in ts)
        bits = 4.0 if case["sched"] == "4bpw" else 3.0
        x = {t[2]: t[1] for t in ts} if kind == "product" else {i: t[1] for i, t in enumerate(ts)}
        io = 2 * n * sum(x.values()) + 4 * n * sum(t[0] for t in ts)
        return {"bytes": int(w * bits / 8 + io), "flops": int(w * (2 * _mean_k(case["sched"]) + 2 * n))}
    if kind == "decode":
        w = case["R"] * case["C"]
        bits = 4.0 if case["sched"] == "4bpw" else 3.0
        return {"bytes": int(w * (bits / 8 + 4)), "flops": int(w * 2 * _mean_k(case["sched"]))}
    if kind == "encode_blocks":
        # Every seed's span against every block: 8 products for each of the k directions.
        blocks, seeds, k = case["blocks"], 2 ** case["S"], case["k"]
        return {"bytes": blocks * (32 + 4 + 1 + 6 + 8), "flops": blocks * seeds * k * 18}
    if kind == "encode_layer":
        blocks = case["R"] * (case["C"] // 8)
        bits = 4.0 if case["sched"] == "4bpw" else 3.0
        seeds = 2 ** 14 if case["sched"] == "4bpw" else 2 ** 11
        return {"bytes": int(blocks * (32 + 2 * 11 + 8 + bits)),
                "flops": int(blocks * seeds * _mean_k(case["sched"]) * 18)}
    if kind == "importance":
        s = _spec(case, 0)
        return {"bytes": 2 * s.weights + 8 * s.n_layers * (s.q_dim + s.d_ff + 2 * s.d_model),
                "flops": 4 * s.weights}
    ts = _allocation_tensors(case)
    values = sum(t[1] + (t[0] if t[3] else 0) for t in ts)
    return {"bytes": 4 * values, "flops": 8 * values}


# -------------------------------------------------------------------- exact

def _i64(v):
    """A 64-bit pattern as the signed value torch stores."""
    return v - (1 << 64) if v >= 1 << 63 else v


def _lsr(z, s):
    return (z >> s) & ((1 << (64 - s)) - 1)


def _splitmix(key, idx):
    z = idx + 1
    z = z * _i64(0x9E3779B97F4A7C15) + _i64(key)
    z = (z ^ _lsr(z, 30)) * _i64(0xBF58476D1CE4E5B9)
    z = (z ^ _lsr(z, 27)) * _i64(0x94D049BB133111EB)
    return z ^ _lsr(z, 31)


def _sequences(S):
    """First 64 output bits of the width-S register from every seed."""
    s = np.arange(1 << S, dtype=np.uint64)
    for t in range(S, 64):
        bit = np.zeros_like(s)
        for i in range(S):
            if TAPS[S] >> i & 1:
                bit ^= s >> np.uint64(t - S + i)
        s |= (bit & np.uint64(1)) << np.uint64(t)
    return torch.from_numpy(s.view(np.int64)).cuda()


def _weights64(plan, R, C, key, r0, r1, done, seqs):
    """Rows [r0, r1) of the decoded matrix in permuted column order, fp64."""
    nb = C // 8
    rung, done = plan.rungs(r0, r1, done)
    idx = torch.arange(r0 * nb, r1 * nb, device="cuda", dtype=torch.int64).view(r1 - r0, nb)
    h = _splitmix(key, idx)
    out = torch.zeros((r1 - r0, nb, 8), dtype=torch.float64, device="cuda")
    for j, (S, k) in enumerate(plan.sched["rungs"]):
        sel = rung == j
        hb = h[sel]
        if not hb.numel():
            continue
        seq = seqs[S][1 + _lsr(hb, 32) % ((1 << S) - 1)]
        E = -8 + ((hb >> 24) & 255) % 6
        t = [((hb >> (4 * c)) & 15) - 8 for c in range(k)]
        w = torch.zeros((hb.numel(), 8), dtype=torch.int64, device="cuda")
        for i in range(8):
            for c in range(k):
                w[:, i] += t[c] * (((seq >> (i * k + c)) & ((1 << S) - 1)) - (1 << (S - 1)))
        out[sel] = w.to(torch.float64) * torch.exp2((E - (S - 1)).to(torch.float64))[:, None]
    return out.view(r1 - r0, C), done


def _exact_tensor(case, seed, i, t, x, seqs):
    """y = W_hat x of one tensor (n x R), or W_hat itself when x is None."""
    R, C, _, _ = t
    a, rho = _factors(case, seed, i, t)
    plan = _Plan(R, a, rho, SCHEDULES[case["sched"]])
    perm = torch.from_numpy(plan.perm).cuda()
    count = case.get("outliers", 0)
    parts, done, step = [], 0, max(32, (1 << 24) // C)
    for r0 in range(0, R, step):
        r1 = min(R, r0 + step)
        wp, done = _weights64(plan, R, C, _key(seed, i), r0, r1, done, seqs)
        w = torch.empty_like(wp)
        w[:, perm] = wp
        if count:
            cols, vals = _outliers(seed, i, R, C, count)
            w[:, torch.from_numpy(cols).long().cuda()] = torch.from_numpy(vals[r0:r1].astype(np.float64)).cuda()
        parts.append(w if x is None else x.to(torch.float64) @ w.T)
    return torch.cat(parts, 0 if x is None else 1)


def _seqs(case):
    return {S: _sequences(S) for S in sorted({r[0] for r in SCHEDULES[case["sched"]]["rungs"]})}


def _sq_cols(w, g):
    """(W o W)^T g in row chunks (W: FP16 bits)."""
    out = torch.zeros(w.shape[1], dtype=torch.float64, device="cuda")
    for r in range(0, w.shape[0], 4096):
        c = w[r:r + 4096].view(torch.float16).to(torch.float64)
        out += (c * c).T @ g[r:r + 4096]
    return out


def _sq_rows(w, v):
    return torch.cat([(lambda c: (c * c) @ v)(w[r:r + 4096].view(torch.float16).to(torch.float64))
                      for r in range(0, w.shape[0], 4096)])


def _dynamic_range(w):
    """max |W_ij| / (median |W_ij| + 2^-24) per column where it reaches 1000, else 0."""
    a = w.view(torch.float16).abs()
    R = a.shape[0]
    mx = a.amax(0).to(torch.float64)
    out = torch.zeros_like(mx)
    low = (a <= (mx / 1000.0).to(torch.float16)).sum(0)
    for c in torch.nonzero(2 * low >= R - 1).flatten().tolist():
        s = torch.sort(a[:, c].to(torch.float64)).values
        dr = mx[c] / (0.5 * (s[(R - 1) // 2] + s[R // 2]) + 2.0 ** -24)
        out[c] = dr if dr >= 1000.0 else 0.0
    return out


def _exact_importance(case, seed):
    spec = _spec(case, seed)
    m = G.synth_model_device(spec)
    gain2 = lambda g: g.view(torch.float16).to(torch.float64) ** 2
    nodes, weights = np.polynomial.hermite.hermgauss(64)
    nodes, weights = torch.from_numpy(nodes).cuda(), torch.from_numpy(weights / np.sqrt(np.pi)).cuda()
    rep = spec.n_heads // spec.n_kv_heads
    L = spec.n_layers
    a_o, a_down, rho_o, rho_down = [None] * L, [None] * L, [None] * L, [None] * L
    g = _sq_cols(m.lm_head, torch.ones(spec.vocab, dtype=torch.float64, device="cuda"))
    for l in reversed(range(L)):
        y = m.layers[l]
        g = g / g.mean()  # rho has unit mean, so the stream's scale is free
        rho_down[l] = g
        gh = _sq_cols(y["wdown"], g)
        g = g + _sq_cols(y["wgate"], gh) + _sq_cols(y["wup"], gh)
        rho_o[l] = g / g.mean()
        ga = _sq_cols(y["wo"], g)
        g = g + _sq_cols(y["wv"], ga.view(spec.n_kv_heads, rep, spec.head_dim).sum(1).flatten())
        av, am = gain2(y["attn_norm"]), gain2(y["mlp_norm"])
        v = _sq_rows(y["wv"], av).view(spec.n_kv_heads, 1, spec.head_dim)
        a_o[l] = v.expand(-1, rep, -1).flatten()
        z = torch.sqrt(2.0 * _sq_rows(y["wgate"], am))[:, None] * nodes
        a_down[l] = ((z / (1.0 + torch.exp(-z))) ** 2) @ weights * _sq_rows(y["wup"], am)
    dyn, act = [], []
    for l in range(L):
        y = m.layers[l]
        av, am = gain2(y["attn_norm"]), gain2(y["mlp_norm"])
        for name, a in (("wq", av), ("wk", av), ("wv", av), ("wo", a_o[l]), ("wgate", am), ("wup", am),
                        ("wdown", a_down[l])):
            dyn.append(_dynamic_range(y[name]))
            act.append(a / a.mean())
    dyn.append(_dynamic_range(m.lm_head))
    af = gain2(m.final_norm)
    act.append(af / af.mean())
    return {"a_o": torch.cat(a_o), "a_down": torch.cat(a_down), "rho_o": torch.cat(rho_o),
            "rho_down": torch.cat(rho_down), "dyn_range": torch.cat(dyn), "act_ratio": torch.cat(act),
            "outliers": None}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("product", "set"):
        ts, seqs, n = _tensors(case), _seqs(case), case["n"]
        ys = [_exact_tensor(case, seed, i, t, _activations(seed, t[2], n, t[1]), seqs)
              for i, t in enumerate(ts)]
        return ys if kind == "product" else torch.cat([y.flatten() for y in ys])
    if kind == "decode":
        t = (case["R"], case["C"], "in", case["rho"])
        return _exact_tensor(case, seed, 0, t, None, _seqs(case))
    if kind == "importance":
        return _exact_importance(case, seed)
    if kind == "allocate":
        # The floor is an order statistic of the importance; the rest follows a search.
        imp, counts = [], []
        for i, t in enumerate(_allocation_tensors(case)):
            p = _Plan(t[0], *_factors(case, seed, i, t), SCHEDULES["4bpw"])
            rho = np.ones(1) if p.rho is None else p.rho
            imp.append((p.abar * rho[:, None]).ravel())
            counts.append(np.full(imp[-1].size, t[0] // rho.size))
        imp, counts = np.concatenate(imp), np.concatenate(counts)
        order = np.argsort(imp)
        m = int(np.ceil(0.06 * counts.sum()))
        q = imp[order][np.searchsorted(np.cumsum(counts[order]), m)]
        return {"theta": None, "j_tie": None, "q": float(q), "ties": None, "bits": None}
    return None  # the search over every seed in 64 bits takes minutes
