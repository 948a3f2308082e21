"""Performance cases: the work a program that uses this library has it do.

Each case is one call sequence through the public Python binding, with
synthetic data of the shapes that `workloads/` and `bench.py` describe (made
on the GPU from the seed).  A case is a dict of plain values:

  op       "encode"  Encoder.run on device data (plan, placement, records, ANS)
           "decode"  Decoder.run on records encoded beforehand
           "round"   Encoder.run, then Decoder.run on its records
           "call"    the one-line calls encode() and decode(), which allocate
                     their buffers and read sizes back, as a first user writes
           "host"    HostCodec.compress and .decompress on pinned host memory
           "golomb"  golomb_encode() and golomb_decode()
           "access"  random access to single symbols of prepared records
  dist     "hot"     byte 0 with probability p, the others uniform (tail 0)
                     or Zipf with exponent `tail`
           "zipf"    Zipf with an alphabet and an exponent per block, uniform
                     in [a_lo, a_hi] and [s_lo, s_hi]
           "geom"    geometric values with mean code length `avg` (Golomb)
  nblk, lo, hi       blocks and their size range in bytes (log-uniform)
  ans, flat          encoder options: selective ANS, regrouped (flat) tree
  batched, graph     decoder options: one persistent launch; replayed as a
                     captured CUDA graph
"""
import math
import random

import numpy as np
import torch

import paper_2606_05765_gb300 as P

KiB, MiB = 1024, 1024 * 1024


def listed():
    hot80 = dict(dist="hot", p=0.8, tail=0.0)
    hot95 = dict(dist="hot", p=0.95, tail=1.3)
    mixed = dict(dist="zipf", a_lo=2, a_hi=256, s_lo=0.5, s_hi=2.0)
    return [
        # bulk compression of a large buffer cut into equal blocks: bench.py's headline workload, each direction
        dict(name="encode_skew80", op="encode", nblk=4096, lo=64 * KiB, hi=64 * KiB, ans=False, flat=True, **hot80),
        dict(name="decode_skew80", op="decode", nblk=4096, lo=64 * KiB, hi=64 * KiB, ans=False, flat=True,
             batched=True, graph=False, **hot80),
        # very skewed data (sparse tensors, masks), where the node bitmaps are worth ANS coding
        dict(name="encode_skew95_ans", op="encode", nblk=2048, lo=128 * KiB, hi=128 * KiB, ans=True, flat=False, **hot95),
        dict(name="decode_skew95_ans", op="decode", nblk=2048, lo=128 * KiB, hi=128 * KiB, ans=True, flat=False,
             batched=True, graph=False, **hot95),
        # a batch of unrelated blocks of uneven size, alphabet and skew (a store's pages, columns, chunks);
        # decoded as a serving loop does, by replaying a captured graph
        dict(name="encode_mixed_ans", op="encode", nblk=1024, lo=4 * KiB, hi=MiB, ans=True, flat=True, **mixed),
        dict(name="decode_mixed_ans", op="decode", nblk=1024, lo=4 * KiB, hi=MiB, ans=True, flat=True, batched=True,
             graph=True, **mixed),
        # one large block alone (one file, one column), both directions
        dict(name="round_zipf_1x1m", op="round", nblk=1, lo=MiB, hi=MiB, ans=False, flat=False, batched=False,
             graph=False, dist="zipf", a_lo=256, a_hi=256, s_lo=1.0, s_hi=1.0),
        # the smallest requests: a handful of short blocks through the one-line calls, where latency counts
        dict(name="call_small", op="call", nblk=12, lo=KiB, hi=16 * KiB, ans=False, flat=False, batched=False,
             graph=False, **hot80),
        # text-like blocks of odd sizes with the default parameters (canonical tree) and the plain decoder
        dict(name="round_text_canonical", op="round", nblk=509, lo=20011, hi=300007, ans=False, flat=False,
             batched=False, graph=False, dist="zipf", a_lo=60, a_hi=120, s_lo=0.8, s_hi=1.2),
        # a batch held in host memory, copies overlapped with the kernels
        dict(name="host_skew80", op="host", nblk=1024, lo=64 * KiB, hi=64 * KiB, ans=False, flat=True, **hot80),
        # small integers (gaps, run lengths) with the Golomb coder, blocks of odd sizes
        dict(name="golomb_2", op="golomb", nblk=2048, lo=9001, hi=32 * KiB, dist="geom", avg=2.0),
        # point lookups in compressed records
        dict(name="access_1m", op="access", nblk=1024, lo=64 * KiB, hi=64 * KiB, ans=False, flat=True, nq=1 << 20,
             **hot80),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["encode", "encode", "decode", "decode", "round", "call", "host", "golomb", "access"])
    if op == "golomb":
        hi = _log_int(rng, 2 * KiB, 32 * KiB)
        return dict(op=op, nblk=_log_int(rng, 1, 2048), lo=max(1, hi // rng.randint(1, 8)), hi=hi, dist="geom",
                    avg=round(rng.uniform(1.25, 5.0), 2))
    c = dict(op=op, ans=rng.random() < 0.5, flat=rng.random() < 0.6, batched=rng.random() < 0.5,
             graph=rng.random() < 0.25)
    if op in ("encode", "host", "access", "call"):
        c.pop("graph")
    if op in ("encode", "host", "access"):
        c.pop("batched")
    hi = _log_int(rng, KiB, MiB)
    c["hi"], c["lo"] = hi, max(64, hi // rng.choice([1, 1, 2, 16, 200]))
    mean = (c["hi"] + c["lo"]) / 2 if c["lo"] == c["hi"] else (c["hi"] - c["lo"]) / math.log(c["hi"] / c["lo"])
    # the ANS coder and wide alphabets cost more per byte: the batch stays below the largest listed one's time
    most = {"encode": 128 * MiB, "decode": 128 * MiB, "round": 64 * MiB, "call": MiB, "host": 64 * MiB,
            "access": 64 * MiB}[op]
    c["nblk"] = _log_int(rng, 1, max(1, min(4096 if op != "call" else 64, int(most / mean))))
    if op == "access":
        c["nq"] = _log_int(rng, 1000, 1 << 20)
    if rng.random() < 0.5:
        c.update(dist="hot", p=round(rng.uniform(0.5, 0.98), 3), tail=rng.choice([0.0, 1.0, 1.3]))
    else:
        a = _log_int(rng, 2, 256)
        s = rng.uniform(0.4, 1.8)
        c.update(dist="zipf", a_lo=max(2, a // rng.choice([1, 2, 16])), a_hi=a, s_lo=round(s, 2),
                 s_hi=round(s + rng.choice([0.0, 0.3, 0.8]), 2))
    return c


# ------------------------------------------------------------------ inputs ----
def _sizes(case):
    """The blocks' sizes: a property of the case (not of the seed)."""
    lo, hi, n = case["lo"], case["hi"], case["nblk"]
    if lo == hi:
        return np.full(n, lo, np.int64)
    r = np.random.Generator(np.random.PCG64(n * 1000003 + lo * 31 + hi))
    return np.clip(np.floor(np.exp(r.uniform(math.log(lo), math.log(hi + 1), n))), lo, hi).astype(np.int64)


def _hot_probs(case):
    k = np.arange(1, 256, dtype=np.float64)
    t = k ** -case["tail"]
    return np.concatenate([[case["p"]], (1.0 - case["p"]) * t / t.sum()])


def _draw_symbols(g, probs, n, out):
    """n i.i.d. draws by inverse CDF into out (uint8, device)."""
    cdf = torch.from_numpy(np.cumsum(probs / probs.sum()).astype(np.float32)).to(out.device)
    step = 1 << 26
    for i in range(0, n, step):
        m = min(step, n - i)
        u = torch.rand(m, generator=g, device=out.device)
        out[i:i + m] = torch.searchsorted(cdf, u, right=True).clamp_(max=len(probs) - 1).to(torch.uint8)


def _data(case, seed):
    """(data, block offsets) on the GPU, from the seed alone."""
    sizes = _sizes(case)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n = int(off[-1])
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    data = torch.empty(n, dtype=torch.uint8, device="cuda")
    if case["dist"] == "hot":
        _draw_symbols(g, _hot_probs(case), n, data)
    elif case["dist"] == "geom":
        q = 1.0 / case["avg"]
        for i in range(0, n, 1 << 26):
            m = min(1 << 26, n - i)
            u = torch.rand(m, generator=g, device="cuda").clamp_(min=1e-30)
            data[i:i + m] = torch.floor(torch.log(u) / math.log1p(-q)).clamp_(max=255).to(torch.uint8)
    else:
        r = np.random.Generator(np.random.PCG64(seed))
        a = r.integers(case["a_lo"], case["a_hi"] + 1, len(sizes))
        s = r.uniform(case["s_lo"], case["s_hi"], len(sizes))
        for b in range(len(sizes)):
            k = np.arange(1, int(a[b]) + 1, dtype=np.float64)
            _draw_symbols(g, k ** -s[b], int(sizes[b]), data[int(off[b]):int(off[b + 1])])
    return data, torch.from_numpy(off).to("cuda")


class State:
    pass


def prepare(case, seed):
    s = State()
    s.op = case["op"]
    s.data, s.off = _data(case, seed)
    n = case["nblk"]
    # room for the records: the largest they can be, so that a buffer serves any data of these sizes
    room = int((2 * _sizes(case) + 2720).sum())
    if s.op == "golomb":
        s.store = torch.zeros(room, dtype=torch.uint8, device="cuda")
        s.out = torch.empty_like(s.data)
        s.status = torch.empty(n, dtype=torch.int32, device="cuda")
        return s
    s.prm = P.params(ans=case["ans"], flat=case["flat"])
    if s.op == "call":
        s.batched = case["batched"]
        s.store = torch.zeros(room, dtype=torch.uint8, device="cuda")
        return s
    if s.op == "host":
        boff = s.off.cpu().numpy().astype(np.uint64)
        s.codec = P.HostCodec(boff, s.prm, segments=4)
        s.raw = torch.empty(s.data.numel(), dtype=torch.uint8, pin_memory=True)
        s.raw.copy_(s.data)
        # pages of the record buffer that a call leaves alone stay as they are: the same for every pass
        s.comp = torch.zeros(s.codec.capacity, dtype=torch.uint8).pin_memory()
        s.back = torch.empty(s.data.numel(), dtype=torch.uint8, pin_memory=True)
        s.data = None
        return s
    s.enc = P.Encoder(n, s.prm)
    s.enc.ensure(room)
    s.enc.comp.zero_()
    if s.op == "encode":
        return s
    e = s.enc.run(s.data, s.off)
    if s.op == "access":
        r = torch.Generator(device="cuda")
        r.manual_seed(seed + 1)
        nq = case["nq"]
        qb = torch.randint(0, n, (nq,), generator=r, device="cuda")
        size = (s.off[1:] - s.off[:-1])[qb]
        s.qpos = (torch.rand(nq, generator=r, device="cuda", dtype=torch.float64) * size).to(torch.int64)
        s.qpos = torch.minimum(s.qpos, size - 1).to(torch.int32)
        s.qblk = qb.to(torch.int32)
        s.access = P.Access(e.comp, e.off, n)
        s.data = None
        return s
    s.dec = P.Decoder(n, batched=case["batched"])
    s.dec.prepare(e.comp, e.off)
    s.out = torch.empty_like(s.data)
    s.comp, s.coff = e.comp, e.off
    s.graph = None
    if case["graph"] and s.op == "decode":
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        s.dec.run(s.comp, s.coff, s.out, s.off, stream=side)
        side.synchronize()
        s.graph = P.Graph(side)
        with s.graph:
            s.dec.run(s.comp, s.coff, s.out, s.off, stream=side)
    if s.op == "decode":
        s.enc = s.data = None
    return s


def run(s):
    if s.op == "encode":
        e = s.enc.run(s.data, s.off)
        return {"comp": e.comp, "off": e.off, "rec_bytes": e.rec_bytes, "status": e.status}
    if s.op == "decode":
        if s.graph is not None:
            s.graph.launch(torch.cuda.current_stream())
        else:
            s.dec.run(s.comp, s.coff, s.out, s.off)
        return {"out": s.out, "status": s.dec.status}
    if s.op == "round":
        e = s.enc.run(s.data, s.off)
        s.dec.run(e.comp, e.off, s.out, s.off)
        return {"comp": e.comp, "rec_bytes": e.rec_bytes, "status": e.status, "out": s.out, "dstatus": s.dec.status}
    if s.op == "call":
        e = P.encode(s.data, s.off, s.prm)
        out, st = P.decode(e.comp, e.off, s.off, batched=s.batched)
        s.store[:e.comp.numel()].copy_(e.comp)   # into the program's own store
        return {"comp": s.store, "rec_bytes": e.rec_bytes, "status": e.status, "out": out, "dstatus": st}
    if s.op == "host":
        coff, st = s.codec.compress(s.raw, s.comp)
        coff, st = coff.copy(), st.copy()
        dst = s.codec.decompress(s.comp, coff, s.back)
        return {"comp": s.comp, "off": coff.astype(np.int64), "status": st, "out": s.back, "dstatus": dst.copy()}
    if s.op == "golomb":
        e = P.golomb_encode(s.data, s.off)
        P.golomb_decode(e.comp, e.off, s.out, s.off, s.status)
        s.store[:e.comp.numel()].copy_(e.comp)
        return {"comp": s.store, "rec_bytes": e.rec_bytes, "status": e.status, "out": s.out, "dstatus": s.status}
    sym, qst = s.access(s.qblk, s.qpos)
    return {"sym": sym, "status": qst}


# --------------------------------------------------------------------- work ----
def _entropy(p):
    p = p[p > 0] / p.sum()
    return float(-(p * np.log2(p)).sum())


def _bits(case):
    """Expected code bits per symbol of the case's data (its entropy)."""
    if case["dist"] == "geom":
        return case["avg"]
    if case["dist"] == "hot":
        h = _entropy(_hot_probs(case))
        return h if case["ans"] else max(1.0, h)
    r = random.Random(1)
    tot = 0.0
    for _ in range(64):
        a, x = r.randint(case["a_lo"], case["a_hi"]), r.uniform(case["s_lo"], case["s_hi"])
        h = _entropy(np.arange(1, a + 1, dtype=np.float64) ** -x)
        tot += h if case["ans"] else max(1.0, h)
    return tot / 64


def work(case):
    """Raw bytes read once and records written once (encode), the reverse (decode)."""
    n = int(_sizes(case).sum())
    if case["op"] == "access":
        # each query's block, position, symbol and status, and the bit it decides on at each node of its walk
        return {"bytes": case["nq"] * (4 + 4 + 1 + 4 + _bits(case) / 8), "flops": 0}
    one = n + n * _bits(case) / 8 + 200 * case["nblk"]
    return {"bytes": one * (1 if case["op"] in ("encode", "decode") else 2), "flops": 0}


def exact(case, seed):
    """Decoding gives back the data; the records have no value in plain arithmetic."""
    if case["op"] in ("encode", "access"):
        return None
    data, _ = _data(case, seed)
    zero = torch.zeros(case["nblk"], dtype=torch.int32, device="cuda")
    if case["op"] == "decode":
        return {"out": data, "status": zero}
    if case["op"] == "host":
        return {"comp": None, "off": None, "status": zero, "out": data, "dstatus": zero}
    return {"comp": None, "rec_bytes": None, "status": zero, "out": data, "dstatus": zero}
