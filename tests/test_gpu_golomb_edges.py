"""GPU: PivCo-Golomb at the sizes where its paths meet: blocks around whole
groups of 32 values per warp and windows of 1024 bits, blocks of few values and
of one long run, input, records and output at every misalignment, and records
with one wrong bit (a stop moved, added or taken out, a pad bit set)."""
import numpy as np
import pytest

from test_gpu_decode_edges import P   # noqa: F401  (fixture)
from test_gpu_parity import dev, off64

pytestmark = pytest.mark.gpu


def values(rng, n, kind):
    if kind == "geom":
        return (rng.geometric(0.45, n) - 1).clip(0, 255).astype(np.uint8)
    if kind == "long":
        return (rng.geometric(0.03, n) - 1).clip(0, 255).astype(np.uint8)
    if kind == "one":
        return np.where(np.arange(n) == n // 2, 200, 0).astype(np.uint8)
    return np.repeat(rng.integers(0, 256, n // 700 + 1).astype(np.uint8), 700)[:n]


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
@pytest.mark.parametrize("kind", ["geom", "long", "one", "runs"])
def test_golomb_edges(P, kind, shift):   # noqa: F811
    import oracle
    import torch
    oracle.build()
    rng = np.random.default_rng(40 + shift)
    sizes = [1, 2, 31, 32, 33, 255, 256, 257, 511, 513, 1025, 8191, 8192, 8193, 8448, 9001, 16385, 32767, 32768]
    vals = [values(rng, n, kind) for n in sizes]
    refs = [oracle.golomb_encode(v) for v in vals]
    off = np.concatenate([[0], np.cumsum(sizes)])
    n = len(sizes)
    data = dev(np.concatenate([np.zeros(shift, np.uint8)] + vals))[shift:]
    # records at odd places, a guard byte of 0xA5 before, between and after them
    roff = np.concatenate([[0], np.cumsum([r.size for r in refs])]) + shift
    comp = torch.full((int(roff[-1]) + 8,), 0xA5, dtype=torch.uint8, device="cuda")
    rb = torch.zeros(n, dtype=torch.int64, device="cuda")
    st = torch.full((n,), 9, dtype=torch.int32, device="cuda")
    d_off, d_roff = off64(off), off64(roff)
    P._check(P.lib().pivco_golomb_encode(P._ptr(data), P._ptr(d_off), n, P._ptr(comp), P._ptr(d_roff), P._ptr(rb),
                                         P._ptr(st), P._stream(None)), "encode")
    assert not st.cpu().numpy().any()
    c = comp.cpu().numpy()
    for b in range(n):
        assert int(rb[b]) == refs[b].size and np.array_equal(c[roff[b]:roff[b + 1]], refs[b]), (kind, sizes[b])
    assert (c[:shift] == 0xA5).all() and (c[roff[-1]:] == 0xA5).all()
    out = torch.full((int(off[-1]) + 8,), 0xA5, dtype=torch.uint8, device="cuda")
    P.golomb_decode(comp, off64(roff), out, off64(off + shift), st)
    assert not st.cpu().numpy().any()
    o = out.cpu().numpy()
    assert np.array_equal(o[shift:shift + int(off[-1])], np.concatenate(vals))
    assert (o[:shift] == 0xA5).all() and (o[shift + int(off[-1]):] == 0xA5).all()


def test_golomb_rejects_wrong_bits(P):   # noqa: F811
    import oracle
    import torch
    oracle.build()
    rng = np.random.default_rng(8)
    vals = values(rng, 5003, "geom")
    good = oracle.golomb_encode(vals)
    m = int(good[8]) | int(good[9]) << 8
    nj = good[16:16 + 4 * m].view(np.uint32).astype(np.int64)
    start = 16 + 4 * m + np.concatenate([[0], np.cumsum((nj + 7) // 8)])
    recs = [good]
    for j in range(min(m, 6)):
        r = good.copy()                       # one bit the other way round: the level's count is wrong
        r[start[j] + int(nj[j]) // 16] ^= 4
        recs.append(r)
        if nj[j] % 8:
            r = good.copy()                   # a pad bit
            r[start[j + 1] - 1] |= 0x80
            recs.append(r)
    n = len(recs)
    roff = np.concatenate([[0], np.cumsum([r.size for r in recs])])
    out = torch.full((n * vals.size,), 0xA5, dtype=torch.uint8, device="cuda")
    st = torch.full((n,), 9, dtype=torch.int32, device="cuda")
    P.golomb_decode(dev(np.concatenate(recs)), off64(roff), out, off64(np.arange(n + 1) * vals.size), st)
    assert list(st.cpu().numpy()) == [0] + [P.ERR_CORRUPT] * (n - 1)
    o = out.cpu().numpy().reshape(n, -1)
    assert np.array_equal(o[0], vals) and (o[1:] == 0xA5).all()
