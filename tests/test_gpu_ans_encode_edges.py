"""GPU: ANS-coded records byte for byte against the oracle, and decoded again,
at the sizes where the units of the ANS coder meet: bitmaps of one byte to several 16 KiB
segments, last segments too short to hold their own states (or that grow when
coded), nodes kept raw between coded ones, and a scratch buffer with no room
for the last block's mirror (one warp codes that block)."""
import numpy as np
import pytest

from test_gpu_decode_edges import P, draw   # noqa: F401  (P: fixture)
from test_gpu_parity import dev, off64

pytestmark = pytest.mark.gpu


def bitmap_blocks(rng, sizes):
    """Two-symbol blocks: one bitmap of that many bytes each."""
    return [draw(rng, 8 * s - int(rng.integers(0, 8)), 0.96, 2) for s in sizes]


def blocks_of(kind, rng):
    if kind == "tiny":
        return bitmap_blocks(rng, list(range(1, 40)) + [63, 64, 65, 127, 129, 511, 512, 513, 1023, 1025])
    if kind == "segments":
        return bitmap_blocks(rng, [16383, 16384] + [16384 + k for k in (1, 2, 3, 5, 9, 13, 16, 17, 31, 40, 511, 513, 8191)]
                             + [32767, 32768, 32769, 32768 + 15])
    if kind == "dense":     # bitmaps that hardly compress: more words than a unit's windows hold at once
        return [draw(rng, 8 * s, p, 2) for s in (300, 600, 3000, 8480, 8704, 12000, 16383) for p in (0.72, 0.8)]
    if kind == "growing":   # the last segment, or a whole one, does not compress
        out = []
        for n, m in ((16384, 20), (16384, 700), (16384, 4000), (32768, 11000), (16384, 16384), (32768, 16384 + 300)):
            out.append(np.concatenate([draw(rng, 8 * n, 0.99, 2), rng.integers(0, 2, 8 * m).astype(np.uint8)]))
            out.append(np.concatenate([rng.integers(0, 2, 8 * m).astype(np.uint8), draw(rng, 8 * n, 0.99, 2)]))
        return out
    # many nodes, some kept raw
    return [draw(rng, int(rng.integers(300, 60000)), float(rng.choice([0.5, 0.9, 0.97])), int(rng.integers(2, 40)))
            for _ in range(40)] + [draw(rng, 300000, 0.9, 30)]


@pytest.mark.parametrize("kind", ["tiny", "segments", "dense", "growing", "nodes"])
def test_ans_encode_edges(P, kind):   # noqa: F811
    import oracle
    oracle.build()
    blocks = blocks_of(kind, np.random.default_rng(len(kind)))
    n = len(blocks)
    data = np.concatenate(blocks)
    off = np.concatenate([[0], np.cumsum([b.size for b in blocks])]).astype(np.uint64)
    ref, rec_off, sizes = oracle.encode_batch(data, off, oracle.params(ans=True, flat=False))
    e = P.Encoder(n, P.params(ans=True, flat=False))
    total = e.plan(dev(data), off64(off))
    e.ensure(total)
    for room in (total, total - 1):
        e.run(dev(data), off64(off))   # (all of it, then its ANS step again on raw records below)
        if room < total:
            P.encode_blocks(dev(data), off64(off), n, e.layout, e.comp, e.off, e.rec_bytes, e.status)
            P.ans_encode_blocks(e.layout, n, e.comp, e.off, e.rec_bytes, e.ans_ws[:room], e.status)
        assert not e.status.cpu().numpy().any()
        comp, eo, rb = e.comp.cpu().numpy(), e.off.cpu().numpy(), e.rec_bytes.cpu().numpy()
        for b in range(n):
            assert rb[b] == sizes[b], (kind, room < total, b)
            assert np.array_equal(comp[eo[b]:eo[b] + rb[b]], ref[int(rec_off[b]):int(rec_off[b]) + int(sizes[b])]), (kind, b)
    for batched in (False, True):
        out, st = P.decode(e.comp, e.off, off64(off), batched=batched)
        assert not st.cpu().numpy().any()
        assert np.array_equal(out.cpu().numpy()[: data.size], data), (kind, batched)
