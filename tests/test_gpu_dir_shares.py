"""GPU: rank directories of more shares than tiles (batches of few tiles).

The shares' tails live between the tile cursors: trees of one node to a full
alphabet, two tiles and many, every directory granularity, plain and batched,
and random access (which also has directories for blocks of one tile) all give
the input back."""
import numpy as np
import pytest

from test_gpu_decode_edges import P, draw   # noqa: F401  (P: fixture)
from test_gpu_parity import dev, off64

pytestmark = pytest.mark.gpu

BATCHES = {
    "shallow": [(60000, 0.4, 4), (75100, 0.4, 6), (60001, 0.4, 3), (33000, 0.9, 2), (5, 0.5, 2)],
    "one": [(1 << 20, 0.9, 4)],
    "root": [((1 << 20) + 4099, 0.5, 2)],
    "wide": [(200003, 0.02, 256), (90000, 0.3, 120)],
}


@pytest.mark.parametrize("dir_bits,tile_max", [(128, 1 << 20), (32, 1 << 20), (256, 1 << 16), (64, 8192)])
@pytest.mark.parametrize("kind", sorted(BATCHES))
@pytest.mark.parametrize("flat", [False, True])
def test_more_shares_than_tiles(P, kind, flat, dir_bits, tile_max):   # noqa: F811
    rng = np.random.default_rng(sorted(BATCHES).index(kind))
    blocks = [draw(rng, *b) for b in BATCHES[kind]]
    data = np.concatenate(blocks)
    off = np.concatenate([[0], np.cumsum([b.size for b in blocks])]).astype(np.uint64)
    enc = P.encode(dev(data), off64(off), P.params(ans=kind == "one", flat=flat))
    assert not enc.status.cpu().numpy().any()
    try:
        P.set_tuning(tile_max=tile_max, dir_bits=dir_bits)
        for batched in (False, True):
            out, st = P.decode(enc.comp, enc.off, off64(off), batched=batched)
            assert not st.cpu().numpy().any(), batched
            assert np.array_equal(out.cpu().numpy()[: data.size], data), batched
        qb = rng.integers(0, len(blocks), 4000).astype(np.int32)
        qp = (rng.random(4000) * np.array([blocks[b].size for b in qb])).astype(np.int32)
        sym, qst = P.Access(enc.comp, enc.off, len(blocks))(dev(qb), dev(qp))
        assert not qst.cpu().numpy().any()
        assert np.array_equal(sym.cpu().numpy(), np.array([blocks[b][p] for b, p in zip(qb, qp)]))
    finally:
        P.set_tuning()
