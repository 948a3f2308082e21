"""GPU: records whose bitmaps send a child more symbols than it has.

The last tile of a block is decoded in shorter chunks when its levels do not
fit the buffers (the block's statistics drift), with the chunks' demands
counted from the bitmaps themselves.  Bits set in the root's bitmap there make
a child's demand run past its body, here the record's last one: the tile must
be refused before anything of it is read, and the records and outputs beside
it stay as they are."""
import numpy as np
import pytest

from test_gpu_decode_edges import P, draw   # noqa: F401  (P: fixture)
from test_gpu_parity import dev, off64

pytestmark = pytest.mark.gpu

N, HOT, A = 460000, 230000, 65      # byte 0 alone, then half of it byte 0 and half 64 others
TAIL = 40000                        # symbols at the end whose root bits are set: within the last tile


def corrupt_tail(rec):
    """The record with the last TAIL bits of its root's bitmap set, and the
    bits by which the record's last node then runs past the record."""
    V = int(rec[8])
    alen = (144 + 5 * V + 3) & ~3   # no node is listed: the bodies start here, the root's first
    root = np.unpackbits(rec[alen:alen + (N + 7) // 8], bitorder="little")
    assert root[:N].sum() < N // 3  # byte 0 is the left leaf, ones go to the only internal child
    more = TAIL - int(root[N - TAIL:N].sum())
    root[N - TAIL:N] = 1
    bad = rec.copy()
    bad[alen:alen + (N + 7) // 8] = np.packbits(root, bitorder="little")
    return bad, more


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("flat", [False, True])
def test_demand_past_the_body_is_refused(P, flat, batched):   # noqa: F811
    import oracle
    oracle.build()
    rng = np.random.default_rng(11)
    x = np.concatenate([np.zeros(HOT, np.uint8), draw(rng, N - HOT, 0.5, A)])
    prm = oracle.params(flat=flat)
    rec = oracle.encode_block(x, prm)
    bad, more = corrupt_tail(rec)
    assert more > 8 * 16            # past the body, the record's padding and more
    assert oracle.decode_block(bad)[0] != 0
    side = [draw(rng, 3000 + 7 * i, 0.7, 30) for i in range(6)]
    recs = [oracle.encode_block(s, prm) for s in side]
    for first, want in ((rec, 0), (bad, P.ERR_CORRUPT)):
        comp = np.concatenate([recs[0], first] + recs[1:])
        blocks = [side[0], x] + side[1:]
        coff = np.concatenate([[0], np.cumsum([r.size for r in [recs[0], first] + recs[1:]])])
        ooff = np.concatenate([[0], np.cumsum([b.size for b in blocks])])
        out, st = P.decode(dev(comp), off64(coff), off64(ooff), batched=batched)
        st, out = st.cpu().numpy(), out.cpu().numpy()
        assert st[1] == want and not np.delete(st, 1).any()
        for b in range(len(blocks)):
            if st[b] == 0:
                assert np.array_equal(out[int(ooff[b]):int(ooff[b + 1])], blocks[b]), b
