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


def test_scratch_of_a_corrupt_record(P):   # noqa: F811
    """255 ANS-coded nodes whose counts ask for more than 2^32 bytes of scratch:
    refused by the plan (by one CTA a record, and by warps), not given a place
    as small as the sum's low 32 bits."""
    import torch
    V, nv = 255, 8 * 17_000_000
    S = (nv // 8 + 16383) // 16384
    tail = (nv // 8) % 16384
    alen = 4 * S + 128 * (S - 1) + 4 * ((tail + 511) // 512)
    hdr = np.zeros((144 + 5 * V + 3) // 4 * 4 + 4 * V, np.uint8)
    size = (hdr.size + V * alen + 15) & ~15
    hdr[0:8] = np.array([size, nv], np.uint32).view(np.uint8)
    hdr[8], hdr[10] = V, 2
    hdr[12:16] = np.frombuffer(b"PVC1", np.uint8)
    hdr[16:144] = 0x88                              # 256 codes of 8 bits
    hdr[144:144 + 4 * V] = np.full(V, nv, np.uint32).view(np.uint8)
    hdr[144 + 4 * V:144 + 5 * V] = 30
    hdr[-4 * V:] = np.full(V, alen, np.uint32).view(np.uint8)
    comp = torch.zeros(size, dtype=torch.uint8, device="cuda")
    comp[:hdr.size] = torch.from_numpy(hdr).cuda()
    assert V * ((nv // 8 + 15) // 16 * 16 + 16) >> 32
    # (sizing alone: the plan is all that runs)
    for n in (1, 700):
        # the same record, then records of constant blocks
        one = np.zeros(16, np.uint8)
        one[0:8] = np.array([16, 5], np.uint32).view(np.uint8)
        one[10], one[11] = 1, 7
        one[12:16] = hdr[12:16]
        buf = torch.cat([comp, torch.from_numpy(np.tile(one, n - 1)).cuda()])
        coff = np.concatenate([[0], size + 16 * np.arange(n)])
        d = P.Decoder(n)
        d.prepare(buf, off64(coff))
        st = d.status.cpu().numpy()
        assert st[0] == P.ERR_CORRUPT and not st[1:].any()
