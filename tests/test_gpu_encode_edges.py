"""GPU: records byte for byte against the oracle at the sizes where the
encoder's paths meet: windows of 1024 root symbols at every misalignment of
the input, roots with one leaf child and with two internal ones, levels of
more than eight windows, flat nodes of every depth, big blocks coded in parts
and by shares of a planning chunk, ANS bitmaps of one to 32 lanes."""
import numpy as np
import pytest

from test_gpu_decode_edges import KINDS, P, blocks_of   # noqa: F401  (P: fixture)
from test_gpu_parity import dev, off64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flat", [False, True])
@pytest.mark.parametrize("kind", [k for k in KINDS if k != "many"])
def test_encode_edges(P, kind, flat):   # noqa: F811
    import oracle
    oracle.build()
    blocks = blocks_of(kind, np.random.default_rng(50 + KINDS.index(kind)))
    data = np.concatenate(blocks)
    off = np.concatenate([[0], np.cumsum([b.size for b in blocks])]).astype(np.uint64)
    ans = kind == "ans"
    ref, rec_off, sizes = oracle.encode_batch(data, off, oracle.params(ans=ans, flat=flat))
    enc = P.encode(dev(data), off64(off), P.params(ans=ans, flat=flat))
    assert not enc.status.cpu().numpy().any()
    comp, eo, rb = enc.comp.cpu().numpy(), enc.off.cpu().numpy(), enc.rec_bytes.cpu().numpy()
    for b in range(len(blocks)):
        assert rb[b] == sizes[b], (kind, b)
        assert np.array_equal(comp[eo[b]:eo[b] + rb[b]], ref[int(rec_off[b]):int(rec_off[b]) + int(sizes[b])]), (kind, b)
    # without the chunk histograms every block is coded by one CTA, big ones in parts counted from the input
    e = P.Encoder(len(blocks), P.params(ans=False, flat=flat))
    total = e.plan(dev(data), off64(off))
    e.ensure(total)
    P.encode_blocks(dev(data), off64(off), len(blocks), e.layout, e.comp, e.off, e.rec_bytes, e.status)
    c1, r1 = e.comp[:total].cpu().numpy(), e.rec_bytes.cpu().numpy()
    assert not e.status.cpu().numpy().any()
    e.comp.zero_()
    e.run(dev(data), off64(off))
    assert np.array_equal(c1, e.comp[:total].cpu().numpy()) and np.array_equal(r1, e.rec_bytes.cpu().numpy())
