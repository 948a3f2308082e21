"""GPU: ANS-coded nodes whose segments do not all compress (the block's
statistics drift): segments larger coded than raw at every place of a node, in
several nodes of a block, more of them than the coder takes beside the others,
and in a node that is kept raw in the end.  Byte for byte against the oracle,
and decoded again."""
import numpy as np
import pytest

from test_gpu_decode_edges import P, draw   # noqa: F401  (P: fixture)
from test_gpu_parity import dev, off64

pytestmark = pytest.mark.gpu

SEG = 8 * 16384     # symbols of a two-symbol block per segment


def noise(rng, n):
    return rng.integers(0, 2, n).astype(np.uint8)


def blocks_of(kind, rng):
    if kind == "places":
        out = []
        for pat in ("NZZ", "ZNZ", "ZZN", "NZNZZ", "ZZZNN", "NNZZ", "NNNZZ"):
            out.append(np.concatenate([noise(rng, SEG) if c == "N" else draw(rng, SEG, 0.98, 2) for c in pat]))
            out.append(out[-1][: -int(rng.integers(1, SEG - 200))])                 # a last segment of its own
            out.append(np.concatenate([out[-2], noise(rng, int(rng.integers(8, 4000)))]))
        return out
    if kind == "nodes":         # several nodes with such segments, and raw ones between
        return [np.concatenate([draw(rng, 3 * SEG, 0.95, 12), draw(rng, 2 * SEG, 0.4, 60), draw(rng, 3 * SEG, 0.93, 5)])
                for _ in range(3)]
    # more than the coder's list holds
    return [np.concatenate([draw(rng, 130 * SEG, 0.99, 2), noise(rng, 70 * SEG)])]


@pytest.mark.parametrize("flat", [False, True])
@pytest.mark.parametrize("kind", ["places", "nodes", "many"])
def test_ans_drift(P, kind, flat):   # noqa: F811
    import oracle
    oracle.build()
    blocks = blocks_of(kind, np.random.default_rng(len(kind)))
    data = np.concatenate(blocks)
    off = np.concatenate([[0], np.cumsum([b.size for b in blocks])]).astype(np.uint64)
    ref, rec_off, sizes = oracle.encode_batch(data, off, oracle.params(ans=True, flat=flat))
    enc = P.encode(dev(data), off64(off), P.params(ans=True, flat=flat))
    assert not enc.status.cpu().numpy().any()
    comp, eo, rb = enc.comp.cpu().numpy(), enc.off.cpu().numpy(), enc.rec_bytes.cpu().numpy()
    for b in range(len(blocks)):
        assert rb[b] == sizes[b], b
        assert np.array_equal(comp[eo[b]:eo[b] + rb[b]], ref[int(rec_off[b]):int(rec_off[b]) + int(sizes[b])]), b
    out, st = P.decode(enc.comp, enc.off, off64(off), batched=True)
    assert not st.cpu().numpy().any()
    assert np.array_equal(out.cpu().numpy()[: data.size], data)
