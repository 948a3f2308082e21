"""GPU: the decode at the sizes where its paths meet.

Every case decodes to its input exactly (bytes), plain and batched:
windows of 1024 root symbols at every misalignment of the output, root strips
of several windows (tiles above 2^18 symbols), levels of more than eight
windows, flat roots, both plan kernels (few and many records), directory
shares (blocks of many tiles) read by random access, and ANS bitmaps of one to
32 lanes sharing a unit."""
import numpy as np
import pytest

from test_gpu_parity import dev, off64

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2606_05765_gb300 as P
    P.set_tuning()
    return P


def draw(rng, n, p_hot, a):
    """n symbols: 0 with probability p_hot, the other a - 1 uniform."""
    x = rng.integers(1, a, n).astype(np.uint8) if a > 1 else np.zeros(n, np.uint8)
    x[rng.random(n) < p_hot] = 0
    return x


def blocks_of(kind, rng):
    if kind == "windows":       # sizes around windows and groups; odd sizes move the next block's output
        sizes = [1, 2, 31, 33, 255, 257, 1015, 1016, 1017, 1021, 1022, 1023, 1024, 1025, 1031, 2047, 2049, 8191, 8193]
        return [draw(rng, s + d, 0.6, 9) for s in sizes for d in (0, 1, 5)]
    if kind == "strips":        # one tile above 2^18 symbols: several windows to a strip
        return [draw(rng, n, 0.995, 40) for n in (262143, 262145, 700001)]
    if kind == "levels":        # levels of 10 to 24 windows, and tiles whose levels must be split
        return [draw(rng, 24000, 0.05, 5), draw(rng, 60000, 0.3, 6),
                np.concatenate([draw(rng, 30000, 0.999, 3), draw(rng, 30000, 0.0, 200)])]
    if kind == "flat":          # power-of-two alphabets: flat roots and flat nodes of every depth
        return [np.resize(rng.permutation(a), n).astype(np.uint8) for a in (4, 8, 16, 32, 64, 128, 256)
                for n in (a * 8, 4096 + a, 5000)]
    if kind == "many":          # more records than the batched launch has CTAs
        return [draw(rng, 40 + i % 97, 0.5, 2 + i % 30) for i in range(1500)]
    if kind == "shares":        # several directory shares
        return [draw(rng, 400000, 0.1, 250), draw(rng, 1 << 20, 0.2, 100)]
    # ANS bitmaps of every lane count: skewed nodes of 32 bytes to 40 KiB
    return [draw(rng, n, p, a) for n in (700, 5000, 40000, 131072, 330000) for p, a in ((0.9, 2), (0.93, 17), (0.97, 6))]


KINDS = ["windows", "strips", "levels", "flat", "many", "shares", "ans"]


@pytest.mark.parametrize("flat", [False, True])
@pytest.mark.parametrize("kind", KINDS)
def test_decode_edges(P, kind, flat):
    blocks = blocks_of(kind, np.random.default_rng(KINDS.index(kind)))
    data = np.concatenate(blocks)
    off = np.concatenate([[0], np.cumsum([b.size for b in blocks])]).astype(np.uint64)
    enc = P.encode(dev(data), off64(off), P.params(ans=kind == "ans", flat=flat))
    assert not enc.status.cpu().numpy().any()
    for batched in (False, True):
        out, st = P.decode(enc.comp, enc.off, off64(off), batched=batched)
        assert not st.cpu().numpy().any(), (kind, batched)
        assert np.array_equal(out.cpu().numpy()[: data.size], data), (kind, batched)
    if kind in ("shares", "ans", "strips"):
        rng = np.random.default_rng(99)
        qb = rng.integers(0, len(blocks), 5000).astype(np.int32)
        qp = (rng.random(5000) * np.array([blocks[b].size for b in qb])).astype(np.int32)
        sym, qst = P.Access(enc.comp, enc.off, len(blocks))(dev(qb), dev(qp))
        assert not qst.cpu().numpy().any()
        assert np.array_equal(sym.cpu().numpy(), np.array([blocks[b][p] for b, p in zip(qb, qp)]))
