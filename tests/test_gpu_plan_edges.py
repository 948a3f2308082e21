"""GPU: the planning pass at the sizes where its paths meet: code lengths for
symbol counts around the powers of two that the sort is cut to and for counts
around 2^24 (wider keys) against the oracle; the plan of few blocks (a cluster
per block, blocks counted by all its CTAs or by one) and of many against the
step-by-step calls."""
import numpy as np
import pytest

from test_gpu_decode_edges import P, draw   # noqa: F401  (P: fixture)
from test_gpu_parity import dev, off64

pytestmark = pytest.mark.gpu


def test_code_length_edges(P):   # noqa: F811
    import oracle
    import torch
    oracle.build()
    rng = np.random.default_rng(5)
    hs = []
    for K in (2, 3, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256):
        for top in (1, 3, 1000, 2 ** 24 - 2, 2 ** 24 - 1, 2 ** 24, 2 ** 30):
            h = np.zeros(256, np.uint32)
            h[rng.permutation(256)[:K]] = rng.integers(1, min(top, 50) + 1, K)
            h[np.flatnonzero(h)[:K // 2]] = top
            hs.append(h)
    H = np.stack(hs)
    lens = torch.empty(len(hs) * 256, dtype=torch.uint8, device="cuda")
    st = torch.full((len(hs),), 9, dtype=torch.int32, device="cuda")
    for L in (8, 11, 15):
        P.code_lengths(dev(H.reshape(-1).view(np.int32)), len(hs), L, lens, st)
        got = lens.cpu().numpy().reshape(-1, 256)
        assert not st.cpu().numpy().any()
        for i, h in enumerate(hs):
            assert np.array_equal(got[i], oracle.code_lengths(h, L)), (L, i)


@pytest.mark.parametrize("many", [False, True])
def test_plan_edges(P, many):   # noqa: F811
    import torch
    rng = np.random.default_rng(6)
    blocks = [draw(rng, n, p, a) for n in (0, 1, 4095, 32767, 32768, 32769, 40001, 262144, 1000003)
              for p, a in ((0.8, 256), (0.2, 7))]
    if many:
        blocks = blocks + [draw(rng, int(n), 0.5, 90) for n in rng.integers(1, 2000, 200)]
    n = len(blocks)
    off = off64(np.concatenate([[0], np.cumsum([b.size for b in blocks])]))
    for shift in (0, 5):
        data = dev(np.concatenate([np.zeros(shift, np.uint8)] + blocks))[shift:]

        def bufs():
            return [torch.zeros(n * k, dtype=d, device="cuda") for k, d in
                    ((256, torch.int32), (256 * P.CHUNKS, torch.int32), (256, torch.uint8),
                     (P.layout_bytes(), torch.uint8), (1, torch.int64), (1, torch.int32))]
        h1, c1, l1, y1, r1, s1 = one = bufs()
        P.histogram_chunks(data, off, h1, c1)
        P.code_lengths(h1, n, 11, l1, s1)
        P.build_layout(h1, l1, n, P.params(ans=True), y1, r1, s1)
        ref = np.stack([np.bincount(b, minlength=256) for b in blocks])
        assert np.array_equal(h1.cpu().numpy().reshape(n, 256), ref)
        assert np.array_equal(c1.cpu().numpy().reshape(n, P.CHUNKS, 256).sum(1), ref)
        two = bufs()
        P.plan_blocks(data, off, P.params(ans=True), *two)
        for a, b in zip(one, two):
            assert torch.equal(a, b)
