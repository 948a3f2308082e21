"""GPU: a plan and chunk histograms of older data of the same sizes.

The counts they give every node add up to the block, but a node with a leaf
on one side may be sent more symbols for the leaf and fewer for its other
child.  A block is then refused; only where every count is right after all
does it report OK, and its record decodes to the data."""
import numpy as np
import pytest

from test_gpu_decode_edges import P, draw   # noqa: F401  (P: fixture)
from test_gpu_parity import dev, off64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [(700, 9000, 15000), (30000, 20000)])   # (the second: enough blocks to code them whole)
@pytest.mark.parametrize("flat", [False, True])
def test_plan_of_older_data(P, sizes, flat):   # noqa: F811
    rng = np.random.default_rng(23)
    n = 160 if max(sizes) > 16000 else 12
    old = [draw(rng, sizes[b % len(sizes)], 0.6 + 0.02 * (b % 5), 3 + 5 * (b % 7)) for b in range(n)]
    new = []
    for b, x in enumerate(old):
        y = x.copy()
        if b % 4 == 0:      # some of the others become the most frequent symbol, whose leaf the root holds
            y[np.flatnonzero(y)[: 1 + b]] = 0
        elif b % 4 == 1:    # and the other way round
            y[np.flatnonzero(y == 0)[: 1 + b]] = 1
        elif b % 4 == 2:    # one symbol becomes another: a deeper node's counts
            k = np.flatnonzero(y == y.max())
            y[k[: max(1, k.size // 2)]] = 1
        else:
            y = rng.permutation(y)   # every block total is the same
        new.append(y)
    data0, data1 = np.concatenate(old), np.concatenate(new)
    off = np.concatenate([[0], np.cumsum([x.size for x in old])]).astype(np.uint64)
    e = P.Encoder(n, P.params(flat=flat))
    e.ensure(e.plan(dev(data0), off64(off)))
    enc = e.run(dev(data1), off64(off), replan=False)
    st = enc.status.cpu().numpy()
    assert set(np.unique(st)) <= {P.OK, P.ERR_INVALID_ARG}
    for b in range(n):
        # (the second kind may swap two leaves of one node: exact again)
        if b % 4 in (0, 1):
            assert st[b] == P.ERR_INVALID_ARG, b
    out, dst = P.decode(enc.comp, enc.off, off64(off))
    out, dst = out.cpu().numpy(), dst.cpu().numpy()
    for b in np.flatnonzero(st == P.OK):
        assert dst[b] == 0, b
        assert np.array_equal(out[int(off[b]):int(off[b + 1])], new[b]), b
    if max(sizes) > 16000:   # (coded whole: only the sums are used)
        assert (st[3::4] == P.OK).all()
