"""GPU: the big blocks' chunks coded while the last whole blocks still run (batches of more
blocks than SMs), launched directly and from a captured graph: the same
records as the oracle's, whatever ran on the buffers before."""
import numpy as np
import pytest

from test_gpu_decode_edges import P, draw   # noqa: F401  (P: fixture)
from test_gpu_parity import dev, off64

pytestmark = pytest.mark.gpu


def batch(rng, n):
    """Every third block big (a level of it does not fit), in sizes that make its place in the list matter."""
    out = []
    for b in range(n):
        if b % 3 == 0:
            out.append(draw(rng, int(rng.integers(40000, 90000)), 0.1, 120))
        else:
            out.append(draw(rng, int(rng.integers(500, 9000)), 0.7, 2 + b % 50))
    return out


@pytest.mark.parametrize("ans", [False, True])
def test_overlapped_chunks(P, ans):   # noqa: F811
    import oracle
    import torch
    oracle.build()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 2 * sms + 1
    rng = np.random.default_rng(5)
    a, b = batch(rng, n), batch(rng, n)
    b = [np.resize(y, x.size) for x, y in zip(a, b[::-1])]   # the same sizes, other data
    off = np.concatenate([[0], np.cumsum([x.size for x in a])]).astype(np.uint64)
    boff = off64(off)
    refs = []
    for blocks in (a, b):
        refs.append(oracle.encode_batch(np.concatenate(blocks), off, oracle.params(ans=ans)))
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        data = dev(np.concatenate(a))
        e = P.Encoder(n, P.params(ans=ans))
        e.ensure(max(e.plan(dev(np.concatenate(x)), boff, stream) for x in (a, b)) + 64)
        e.run(data, boff, stream)
        stream.synchronize()
        g = P.Graph(stream)
        with g:
            e.run(data, boff, stream)
        for k in range(6):
            blocks, (ref, rec_off, sizes) = (a, b)[k % 2], refs[k % 2]
            data.copy_(dev(np.concatenate(blocks)))
            e.comp.fill_(0x5A)
            if k < 4:
                g.launch(stream)
            else:
                e.run(data, boff, stream)
            stream.synchronize()
            assert not e.status.cpu().numpy().any()
            comp, eo, rb = e.comp.cpu().numpy(), e.off.cpu().numpy(), e.rec_bytes.cpu().numpy()
            assert np.array_equal(rb, np.asarray(sizes, np.int64))
            for i in range(n):
                assert np.array_equal(comp[eo[i]:eo[i] + rb[i]],
                                      ref[int(rec_off[i]):int(rec_off[i]) + int(sizes[i])]), (k, i)
