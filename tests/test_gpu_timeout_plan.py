"""GPU: a block's own item gives up waiting for its plan, and the plan comes
later all the same.  The batch has so many blocks that nearly every CTA of the
launch plans; the few that are left take the first blocks' items, whose
plans are not there yet.  Whatever the bound, a block that reports OK holds
its input."""
import numpy as np
import pytest

from test_gpu_decode_edges import draw
from test_gpu_timeout import P, TIMEOUT   # noqa: F401  (P: fixture)
from test_gpu_parity import dev, off64

pytestmark = pytest.mark.gpu


def test_late_plans(P):   # noqa: F811
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 8 * (4 * sms - 8)
    rng = np.random.default_rng(3)
    data = np.tile(draw(rng, 997, 0.5, 90), n)
    off = off64(997 * np.arange(n + 1))
    enc = P.encode(dev(data), off)
    assert not enc.status.cpu().numpy().any()
    dec = P.Decoder(n, "cuda", batched=True)
    dec.prepare(enc.comp, enc.off)
    out = torch.empty(data.size, dtype=torch.uint8, device="cuda")
    for limit in 4 * (2000, 4000, 6000, 8000, 9000, 10000, 11000, 12000, 16000, 20000):
        out.fill_(0x5A)
        P.set_wait_limit(limit)
        try:
            dec.run(enc.comp, enc.off, out, off)
            torch.cuda.synchronize()
        finally:
            P.set_wait_limit()
        st = dec.status.cpu().numpy()
        assert set(np.unique(st)) <= {0, TIMEOUT}
        same = (out.cpu().numpy().reshape(n, 997) == data.reshape(n, 997)).all(axis=1)
        assert same[st == 0].all(), (limit, np.flatnonzero((st == 0) & ~same)[:10])
    dec.run(enc.comp, enc.off, out, off)
    torch.cuda.synchronize()
    assert not dec.status.cpu().numpy().any() and np.array_equal(out.cpu().numpy(), data)
