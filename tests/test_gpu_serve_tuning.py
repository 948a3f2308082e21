"""GPU: the tuning changed while requests are being served.

A request's items are taken by several launches of the serving loop (here
with epochs much shorter than a request), each with as many CTAs as the tuning
of its moment asks for.  Whatever it is, every request's bytes are its input:
requests of block counts between the two grids and on either side of them."""
import numpy as np
import pytest

from test_gpu_serve import P, _pinned   # noqa: F401  (P: fixture)
from test_gpu_parity import dev, off64

pytestmark = pytest.mark.gpu


def test_tuning_changes_while_serving(P):   # noqa: F811
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(17)
    items = []
    for nblk in (sms - 1, 2 * sms, 2 * sms + 1, 2 * sms + 96, 3 * sms, 4 * sms, 4 * sms + 1, 5 * sms):
        sizes = rng.integers(2000, 30000, nblk)
        off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
        data = rng.integers(1, 40, int(off[-1])).astype(np.uint8)
        data[rng.random(data.size) < 0.8] = 0
        enc = P.encode(dev(data), off64(off), P.params(ans=bool(nblk % 2), flat=True))
        assert not enc.status.cpu().numpy().any()
        items.append((_pinned(enc.comp.cpu().numpy()), enc.off.cpu().numpy().astype(np.uint64), off, data))
    arena = torch.empty(1 << 30, dtype=torch.uint8, device="cuda")
    try:
        for rep in range(6):
            outs = []
            with P.Server(arena, epoch_us=40) as srv:
                for comp, coff, off, data in items:
                    out = torch.zeros(data.size, dtype=torch.uint8, pin_memory=True)
                    outs.append((srv.submit(comp, coff, off, out), out, data))
                for k in range(4000):
                    P.set_tuning(ctas_per_sm=(2, 0, 1, 0)[k % 4])
                    if all(srv.poll(rid)[0] == P.DONE for rid, _, _ in outs):
                        break
                srv.drain(60000)
                for rid, out, data in outs:
                    assert srv.poll(rid)[:2] == (P.DONE, 0)
                    assert np.array_equal(out.numpy(), data)
    finally:
        P.set_tuning()
