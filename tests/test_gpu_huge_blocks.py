"""GPU: blocks whose records pass the bit addresses of the kernels.

Bitmaps that end within the first 2^28 bytes of a record decode; a record with
any later is refused by every decode call and by random access (whose walk
reads them without a limit of its own), and a block whose record would pass
2^29 bytes is refused by the encoder's plan."""
import numpy as np
import pytest

from test_gpu_decode_edges import P   # noqa: F401  (fixture)
from test_gpu_parity import off64

pytestmark = pytest.mark.gpu


def uniform(n):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    return torch.randint(0, 256, (n,), generator=g, device="cuda", dtype=torch.uint8)


# (uniform bytes: 8 bits a symbol; the largest block that decodes, and one just past it)
@pytest.mark.parametrize("n,want", [((1 << 28) - 4096, 0), ((1 << 28) + 4096, 1)])
@pytest.mark.parametrize("batched", [False, True])
def test_largest_record(P, n, want, batched):   # noqa: F811
    import torch
    data = uniform(n)
    enc = P.encode(data, off64([0, n]))
    assert int(enc.status.cpu()[0]) == 0
    assert (int(enc.rec_bytes.cpu()[0]) > 1 << 28) == bool(want)
    out, st = P.decode(enc.comp, enc.off, off64([0, n]), batched=batched)
    assert int(st.cpu()[0]) == (P.ERR_CORRUPT if want else 0)
    if not want:
        assert torch.equal(out[:n], data)
    access = P.Access(enc.comp, enc.off, 1)
    pos = torch.cat([torch.randint(0, n, (2000,), device="cuda"), torch.tensor([0, n - 1], device="cuda")]).to(torch.int32)
    if want:
        assert int(access.status.cpu()[0]) == P.ERR_CORRUPT
    sym, qst = access(torch.zeros_like(pos), pos)
    assert (qst == (P.ERR_CORRUPT if want else 0)).all()
    if not want:
        assert torch.equal(sym, data[pos.to(torch.int64)])


def test_too_large_for_the_encoder(P):   # noqa: F811
    n = (1 << 29) + 4096
    e = P.Encoder(1)
    e.plan(uniform(n), off64([0, n]))
    assert int(e.status.cpu()[0]) == P.ERR_INVALID_ARG
