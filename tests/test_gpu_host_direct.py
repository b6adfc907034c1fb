"""Host estimates that read and write page-locked buffers over the link in one launch: the
device path's bits for one row, rows that do not fill a team, more rows than are in flight at
once, few lags, buffers that begin inside an allocation; one buffer page-locked and the other
not, and a pilot without a transform, which keep the chunked pipeline."""
import numpy as np
import pytest
import torch

from synth import mseq

pytestmark = pytest.mark.gpu


def _blocks(seed, *shape):
    return torch.randn(*shape, dtype=torch.complex64, generator=torch.Generator().manual_seed(seed))


def _pinned(x, lead=3):
    buf = torch.zeros(x.numel() + 2 * lead, dtype=torch.complex64).pin_memory()
    y = buf[lead:lead + x.numel()].view(x.shape)
    y.copy_(x)
    return buf, y


@pytest.mark.parametrize("r, F, M, K, L", [(7, 1, 1, 1, 1), (7, 70, 401, 3, 20), (8, 1, 3, 1, 200),
                                           (10, 5, 101, 2, 8), (11, 16, 63, 4, 128), (12, 3, 171, 1, 4095)])
@pytest.mark.parametrize("dtype", ["fp32", "fp16"])
def test_page_locked_buffers(r, F, M, K, L, dtype):
    import paper_2206_05506_gb300 as pk
    dev = torch.device("cuda", 0)
    bits = mseq.mseq_bits(r, 1)
    pilot = pk.Pilot(bits, device=dev)
    _, Y = _pinned(_blocks(r, F, M, bits.size))
    buf, H = _pinned(torch.zeros(F, M, K, L, dtype=torch.complex64))
    buf.fill_(complex(3.0, 3.0))
    pk.estimate_host(Y, pilot, K, L, dtype=dtype, out=H)
    assert torch.equal(H, pk.estimate(Y.to(dev), pilot, K, L, dtype=dtype).cpu())
    assert bool((torch.cat([buf[:3], buf[-3:]]) == complex(3.0, 3.0)).all()), "write outside H"


def test_other_buffers_and_pilots():
    import paper_2206_05506_gb300 as pk
    dev = torch.device("cuda", 0)
    bits = mseq.mseq_bits(10, 1)
    flipped = bits.copy()
    flipped[7] ^= 1
    x = _blocks(1, 4, 33, bits.size)
    for b in (bits, flipped):
        pilot = pk.Pilot(b, device=dev)
        want = pk.estimate(x.to(dev), pilot, 2, 40, dtype="fp32").cpu()
        for y_pinned in (False, True):
            for h_pinned in (False, True):
                Y = _pinned(x)[1] if y_pinned else x
                H = torch.zeros(4, 33, 2, 40, dtype=torch.complex64)
                H = _pinned(H)[1] if h_pinned else H
                pk.estimate_host(Y, pilot, 2, 40, dtype="fp32", out=H)
                assert torch.equal(H, want), (y_pinned, h_pinned)
