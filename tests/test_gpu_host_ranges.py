"""Host buffers that are page-locked in pieces: neighbouring pieces are one buffer to the GPU; a
buffer with a hole between its page-locked ends is not read or written by a kernel.  (The copies
that it takes instead may refuse it, as CUDA documents for a copy over both kinds of memory.)"""
import mmap

import pytest
import torch

from synth import mseq

pytestmark = pytest.mark.gpu


class _Pieces:
    """`count` complex64 in pages of their own, of which the ranges [a, b) are page-locked
    (fractions of the buffer, rounded to pages)"""

    def __init__(self, count, ranges):
        page = mmap.PAGESIZE
        self.pages = (8 * count + page - 1) // page
        self.map = mmap.mmap(-1, self.pages * page)
        raw = torch.frombuffer(self.map, dtype=torch.uint8)
        self.x = raw[:8 * count].view(torch.complex64)
        self.locked = []
        for a, b in ranges:
            first, last = round(a * self.pages), round(b * self.pages)
            ptr = raw.data_ptr() + first * page
            assert int(torch.cuda.cudart().cudaHostRegister(ptr, (last - first) * page, 0)) == 0
            self.locked.append(ptr)

    def release(self):
        torch.cuda.synchronize()
        for ptr in self.locked:
            assert int(torch.cuda.cudart().cudaHostUnregister(ptr)) == 0


@pytest.mark.parametrize("ranges, hole", [([(0, 1)], False), ([(0, 0.25), (0.25, 0.5), (0.5, 1)], False),
                                          ([(0, 0.25), (0.75, 1)], True)])
@pytest.mark.parametrize("which", ["Y", "H"])
def test_buffers_in_pieces(which, ranges, hole):
    import paper_2206_05506_gb300 as pk
    dev = torch.device("cuda", 0)
    bits = mseq.mseq_bits(10, 0)
    M, N, K, L = 640, bits.size, 4, 128
    pilot = pk.Pilot(bits, device=dev)
    x = torch.randn(1, M, N, dtype=torch.complex64, generator=torch.Generator().manual_seed(1))
    want = pk.estimate(x.to(dev), pilot, K, L, dtype="fp16").cpu()
    pieces = _Pieces(M * (N if which == "Y" else K * L), ranges)
    try:
        if which == "Y":
            Y, H = pieces.x.view(1, M, N), torch.zeros(1, M, K, L, dtype=torch.complex64).pin_memory()
            Y.copy_(x)
        else:
            Y, H = x.pin_memory(), pieces.x.view(1, M, K, L)
            H.zero_()
        try:
            pk.estimate_host(Y, pilot, K, L, dtype="fp16", out=H)
            assert torch.equal(H, want)
        except pk.PnceError:
            assert hole
    finally:
        pieces.release()
    assert pk.get_status(dev) == 0
