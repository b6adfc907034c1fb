"""A pilot's tables are on the device when its creation returns: an estimate on a stream that does
not wait for the default stream may follow at once."""
import pytest
import torch

from synth import mseq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [10, 14])
def test_first_use_on_another_stream(r):
    import paper_2206_05506_gb300 as pk
    dev = torch.device("cuda", 0)
    side = torch.cuda.Stream(dev)                # (PyTorch's streams are non-blocking)
    bits = [mseq.mseq_bits(r, seed) for seed in range(4)]
    Y = torch.randn(1, 8, bits[0].size, dtype=torch.complex64, device=dev, generator=torch.Generator(dev).manual_seed(r))
    want = [pk.estimate(Y, pk.Pilot(b, device=dev), 1, 500).clone() for b in bits]
    torch.cuda.synchronize()
    for i in range(40):
        with torch.cuda.stream(side):
            pilot = pk.Pilot(bits[i % 4], device=dev)
            H = pk.estimate(Y, pilot, 1, 500)
        side.synchronize()
        assert torch.equal(H, want[i % 4])
