"""Estimates that follow each other in a stream overlap their launches: each must still see what
the one before it wrote, and must not overwrite what it reads; also behind copies, event forks
and other estimates in a captured graph."""
import pytest
import torch

from synth import mseq

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


def _randn(seed, *shape):
    return torch.randn(*shape, dtype=torch.complex64, device=DEV, generator=torch.Generator(DEV).manual_seed(seed))


@pytest.mark.parametrize("dtype", ["fp32", "fp16"])
@pytest.mark.parametrize("r, A", [(7, 30000), (10, 6000), (12, 1500), (14, 400)])
def test_each_estimate_reads_the_one_before(r, A, dtype):
    # the result of one call (all N lags) is the input of the next, in two buffers in turn
    import paper_2206_05506_gb300 as pk
    bits = mseq.mseq_bits(r, 0)
    N, pilot = bits.size, pk.Pilot(bits, device=DEV)
    x = _randn(r, 1, A, N) * N ** 0.5

    def chain(wait):
        bufs = [torch.empty(1, A, 1, N, dtype=torch.complex64, device=DEV) for _ in range(2)]
        y = x
        for i in range(12):
            if wait:
                torch.cuda.synchronize()
            pk.estimate(y, pilot, 1, N, dtype=dtype, out=bufs[i % 2])
            y = bufs[i % 2].view(1, A, N)
        torch.cuda.synchronize()
        return y.clone()

    assert torch.equal(chain(False), chain(True))


@pytest.mark.parametrize("KL", [3, 200])
def test_input_rewritten_between_calls(KL):
    import paper_2206_05506_gb300 as pk
    bits = mseq.mseq_bits(11, 0)
    N, A, pilot = bits.size, 3000, pk.Pilot(bits, device=DEV)
    xs = [_randn(i, 1, A, N) for i in range(4)]
    want = [pk.estimate(x, pilot, 1, KL).clone() for x in xs]
    torch.cuda.synchronize()
    Y = torch.empty_like(xs[0])
    got = []
    for x in xs:
        Y.copy_(x)
        got.append(pk.estimate(Y, pilot, 1, KL))
    for a, b in zip(got, want):
        assert torch.equal(a, b)


def test_captured_chain():
    import paper_2206_05506_gb300 as pk
    bits = mseq.mseq_bits(10, 0)
    N, pilot = bits.size, pk.Pilot(bits, device=DEV)
    src = _randn(0, 40, 64, N)
    Y, Y2 = torch.empty_like(src), torch.empty_like(src)
    H, H2, Hc, H3 = (torch.empty(40, 64, 2, 100, dtype=torch.complex64, device=DEV) for _ in range(4))
    ws = torch.empty(pk.workspace_size(40, 64, N, 2, 100, "fp16"), dtype=torch.uint8, device=DEV)
    g, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(g):
        Y.copy_(src)
        pk.estimate(Y, pilot, 2, 100, out=H)
        pk.estimate(Y, pilot, 2, 100, dtype="fp16", out=H2, workspace=ws)
        cur = torch.cuda.current_stream()
        side.wait_stream(cur)
        with torch.cuda.stream(side):
            Hc.copy_(H2)
            Y2.copy_(Y)
        cur.wait_stream(side)
        pk.estimate(Y2, pilot, 2, 100, out=H3)
    for seed in (1, 2, 3):
        src.copy_(_randn(seed, 40, 64, N))
        g.replay()
        torch.cuda.synchronize()
        want = pk.estimate(src, pilot, 2, 100)
        assert torch.equal(H, want) and torch.equal(H3, want)
        assert torch.equal(Hc, pk.estimate(src, pilot, 2, 100, dtype="fp16"))
