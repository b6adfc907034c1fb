"""Real-valued pilots by FFT over many rows, some of which hold values that are not finite or
overflow in the transforms: those rows give what the direct sums give, all others keep their
bits, and the call stays near the cost of the direct sums."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

# transform lengths 128 (rows share a warp) to 4096 (a row is a block)
SHAPES = [(9, 84, 45), (2500, 84, 40), (2500, 128, 128), (1500, 300, 200), (4096, 1023, 512), (600, 2047, 2047)]


def _median_ms(f, n=5):
    f()
    out = []
    for _ in range(n):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        f()
        b.record()
        b.synchronize()
        out.append(a.elapsed_time(b))
    return sorted(out)[n // 2]


@pytest.mark.parametrize("adjoint", [False, True])
@pytest.mark.parametrize("A, N, KL", SHAPES)
def test_rows_that_are_not_finite(A, N, KL, adjoint):
    # tolerance of the overflowing row: sums of at most 2047 products, each rounding below 2^-24
    # of a partial sum that is at most 50 times the result: relative error below 1e-4
    import paper_2206_05506_gb300 as pk
    dev = torch.device("cuda", 0)
    gen = torch.Generator(dev).manual_seed(N + KL)
    cols = KL if adjoint else N
    X = torch.randn(1, A, cols, dtype=torch.complex64, device=dev, generator=gen)
    p = torch.randn(N, device=dev, generator=gen)
    dummy = torch.empty(1, A, N, dtype=torch.complex64, device=dev)

    def call(X, p, pilot_map="real"):
        if adjoint:
            return pk.backward(p, dummy, X.view(1, A, 1, KL), 1, KL, need_dp=False, pilot_map=pilot_map)[0][0]
        return pk.estimate_real_pilot(X, p, 1, KL, pilot_map=pilot_map)[0, :, 0]

    clean = call(X, p)
    odd = X.clone()
    a_nan, a_inf, a_big = 0, A // 2, A - 1
    odd[0, a_nan, 3] = complex(float("nan"), 1)
    odd[0, a_inf, 5] = complex(1, float("-inf"))
    odd[0, a_big] *= 2e37
    got = call(odd, p)
    keep = torch.ones(A, dtype=torch.bool, device=dev)
    keep[[a_nan, a_inf, a_big]] = False
    assert torch.equal(got[keep], clean[keep])
    assert bool(torch.isnan(got[a_nan].real).all()) and bool(torch.isfinite(got[a_nan].imag).all())
    o = torch.arange(got.shape[1], device=dev)
    taps = p[(o - 5) % N] if adjoint else p[(5 - o) % N]
    assert torch.equal(got[a_inf].imag, -torch.sign(taps) * float("inf"))
    assert bool(torch.isfinite(got[a_inf].real).all())
    # the row whose transform overflows: finite where the direct sum in FP32 and in order is
    lag, n = np.arange(KL), np.arange(N)
    P = p.cpu().numpy()[(n[:, None] - lag[None, :]) % N]
    P = P.T if adjoint else P                                           # [terms, outputs]
    x, g = odd[0, a_big].cpu().numpy(), got[a_big].cpu().numpy()
    for part in (np.real, np.imag):
        with np.errstate(over="ignore", invalid="ignore"):
            fine = np.isfinite(np.add.accumulate(part(x)[:, None] * P, axis=0)[-1])
        assert np.array_equal(np.isfinite(part(g)), fine)
        want = (part(x).astype(np.float64) @ P.astype(np.float64) / N)[fine]
        assert np.linalg.norm(part(g)[fine] - want) <= 1e-4 * np.linalg.norm(want)
    # a pilot that holds a NaN reaches every lag, and the samples that have a part in it
    bad = p.clone()
    bad[N // 2] = float("nan")
    hit = (o - N // 2) % N < KL if adjoint else o >= 0
    for pilot_map in ("real", "tanh"):
        nan = torch.isnan(torch.view_as_real(call(X, bad, pilot_map)))
        if not adjoint or KL >= 128:
            assert torch.equal(nan, hit[None, :, None].expand_as(nan))
        else:               # (the dense kernel multiplies a tile's unused lags by zero: more NaN)
            assert bool(nan[:, hit].all())
        t0, t1 = (_median_ms(lambda: call(X, q, pilot_map)) for q in (p, bad))
        assert t1 <= 25 * t0
    assert torch.equal(call(X, p), clean)
