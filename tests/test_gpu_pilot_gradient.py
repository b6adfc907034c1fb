"""The pilot gradient where it is delicate: samples that are not numbers, which reach exactly
the entries whose sums they are part of, for lag counts around the kernels' steps (8 lags, a
chunk of 128) and for pilots shorter and longer than their windows; and, below 128 lags, the
dense sum's exactness."""
import numpy as np
import pytest
import torch

from oracle import pn_oracle as O

pytestmark = pytest.mark.gpu


def _c(rng, *shape):
    return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)


def _dp(p, Y, G, KL):
    import paper_2206_05506_gb300 as pk
    dev = torch.device("cuda", 0)
    Yd, Gd, pd = (torch.from_numpy(x).to(dev) for x in (Y, G, p))
    return pk.backward(pd, Yd, Gd, 1, KL, need_dY=False)[1].cpu().numpy()


@pytest.mark.parametrize("A, N, KL", [(3, 30, 1), (6, 200, 5), (4, 300, 40), (5, 600, 47), (2, 4200, 8),
                                      (3, 4100, 127), (2, 4096, 129), (700, 4500, 131)])
def test_a_sample_that_is_no_number_reaches_its_own_entries(A, N, KL):
    # tolerance of the others: sums of A K L products in FP32, partial sums of at most 2^13
    # terms in order: relative error far below 1e-5
    rng = np.random.default_rng([A, N, KL])
    Y, G, p = _c(rng, 1, A, N), _c(rng, 1, A, 1, KL), rng.standard_normal(N).astype(np.float32)
    at = N // 2
    Y[0, A - 1, at] = complex(0, np.nan)
    dp = _dp(p, Y, G, KL)
    Y[0, A - 1, at] = 0
    want = O.adjoint(G, Y, p.astype(np.float64), 1, KL)[1]
    hit = np.isin(np.arange(N), (at - np.arange(KL)) % N)
    assert np.array_equal(np.isnan(dp), hit)
    if not hit.all():
        assert O.nmse(dp[~hit], want[~hit]) <= 1e-10


@pytest.mark.parametrize("N, KL", [(60, 48), (200, 64), (300, 100), (1023, 127), (2047, 48)])
def test_few_lags_are_summed_directly(N, KL):
    # one gradient that is not zero and whole-numbered samples: every entry is one product, so
    # it is exact but for 1/N and the product with it, 2^-24 each, and zero where the sample is
    rng = np.random.default_rng([N, KL])
    A, a, j = 3, 1, KL - 2
    Y = (rng.integers(-4, 5, (1, A, N)) + 1j * rng.integers(-4, 5, (1, A, N))).astype(np.complex64)
    G = np.zeros((1, A, 1, KL), dtype=np.complex64)
    G[0, a, 0, j] = 1
    dp = _dp(rng.standard_normal(N).astype(np.float32), Y, G, KL).astype(np.float64)
    want = np.roll(Y[0, a].real.astype(np.float64), -j) / N
    assert np.all(np.abs(dp - want) <= 2.0 ** -23 * np.abs(want))


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


@pytest.mark.parametrize("A, N, KL", [(1, 128, 128), (7, 129, 128), (3000, 200, 130), (2500, 1023, 256),
                                      (700, 2047, 512)])
def test_values_that_are_not_finite_by_transform(A, N, KL):
    # A row whose transform overflows while its products do not; a sample that is no number;
    # infinities; a gradient that is no number.  The entries that these reach are what the
    # direct sum gives, the others are the oracle's (tolerance as in test_gpu_fft), and none of
    # it costs more than the direct sums of the blocks concerned: 2 A N K L operations, far
    # below a hundred times the transforms' time.
    import paper_2206_05506_gb300 as pk
    dev = torch.device("cuda", 0)
    gen = torch.Generator(dev).manual_seed(N)
    Y = torch.randn(1, A, N, dtype=torch.complex64, device=dev, generator=gen)
    G = torch.randn(1, A, 1, KL, dtype=torch.complex64, device=dev, generator=gen)
    p = torch.randn(N, device=dev, generator=gen)

    def dp(Y, G):
        return pk.backward(p, Y, G, 1, KL, need_dY=False)[1]

    def want(Y, G):
        Gf = torch.zeros(A, N, dtype=torch.complex128, device=dev)
        Gf[:, :KL] = G[0, :, 0]
        cross = (torch.fft.fft(Gf).conj() * torch.fft.fft(Y[0].to(torch.complex128))).sum(0)
        return torch.fft.ifft(cross).real / N

    def close(a, b):
        return float(torch.linalg.norm(a - b) / torch.linalg.norm(b)) ** 2 <= 1e-11

    n, at, a = torch.arange(N, device=dev), N // 3, A - 1
    hit = torch.isin(n, (at - torch.arange(KL, device=dev)) % N)
    clean = want(Y, G)
    t0 = _median_ms(lambda: dp(Y, G))
    # overflow of the transform alone: partial sums of up to K L numbers near 3e38 / 8
    big, small = G.clone(), Y.clone()
    big[0, a] *= 4e37
    small[0, a] *= 1e-30
    assert close(dp(small, big), want(small, big))
    # one sample that is no number, one that is infinite
    for v in (complex(0, float("nan")), complex(float("inf"), 0)):
        odd = Y.clone()
        odd[0, a, at] = v
        got = dp(odd, G)
        assert torch.equal(torch.isfinite(got), ~hit)
        assert torch.equal(torch.isnan(got), hit & bool(np.isnan(v.imag)))
        if v.real:
            j = (at - n[hit]) % N
            assert torch.equal(torch.sign(got[hit]), torch.sign(G[0, a, 0, j].real))
        odd[0, a, at] = 0
        if not bool(hit.all()):
            assert close(got[~hit], want(odd, G)[~hit])
    # gradients that are no numbers, in one row and in all of them
    for rows in (slice(a, A), slice(0, A)):
        odd = G.clone()
        odd[0, rows, 0, 1] = complex(float("nan"), 0)
        assert bool(torch.isnan(dp(Y, odd)).all())
        assert _median_ms(lambda: dp(Y, odd)) <= 100 * t0
    assert close(dp(Y, G), clean)                # nothing is left behind in the workspace
