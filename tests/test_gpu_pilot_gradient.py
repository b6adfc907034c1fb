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
