"""Real-valued pilots short enough to be summed directly: the estimate of one sample is one
product per lag, exact but for the rounding of 1/N."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N, KL", [(2, 1), (31, 31), (60, 4), (61, 61), (64, 64), (83, 41)])
def test_one_sample_gives_exact_products(N, KL):
    # whole-numbered sample and pilot: the product is exact, 1/N and the product with it are
    # rounded to 2^-24 each
    import paper_2206_05506_gb300 as pk
    dev = torch.device("cuda", 0)
    rng = np.random.default_rng([N, KL])
    p = rng.integers(-3, 4, N).astype(np.float32)
    Y = np.zeros((1, 5, N), dtype=np.complex64)
    n = N - 1
    Y[0, 2, n] = 3 - 2j
    H = pk.estimate_real_pilot(torch.from_numpy(Y).to(dev), torch.from_numpy(p).to(dev), 1, KL)
    H = H.cpu().numpy()[0, :, 0].astype(np.complex128)
    want = np.zeros((5, KL), dtype=np.complex128)
    want[2] = Y[0, 2, n] * p[(n - np.arange(KL)) % N] / N
    for got, ref in ((H.real, want.real), (H.imag, want.imag)):
        assert np.all(np.abs(got - ref) <= 2.0 ** -23 * np.abs(ref))
