"""Real-valued pilots by FFT: forward and both adjoint halves against the FP64 oracle at every
transform length (N + K*L - 1 just at, just above and far below a power of two), one row, rows
that do not fill a block, more rows than fit the GPU at once; values that are not numbers, or
that overflow in the transforms, give what the direct sums give.

Tolerance: two transforms of log2 S <= 12 levels and a product, each level rounded to 2^-24:
relative 2-norm error below 30 x 2^-24 = 2e-6, NMSE 4e-12; the pilot gradient sums rows on top,
1e-11 for all."""
import numpy as np
import pytest
import torch

from oracle import pn_oracle as O

pytestmark = pytest.mark.gpu
TOL = 1e-11

# (A, N, K*L): S = 64 (smallest), 128, 256, 512, 1024, 2048, 4096; N + K*L - 1 = S and S + 1
SHAPES = [(1, 2, 1), (5, 33, 32), (9, 33, 33), (3, 65, 64), (17, 129, 128), (1, 200, 57),
          (40, 300, 213), (7, 1000, 25), (3, 1000, 26), (33, 1023, 1023), (2, 2047, 2047),
          (5, 2100, 1997), (3, 2100, 1998)]


def _c(rng, *shape):
    return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)


@pytest.mark.parametrize("A, N, KL", SHAPES)
def test_fft_matches_oracle(A, N, KL):
    import paper_2206_05506_gb300 as pk
    dev = torch.device("cuda", 0)
    rng = np.random.default_rng([A, N, KL])
    Y, G = _c(rng, 1, A, N), _c(rng, 1, A, 1, KL)
    th = rng.standard_normal(N).astype(np.float32)
    p = np.tanh(th.astype(np.float64))
    Yd, Gd, td = (torch.from_numpy(x).to(dev) for x in (Y, G, th))
    buf = torch.full((A * KL + 64,), complex(3.0, 3.0), dtype=torch.complex64, device=dev)
    H = buf[32:32 + A * KL].view(1, A, 1, KL)
    pk.estimate_real_pilot(Yd, td, 1, KL, out=H, pilot_map="tanh")
    dY, dth = pk.backward(td, Yd, Gd, 1, KL, pilot_map="tanh")
    assert O.nmse(H.cpu().numpy(), O.estimate_real_pilot(Y, p, 1, KL)) <= TOL
    rdY, rdp = O.adjoint(G, Y, p, 1, KL)
    assert O.nmse(dY.cpu().numpy(), rdY) <= TOL
    assert O.nmse(dth.cpu().numpy(), rdp * (1 - p ** 2)) <= TOL
    g = torch.cat([buf[:32], buf[-32:]])
    assert bool((g == complex(3.0, 3.0)).all()), "write outside H"


@pytest.mark.parametrize("A, N, KL", [(20000, 40, 20), (9000, 255, 60), (4001, 1023, 300), (1501, 2047, 100)])
def test_many_rows(A, N, KL):
    import paper_2206_05506_gb300 as pk
    dev = torch.device("cuda", 0)
    gen = torch.Generator(dev).manual_seed(N)
    Y = torch.randn(1, A, N, dtype=torch.complex64, device=dev, generator=gen)
    G = torch.randn(1, A, 1, KL, dtype=torch.complex64, device=dev, generator=gen)
    p = torch.randn(N, device=dev, generator=gen)
    H = pk.estimate_real_pilot(Y, p, 1, KL)
    dY, dp = pk.backward(p, Y, G, 1, KL)
    Yf = torch.fft.fft(Y[0].to(torch.complex128))
    Gf = torch.zeros(A, N, dtype=torch.complex128, device=dev)
    Gf[:, :KL] = G[0, :, 0]
    Gf = torch.fft.fft(Gf)
    pf = torch.fft.fft(p.to(torch.complex128))
    for got, want in ((H[0, :, 0], torch.fft.ifft(Yf * pf.conj())[:, :KL] / N),
                      (dY[0], torch.fft.ifft(Gf * pf) / N),
                      (dp, torch.fft.ifft((Gf.conj() * Yf).sum(0)).real / N)):
        err = torch.linalg.norm(got - want) / torch.linalg.norm(want)
        assert float(err) ** 2 <= TOL
    for a in (0, A // 2, A - 1):                # a row alone gives the same bits
        assert torch.equal(pk.estimate_real_pilot(Y[:, a:a + 1].clone(), p, 1, KL), H[:, a:a + 1])


def test_values_that_are_not_numbers_or_overflow():
    import paper_2206_05506_gb300 as pk
    dev = torch.device("cuda", 0)
    rng = np.random.default_rng(4)
    A, N, KL = 6, 200, 50
    Y, G = _c(rng, 1, A, N), _c(rng, 1, A, 1, KL)
    p = rng.standard_normal(N).astype(np.float32)
    Y[0, 0, 3] = complex(np.nan, 1)
    Y[0, 1, 9] = complex(1, np.inf)
    Y[0, 2] *= np.float32(3e37)                 # transforms overflow, and some of the sums
    G[0, 3, 0, 4] = complex(-np.inf, 0)
    G[0, 4, 0] *= np.float32(3e37)
    Yd, Gd, pd = (torch.from_numpy(x).to(dev) for x in (Y, G, p))
    H = pk.estimate_real_pilot(Yd, pd, 1, KL).cpu().numpy()[0, :, 0]
    dY, _ = pk.backward(pd, Yd, Gd, 1, KL, need_dp=False)
    dY = dY.cpu().numpy()[0]
    j, n = np.arange(KL), np.arange(N)
    P = p[(n[:, None] - j[None, :]) % N]
    with np.errstate(all="ignore"):
        # the direct sums, in FP32 and in order
        sums = [np.add.accumulate(f(Y[0])[:, :, None] * P, axis=1)[:, -1] / np.float32(N)
                for f in (np.real, np.imag)]
        adjs = [np.add.accumulate(f(G[0, :, 0])[:, None, :] * P, axis=2)[:, :, -1] / np.float32(N)
                for f in (np.real, np.imag)]
    for got, want in ((H.real, sums[0]), (H.imag, sums[1]), (dY.real, adjs[0]), (dY.imag, adjs[1])):
        assert np.array_equal(np.isnan(got), np.isnan(want))
        inf = np.isinf(want)
        assert np.array_equal(np.isinf(got), inf) and np.array_equal(np.sign(got[inf]), np.sign(want[inf]))
        for a in range(A):
            f = np.isfinite(want[a])
            if f.any():
                x, w = got[a][f].astype(np.float64), want[a][f].astype(np.float64)
                assert np.linalg.norm(x - w) <= 1e-5 * np.linalg.norm(w)
    # the pilot gradient: one sample that is no number reaches K*L of its N entries only
    Y = _c(rng, 1, A, N)
    G = _c(rng, 1, A, 1, KL)
    Y[0, 2, 100] = complex(np.nan, 0)
    _, dp = pk.backward(pd, torch.from_numpy(Y).to(dev), torch.from_numpy(G).to(dev), 1, KL,
                        need_dY=False)
    dp = dp.cpu().numpy()
    Y0 = Y.copy()
    Y0[0, 2, 100] = 0
    _, want = O.adjoint(G, Y0, p.astype(np.float64), 1, KL)
    hit = np.isin(n, (100 - j) % N)
    assert np.all(np.isnan(dp[hit])) and O.nmse(dp[~hit], want[~hit]) <= 1e-10
