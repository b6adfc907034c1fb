"""FP32 estimates of m-sequence pilots take the fast transform kernel: against the FP64 oracle
for every degree it takes, at the edges of its row teams (one row, a half-filled team, more
rows than fit the GPU at once), the smallest and the largest lag counts it gets, rows with a
prefix and spread shifts; samples that are not numbers; a pilot with one bit flipped, which
keeps the dense kernel.

Tolerance: every output is a sum of N terms +-y over r levels of additions, each rounded to
2^-24 of a partial sum: relative 2-norm error at most about r 2^-24, NMSE (14 2^-24)^2 = 7e-13;
1e-11 leaves room for partial sums that exceed the result."""
import numpy as np
import pytest
import torch

from oracle import pn_oracle as O
from synth import mseq

pytestmark = pytest.mark.gpu
TOL = 1e-11


def _y(rng, *shape):
    return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)


@pytest.mark.parametrize("A, KL", [(1, 33), (2, -1), (3, 40), (37, 64)])
@pytest.mark.parametrize("r", range(7, 15))
def test_fp32_transform_matches_oracle(r, A, KL):
    import paper_2206_05506_gb300 as pk
    dev = torch.device("cuda", 0)
    bits = mseq.mseq_bits(r, 1)
    N = bits.size
    KL = N if KL < 0 else KL
    rng = np.random.default_rng([r, A])
    cp = 5 if A == 37 else 0
    Y = _y(rng, 1, A, N + cp)
    pilot = pk.Pilot(bits, device=dev)
    Yd = torch.from_numpy(Y).to(dev)
    buf = torch.full((A * KL + 64,), complex(3.0, 3.0), dtype=torch.complex64, device=dev)
    H = buf[32:32 + A * KL].view(1, A, 1, KL)
    pk.estimate(Yd, pilot, 1, KL, dtype="fp32", out=H, cp_len=cp)
    ref = O.estimate_fft(Y[..., cp:], bits, 1, KL)
    assert O.nmse(H.cpu().numpy(), ref) <= TOL
    g = torch.cat([buf[:32], buf[-32:]])
    assert bool((g == complex(3.0, 3.0)).all()), "write outside H"
    if A == 37:                                   # spread shifts, several transmitters
        H = pk.estimate(Yd, pilot, 3, 21, dtype="fp32", cp_len=cp, shift_rule="spread")
        ref = O.estimate_general(Y, bits, 3, 21, cp_len=cp, shifts=np.arange(3) * (N // 3))
        assert O.nmse(H.cpu().numpy(), ref) <= TOL


@pytest.mark.parametrize("r, A", [(7, 20011), (8, 12001), (9, 8003), (10, 4001), (11, 2003), (12, 1009)])
def test_rows_beyond_one_wave(r, A):
    # every row alone gives the bits it gives in the batch, on a sample of the rows
    import paper_2206_05506_gb300 as pk
    dev = torch.device("cuda", 0)
    bits = mseq.mseq_bits(r, 0)
    N, KL = bits.size, 50
    gen = torch.Generator(dev).manual_seed(r)
    Y = torch.randn(1, A, N, dtype=torch.complex64, device=dev, generator=gen)
    pilot = pk.Pilot(bits, device=dev)
    H = pk.estimate(Y, pilot, 1, KL, dtype="fp32")
    rows = [0, 1, A // 2, A - 2, A - 1]
    ref = O.estimate(Y[:, rows].cpu().numpy(), bits, 1, KL)
    assert O.nmse(H[:, rows].cpu().numpy(), ref) <= TOL
    for a in rows:
        assert torch.equal(pk.estimate(Y[:, a:a + 1].clone(), pilot, 1, KL, dtype="fp32"), H[:, a:a + 1])


@pytest.mark.parametrize("r", [7, 10, 12])
def test_samples_that_are_not_numbers(r):
    # as in the sum that defines the estimate: a NaN reaches every lag of its part, an
    # infinity takes the pilot's sign at every lag, opposite infinities give NaN
    import paper_2206_05506_gb300 as pk
    dev = torch.device("cuda", 0)
    bits = mseq.mseq_bits(r, 0)
    N, KL = bits.size, 70
    Y = _y(np.random.default_rng(r), 1, 5, N)
    Y[0, 0, 3] = complex(np.nan, 1.0)
    Y[0, 1, 4] = complex(2.0, np.inf)
    Y[0, 2, N - 1] = complex(-np.inf, 0.5)
    Y[0, 3, [5, 9]] = complex(np.inf, 1.0)
    H = pk.estimate(torch.from_numpy(Y).to(dev), pk.Pilot(bits, device=dev), 1, KL,
                    dtype="fp32").cpu().numpy()[0, :, 0]
    p = 1.0 - 2.0 * bits
    P = np.stack([np.roll(p, j) for j in range(KL)], axis=1)
    with np.errstate(invalid="ignore"):
        want = np.stack([(Y[0].real[:, :, None] * P).sum(1), (Y[0].imag[:, :, None] * P).sum(1)])
    for got, w in ((H.real, want[0]), (H.imag, want[1])):
        assert np.array_equal(np.isnan(got), np.isnan(w))
        inf = np.isinf(w)
        assert np.array_equal(np.isinf(got), inf) and np.array_equal(np.sign(got[inf]), np.sign(w[inf]))
        fine = np.isfinite(w)
        assert np.allclose(got[fine], w[fine] / N, rtol=0, atol=1e-5)


def test_other_bits_keep_the_dense_kernel():
    import paper_2206_05506_gb300 as pk
    dev = torch.device("cuda", 0)
    bits = mseq.mseq_bits(10, 0).copy()
    bits[100] ^= 1
    Y = _y(np.random.default_rng(3), 2, 9, bits.size)
    H = pk.estimate(torch.from_numpy(Y).to(dev), pk.Pilot(bits, device=dev), 2, 64, dtype="fp32")
    assert O.nmse(H.cpu().numpy(), O.estimate(Y, bits, 2, 64)) <= TOL


@pytest.mark.parametrize("dtype", ["fp16", "bf16", "e4m3", "tf32"])
@pytest.mark.parametrize("r", range(7, 15))
def test_reduced_formats_in_one_launch(r, dtype, monkeypatch):
    # rounding in registers gives the bits that quantise-then-correlate gives, both are the
    # FP64 estimate of the quantised operand, and the tensor cores agree to their accumulation;
    # powers over decades, zero rows, samples that are not numbers
    import paper_2206_05506_gb300 as pk
    dev = torch.device("cuda", 0)
    bits = mseq.mseq_bits(r, 2)
    N, A, K, L = bits.size, 11, 3, 19
    rng = np.random.default_rng([r, 5])
    Y = _y(rng, 1, A, N) * np.logspace(-4, 4, A, dtype=np.float32)[None, :, None]
    Y[0, 4] = 0
    pilot = pk.Pilot(bits, device=dev)
    Yd = torch.from_numpy(Y).to(dev)
    H = pk.estimate(Yd, pilot, K, L, dtype=dtype)
    q = pk.quantize(Yd, dtype)
    assert torch.equal(pk.correlate_quantized(q["workspace"], pilot, 1, A, K, L, dtype), H)
    ref = O.estimate_quantized(Y, bits, K, L, dtype)
    assert O.nmse(H.cpu().numpy(), ref) <= TOL
    Ys = torch.cat([torch.zeros(1, A, 4, dtype=torch.complex64, device=dev), Yd], dim=2)
    Hs = pk.estimate(Ys, pilot, K, L, dtype=dtype, cp_len=4, shift_rule="spread")
    odd = Yd.clone()
    odd[0, 0, 3], odd[0, 1, 7], odd[0, 2, N - 1] = complex(float("nan"), 1), complex(0, float("inf")), complex(float("-inf"), 2)
    Ho = pk.estimate(odd, pilot, K, L, dtype=dtype)
    monkeypatch.setenv("PNCE_TC_FORCE", "1")                 # the tensor-core kernels
    Ht = pk.estimate(Yd, pilot, K, L, dtype=dtype)
    assert O.nmse(Ht.cpu().numpy(), ref) <= 1e-9
    assert O.nmse(Hs.cpu().numpy(), pk.estimate(Ys, pilot, K, L, dtype=dtype, cp_len=4,
                                                shift_rule="spread").cpu().numpy()) <= 1e-9
    Hto = torch.view_as_real(pk.estimate(odd, pilot, K, L, dtype=dtype))
    Ho = torch.view_as_real(Ho)
    assert torch.equal(torch.isnan(Ho), torch.isnan(Hto))
    assert torch.equal(torch.isinf(Ho), torch.isinf(Hto))
    assert torch.equal(torch.sign(Ho[torch.isinf(Ho)]), torch.sign(Hto[torch.isinf(Hto)]))
    assert pk.get_status(dev) == 0


@pytest.mark.parametrize("dtype", ["fp16", "bf16", "e4m3", "tf32"])
def test_other_bits_keep_the_tensor_cores(dtype):
    import paper_2206_05506_gb300 as pk
    dev = torch.device("cuda", 0)
    for r, F, M, K, L in [(7, 1, 8, 2, 16), (10, 3, 100, 5, 60), (12, 2, 64, 16, 128)]:
        bits = mseq.mseq_bits(r, 0).copy()
        bits[5] ^= 1
        Y = _y(np.random.default_rng(r), F, M, bits.size)
        H = pk.estimate(torch.from_numpy(Y).to(dev), pk.Pilot(bits, device=dev), K, L, dtype=dtype)
        assert O.nmse(H.cpu().numpy(), O.estimate_quantized(Y, bits, K, L, dtype)) <= 1e-9


@pytest.mark.parametrize("dtype", ["fp32", "fp16", "e4m3"])
def test_traced_calls_give_the_same_bits(dtype):
    import paper_2206_05506_gb300 as pk
    dev = torch.device("cuda", 0)
    bits = mseq.mseq_bits(11, 0)
    pilot = pk.Pilot(bits, device=dev)
    Y = torch.from_numpy(_y(np.random.default_rng(1), 2, 21, bits.size)).to(dev)
    H = pk.estimate(Y, pilot, 4, 50, dtype=dtype)
    pk.trace_enable(True, dev)
    Ht = pk.estimate(Y, pilot, 4, 50, dtype=dtype)
    kinds = [k for k, _ in pk.trace_read(dev)]
    pk.trace_enable(False, dev)
    assert torch.equal(H, Ht)
    assert kinds == (["simt"] if dtype == "fp32" else ["quantize", "correlate"])


@pytest.mark.parametrize("r, few", [(7, 8), (8, 8), (9, 8), (10, 16), (11, 32), (12, 32), (13, 32), (14, 32)])
def test_few_lags(r, few):
    # one lag, odd counts, the largest count of the few-lags form and the next one; rows that
    # do not fill a team, rows with a prefix, spread shifts, rounded samples
    import paper_2206_05506_gb300 as pk
    dev = torch.device("cuda", 0)
    bits = mseq.mseq_bits(r, 2)
    N, A, cp = bits.size, 21, 3
    Y = _y(np.random.default_rng(r), 1, A, N + cp)
    pilot = pk.Pilot(bits, device=dev)
    Yd = torch.from_numpy(Y).to(dev)
    ref = O.estimate_fft(Y[..., cp:], bits, 1, few + 1).reshape(A, -1)
    Yc = Yd[..., cp:].contiguous()
    for KL in (1, 2, 3, 5, few - 1, few, few + 1):
        buf = torch.full((A * KL + 64,), complex(3.0, 3.0), dtype=torch.complex64, device=dev)
        H = buf[32:32 + A * KL].view(1, A, 1, KL)
        pk.estimate(Yd, pilot, 1, KL, dtype="fp32", out=H, cp_len=cp)
        assert O.nmse(H.cpu().numpy().reshape(A, KL), ref[:, :KL]) <= TOL
        g = torch.cat([buf[:32], buf[-32:]])
        assert bool((g == complex(3.0, 3.0)).all()), "write outside H"
        assert torch.equal(pk.estimate(Yc[:, 2:3].clone(), pilot, 1, KL, dtype="fp32"), H[:, 2:3])
        for dtype in ("fp16", "e4m3"):
            q = pk.quantize(Yc, dtype)
            Hq = pk.correlate_quantized(q["workspace"], pilot, 1, A, 1, KL, dtype)
            assert torch.equal(pk.estimate(Yc, pilot, 1, KL, dtype=dtype), Hq)
            assert O.nmse(Hq.cpu().numpy(), O.estimate_quantized(Y[..., cp:], bits, 1, KL, dtype)) <= TOL
    H = pk.estimate(Yd, pilot, 3, 2, dtype="fp32", cp_len=cp, shift_rule="spread")
    want = O.estimate_general(Y, bits, 3, 2, cp_len=cp, shifts=np.arange(3) * (N // 3))
    assert O.nmse(H.cpu().numpy(), want) <= TOL


@pytest.mark.parametrize("dtype", ["fp16", "bf16", "e4m3", "tf32"])
def test_rounding_at_the_edges_of_the_formats(dtype):
    # samples half-way between two numbers of the format, down into its subnormals and below;
    # peaks whose scale is clamped at either end, denormal rows: the quantiser's bits
    import paper_2206_05506_gb300 as pk
    dev = torch.device("cuda", 0)
    bits = mseq.mseq_bits(9, 0)
    N = bits.size
    rng = np.random.default_rng(1)
    x = rng.integers(1, 1 << 13, (2, N)).astype(np.float64) * 2.0 ** rng.integers(-44, 3, (2, N))
    x *= rng.choice([-1.0, 1.0], (2, N))
    rows = [(x[0] + 1j * x[1]) * s for s in (1.0, 2.0 ** -14, 2.0 ** -120, 2.0 ** 100, 2.0 ** 110)]
    rows.append(_y(rng, N) * 1e-42)
    rows.append(np.full(N, 3e38 + 1e-38j))
    Y = torch.from_numpy(np.stack(rows).astype(np.complex64)[None]).to(dev)
    pilot = pk.Pilot(bits, device=dev)
    for K, L in ((3, 40), (1, 5)):
        H = pk.estimate(Y, pilot, K, L, dtype=dtype)
        q = pk.quantize(Y, dtype)
        Hq = pk.correlate_quantized(q["workspace"], pilot, 1, len(rows), K, L, dtype)
        a, b = torch.view_as_real(H), torch.view_as_real(Hq)
        assert torch.equal(torch.isnan(a), torch.isnan(b))
        assert torch.equal(torch.nan_to_num(a), torch.nan_to_num(b))


@pytest.mark.parametrize("dtype, KL", [("fp16", 500), ("bf16", 30), ("e4m3", 500), ("tf32", 250)])
def test_large_operands_with_few_lags(dtype, KL):
    # the correlation step alone, on either side of 2^22 samples: the transform's bits below, the
    # tensor cores above (their truncated accumulation: relative error 1e-5, NMSE 1e-10)
    import paper_2206_05506_gb300 as pk
    dev = torch.device("cuda", 0)
    bits = mseq.mseq_bits(9, 0)
    N, pilot = bits.size, pk.Pilot(bits, device=dev)
    for A in (8207, 8209):                       # 8208 x 511 > 2^22 > 8207 x 511
        Y = torch.randn(1, A, N, dtype=torch.complex64, device=dev, generator=torch.Generator(dev).manual_seed(A))
        H = pk.estimate(Y, pilot, 1, KL, dtype=dtype)
        q = pk.quantize(Y, dtype)
        Hq = pk.correlate_quantized(q["workspace"], pilot, 1, A, 1, KL, dtype)
        assert torch.equal(H, Hq) if A * N < 1 << 22 else O.nmse(Hq.cpu().numpy(), H.cpu().numpy()) <= 1e-10
    assert pk.get_status(dev) == 0


@pytest.mark.parametrize("r, KL", [(7, 8), (10, 3), (12, 32)])
def test_few_lags_of_samples_that_are_not_numbers(r, KL):
    import paper_2206_05506_gb300 as pk
    dev = torch.device("cuda", 0)
    bits = mseq.mseq_bits(r, 0)
    N = bits.size
    Y = _y(np.random.default_rng(r), 1, 5, N)
    Y[0, 0, 3] = complex(np.nan, 1.0)
    Y[0, 1, 4] = complex(2.0, np.inf)
    Y[0, 2, N - 1] = complex(-np.inf, 0.5)
    Y[0, 3, [5, 9]] = complex(np.inf, 1.0)
    H = pk.estimate(torch.from_numpy(Y).to(dev), pk.Pilot(bits, device=dev), 1, KL,
                    dtype="fp32").cpu().numpy()[0, :, 0]
    P = np.stack([np.roll(1.0 - 2.0 * bits, j) for j in range(KL)], axis=1)
    with np.errstate(invalid="ignore"):
        want = np.stack([(Y[0].real[:, :, None] * P).sum(1), (Y[0].imag[:, :, None] * P).sum(1)])
    for got, w in ((H.real, want[0]), (H.imag, want[1])):
        assert np.array_equal(np.isnan(got), np.isnan(w))
        inf, fine = np.isinf(w), np.isfinite(w)
        assert np.array_equal(np.isinf(got), inf) and np.array_equal(np.sign(got[inf]), np.sign(w[inf]))
        assert np.allclose(got[fine], w[fine] / N, rtol=0, atol=1e-5)
