"""The kernels of pilots without a fast transform: the tensor-core and dense FP32 estimates, their
batches, the chunked host pipeline and the native loop's graphs, with m-sequences of which one
bit is flipped (no m-sequence any more), and the tensor-core kernels at full size under
PNCE_TC_FORCE.

Tolerances (NMSE): tensor-core formats against the FP64 estimate of the quantised operand as in
test_gpu_parity; dense FP32 1e-10: N <= 16383 additions in order, each rounded to 2^-24 of a
partial sum that grows as its root, give a relative error of about 2^-25 sqrt(N) / 2 = 2e-6."""
import ctypes as C_

import numpy as np
import pytest
import torch

from oracle import pn_oracle as O
from synth import channel as C
from synth import mseq
from synth import serving as S

pytestmark = pytest.mark.gpu

TOL_Q = {"tf32": 1e-9, "fp16": 1e-9, "bf16": 1e-9, "e4m3": 1e-6, "fp32": 1e-10}
TC = ["fp16", "bf16", "e4m3", "tf32"]
ALL = ["fp32"] + TC
DEV = torch.device("cuda", 0)


@pytest.fixture(scope="module")
def pk():
    import paper_2206_05506_gb300 as pk
    pk.lib()
    return pk


def _flipped(r):
    bits = mseq.mseq_bits(r, 0).copy()
    bits[3 * bits.size // 7] ^= 1
    return bits


def _y(rng, *shape):
    return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)


def _reference(Y, bits, K, L, dtype, **kw):
    Y = np.ascontiguousarray(Y)
    Y = Y if dtype == "fp32" else O.dequantize(*O.quantize(Y, dtype))
    return O.estimate_general(Y, bits, K, L, **kw)


# the shapes of test_gpu_parity with N >= 127, few lags, a long sequence
@pytest.mark.parametrize("dtype", ALL)
@pytest.mark.parametrize("r, M, K, L, F", [(7, 8, 2, 16, 1), (10, 100, 5, 60, 3), (12, 64, 16, 128, 2),
                                           (8, 65, 3, 85, 1), (9, 33, 1, 20, 2), (12, 40, 1, 1, 1),
                                           (14, 9, 4, 256, 1)])
def test_estimates(pk, r, M, K, L, F, dtype):
    bits = _flipped(r)
    Y = _y(np.random.default_rng([r, M]), F, M, bits.size)
    buf = torch.full((F * M * K * L + 64,), complex(3.0, 3.0), dtype=torch.complex64, device=DEV)
    H = buf[32:-32].view(F, M, K, L)
    pilot = pk.Pilot(bits, device=DEV)
    Yd = torch.from_numpy(Y).to(DEV)
    pk.estimate(Yd, pilot, K, L, dtype=dtype, out=H)
    assert pk.get_status(DEV) == 0
    assert O.nmse(H.cpu().numpy(), _reference(Y, bits, K, L, dtype)) <= TOL_Q[dtype]
    assert bool((torch.cat([buf[:32], buf[-32:]]) == complex(3.0, 3.0)).all()), "write outside H"
    part = pk.estimate(Yd[F - 1:].clone(), pilot, K, L, dtype=dtype)
    assert torch.equal(part, H[F - 1:])              # independent of the rest of the batch
    if dtype != "fp32":
        q = pk.quantize(Yd, dtype)
        assert torch.equal(pk.correlate_quantized(q["workspace"], pilot, F, M, K, L, dtype), H)


@pytest.mark.parametrize("dtype", ALL)
@pytest.mark.parametrize("rule", ["kl", "spread"])
@pytest.mark.parametrize("r, M, K, L, cp, F", [(7, 3, 3, 20, 20, 2), (10, 37, 4, 100, 100, 2), (9, 5, 3, 45, 50, 1),
                                               (11, 4, 3, 300, 300, 1), (11, 16, 4, 128, 128, 4)])
def test_layouts(pk, r, M, K, L, cp, F, rule, dtype):
    bits = _flipped(r)
    N = bits.size
    if rule == "kl" and K * L > N:
        pytest.skip("K*L > N")
    Y = _y(np.random.default_rng([r, M]), F, M, cp + N)
    H = pk.estimate(torch.from_numpy(Y).to(DEV), pk.Pilot(bits, device=DEV), K, L, dtype=dtype, cp_len=cp,
                    shift_rule=rule)
    assert pk.get_status(DEV) == 0
    sh = (C.shifts_kl if rule == "kl" else C.shifts_spread)(K, L, N)
    ref = _reference(Y[..., cp:], bits, K, L, dtype, shifts=sh)
    assert O.nmse(H.cpu().numpy(), ref) <= TOL_Q[dtype]


@pytest.mark.parametrize("host", [False, True])
@pytest.mark.parametrize("kl_max", [20, 200, 1000])
@pytest.mark.parametrize("dtype", ALL)
def test_batches(pk, dtype, kl_max, host):
    from paper_2206_05506_gb300 import _lib
    bits = _flipped(10)
    N, pilot = bits.size, pk.Pilot(bits, device=DEV)
    rng = np.random.default_rng(kl_max)
    specs = [(5, 2, kl_max // 2), (64, 4, kl_max // 8), (1, 1, 1), (130, 1, kl_max), (7, 5, kl_max // 5)]
    rows = 256
    place = (lambda t: t.pin_memory()) if host else (lambda t: t.to(DEV))
    tab = torch.zeros((len(specs) + 1) * C_.sizeof(_lib.ReqDesc), dtype=torch.uint8).pin_memory()
    arr = (_lib.ReqDesc * (len(specs) + 1)).from_address(tab.data_ptr())
    reqs, off = [], 0
    for d, (M, K, L) in zip(arr, specs):
        Y = place(torch.from_numpy(_y(rng, M, N)))
        H = place(torch.full((M, K * L), complex(5.0, 5.0), dtype=torch.complex64))
        d.Y, d.H, d.M, d.K, d.L, d.row_offset = Y.data_ptr(), H.data_ptr(), M, K, L, off
        off += M
        reqs.append((M, K, L, Y, H))
    ws = torch.empty(pk.grouped_workspace_size(rows, N, kl_max, dtype), dtype=torch.uint8, device=DEV)
    pk.estimate_grouped(pilot, tab.data_ptr(), len(specs) + 1, rows, kl_max, dtype, ws)
    torch.cuda.synchronize()
    assert pk.get_status(DEV) == 0
    for M, K, L, Y, H in reqs:
        one = pk.estimate(Y.to(DEV).view(1, M, N), pilot, K, L, dtype=dtype).cpu().numpy()
        got = H.cpu().numpy().reshape(1, M, K, L)
        ref = _reference(Y.cpu().numpy()[None], bits, K, L, dtype)
        assert O.nmse(got, ref) <= TOL_Q[dtype]
        # (few lags of a request alone: an FP32 kernel of their own, in another order)
        if dtype != "fp32" or K * L > 32:
            assert np.array_equal(got, one)


@pytest.mark.parametrize("dtype", ["fp16", "fp32", "e4m3"])
def test_native_loop(pk, dtype):
    # two passes: the second one replays the graphs that the first one captured
    from paper_2206_05506_gb300 import serve
    pool = S.payload_pool(slots=2, seed=4)
    pinned = {k: torch.from_numpy(v).pin_memory() for k, v in pool.items()}

    def bits_of(N):
        return _flipped(N.bit_length())

    specs = S.poisson_trace(20000.0, 0.01, seed=31, payload_slots=2)
    out = torch.zeros(sum(s.M * s.K * s.L for s in specs), dtype=torch.complex64).pin_memory()
    nat = serve.NativeServer(bits_of, device=DEV, dtype=dtype, slots=3)
    for _ in range(2):
        out.zero_()
        reqs, off = [], 0
        for s in specs:
            reqs.append(serve.Request(s.rid, s.t_arrival, s.M, s.N, s.K, s.L,
                                      pinned[(s.M, s.N)].data_ptr() + s.slot * s.M * s.N * 8,
                                      out.data_ptr() + off * 8))
            off += s.M * s.K * s.L
        st = nat.run(reqs)
        assert st["requests"] == len(reqs) and st["failed"] == 0
        off = 0
        for s in specs:
            n = s.M * s.K * s.L
            if s.rid % 5 == 0:
                Y = pool[(s.M, s.N)][[s.slot]]
                ref = _reference(Y, bits_of(s.N), s.K, s.L, dtype)
                assert O.nmse(out[off:off + n].numpy().reshape(ref.shape), ref) <= TOL_Q[dtype]
            off += n


@pytest.mark.parametrize("pinned", [True, False])
@pytest.mark.parametrize("dtype", ALL)
@pytest.mark.parametrize("r, M, K, L, F", [(7, 8, 2, 16, 3), (10, 37, 4, 100, 13), (12, 130, 8, 256, 9)])
def test_host_pipeline(pk, r, M, K, L, F, dtype, pinned):
    bits = _flipped(r)
    pilot = pk.Pilot(bits, device=DEV)
    Y = torch.from_numpy(_y(np.random.default_rng(r), F, M, bits.size))
    H = torch.full((F, M, K, L), complex(3.0, 3.0), dtype=torch.complex64)
    Y, H = (Y.pin_memory(), H.pin_memory()) if pinned else (Y, H)
    pk.estimate_host(Y, pilot, K, L, dtype=dtype, out=H)
    assert pk.get_status(DEV) == 0
    assert torch.equal(H, pk.estimate(Y.to(DEV), pilot, K, L, dtype=dtype).cpu())


# grids that are split into balanced groups of rows, and frames alone, which are not
@pytest.mark.parametrize("F, M, r, K, L", [(96, 64, 10, 8, 64), (80, 100, 9, 4, 64)])
def test_dense_fp32_is_independent_of_the_grid(pk, F, M, r, K, L):
    bits = _flipped(r)
    N = bits.size
    gen = torch.Generator(DEV).manual_seed(r)
    Y = torch.randn(F, M, N, dtype=torch.complex64, device=DEV, generator=gen)
    H = pk.estimate(Y, pk.Pilot(bits, device=DEV), K, L, dtype="fp32")
    # real-valued pilots by the dense kernel: a transform longer than 4096, fewer than 128 lags
    n = 4001
    Yr = torch.randn(F, M, n, dtype=torch.complex64, device=DEV, generator=gen)
    G = torch.randn(F, M, 1, 96, dtype=torch.complex64, device=DEV, generator=gen)
    th = torch.randn(n, device=DEV, generator=gen)
    Hr = pk.estimate_real_pilot(Yr, th, 1, 97, pilot_map="tanh")
    dY, _ = pk.backward(th, Yr, G, 1, 96, need_dp=False, pilot_map="tanh")
    pilot = pk.Pilot(bits, device=DEV)
    for f in (0, 1, F // 2, F - 1):
        one = slice(f, f + 1)
        assert torch.equal(pk.estimate(Y[one].contiguous(), pilot, K, L, dtype="fp32"), H[one])
        assert torch.equal(pk.estimate_real_pilot(Yr[one].contiguous(), th, 1, 97, pilot_map="tanh"), Hr[one])
        d1, _ = pk.backward(th, Yr[one].contiguous(), G[one].contiguous(), 1, 96, need_dp=False, pilot_map="tanh")
        assert torch.equal(d1, dY[one])
    P = 1.0 - 2.0 * bits
    ref = O.estimate_real_pilot(Y[:1].cpu().numpy(), P, K, L)
    assert O.nmse(H[:1].cpu().numpy(), ref) <= TOL_Q["fp32"]
    p = np.tanh(th.double().cpu().numpy())
    assert O.nmse(Hr[:1, :8].cpu().numpy(), O.estimate_real_pilot(Yr[:1, :8].cpu().numpy(), p, 1, 97)) <= 1e-10


def test_pair_kernel_against_the_single_sm_kernel(pk, monkeypatch):
    # both truncate the accumulator at every MMA: relative error up to 1.4e-6 each at N = 4095
    w = C.Workload("t", r=12, M=128, K=16, L=128, F=16, snr_db=(10.0,), seed=1)
    bits, _, Y = C.make(w)
    Yd, pilot = torch.from_numpy(Y).to(DEV), pk.Pilot(bits, device=DEV)
    monkeypatch.setenv("PNCE_TC_FORCE", "1")
    base = pk.estimate(Yd, pilot, 16, 128, dtype="fp16")
    monkeypatch.setenv("PNCE_TC_PAIRS", "1")
    pair = pk.estimate(Yd, pilot, 16, 128, dtype="fp16")
    assert not torch.equal(base, pair)               # two kernels
    assert O.nmse(pair.cpu().numpy(), base.cpu().numpy()) <= 1e-11


@pytest.fixture(scope="module")
def full(pk):
    w = C.PRECISION
    bits, Y = C.make_received(w)
    return w, bits, torch.from_numpy(Y).to(DEV)


@pytest.mark.parametrize("dtype", TC)
def test_tensor_cores_at_full_size(pk, full, dtype, monkeypatch):
    # every frame of 512 against the transform on the same rounded operand, which
    # test_gpu_fullsize compares with the oracle frame by frame; and in overlapped chunks
    w, bits, Y = full
    pilot = pk.Pilot(bits, device=DEV)
    ref = pk.estimate(Y, pilot, w.K, w.L, dtype=dtype)
    monkeypatch.setenv("PNCE_TC_FORCE", "1")
    H = pk.estimate(Y, pilot, w.K, w.L, dtype=dtype)
    assert pk.get_status(DEV) == 0
    for f in range(0, w.F, 32):
        a, b = H[f:f + 32].to(torch.complex128), ref[f:f + 32].to(torch.complex128)
        num, den = ((x.abs() ** 2).sum((1, 2, 3)) for x in (a - b, b))
        assert float((num / den).max()) <= TOL_Q[dtype]
    if dtype in ("fp16", "e4m3"):
        for chunks in ("2", "4", "8"):
            monkeypatch.setenv("PNCE_OVERLAP_CHUNKS", chunks)
            assert torch.equal(pk.estimate(Y, pilot, w.K, w.L, dtype=dtype), H)


def test_dense_fp32_at_full_size(pk, full):
    w, _, Y = full
    bits = _flipped(w.r)
    H = pk.estimate(Y, pk.Pilot(bits, device=DEV), w.K, w.L, dtype="fp32")
    P = torch.fft.fft(torch.from_numpy(1.0 - 2.0 * bits).to(DEV, torch.complex128)).conj()
    for f in range(0, w.F, 8):
        y = Y[f:f + 8].to(torch.complex128)
        ref = (torch.fft.ifft(torch.fft.fft(y) * P)[..., :w.K * w.L] / w.N).view(8, w.M, w.K, w.L)
        d = H[f:f + 8] - ref
        num, den = ((x.abs() ** 2).sum((1, 2, 3)) for x in (d, ref))
        assert float((num / den).max()) <= TOL_Q["fp32"]
        assert float(d.abs().max()) <= 1e-5 * float(ref.abs().max())
