"""Serving batches of m-sequence pilots: a request's result has the bits of an estimate of its
own, in every format, whatever its lag count and whatever shares the batch (and, for short
pilots, the warp) with it: the few-lags form's largest count and the next one, one lag, odd
counts, rows of few and of many lags side by side; by descriptor table and by the native loop."""
import ctypes as C

import pytest
import torch

from synth import mseq

pytestmark = pytest.mark.gpu

FEW = {7: 8, 8: 8, 9: 8, 10: 16, 11: 32, 12: 32, 13: 32, 14: 32}     # largest of the few-lags form
DTYPES = ["fp32", "fp16", "bf16", "e4m3", "tf32"]


def _requests(r, N, seed):
    """(M, K, L, Y, H) in page-locked memory, few and many lags alternating, a guard after each H"""
    f = FEW[r]
    lags = [1, 60, f, 2, f + 1, 3, 64, f - 1, 5, 7, 33, 1]
    gen = torch.Generator().manual_seed(seed)
    out = []
    for i, KL in enumerate(lags):
        M, K = 1 + i % 3, 2 if KL % 2 == 0 else 1
        Y = torch.randn(M, N, dtype=torch.complex64, generator=gen).pin_memory()
        H = torch.full((M * KL + 1,), complex(7.0, 7.0), dtype=torch.complex64).pin_memory()
        out.append((M, K, KL // K, Y, H))
    return out


def _check(pk, pilot, reqs, dtype):
    for M, K, L, Y, H in reqs:
        ref = pk.estimate(Y.to(pilot.device)[None], pilot, K, L, dtype=dtype).cpu().reshape(-1)
        assert torch.equal(H[:-1], ref), (M, K, L)
        assert H[-1] == complex(7.0, 7.0)


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("r", sorted(FEW))
def test_table(r, dtype):
    import paper_2206_05506_gb300 as pk
    from paper_2206_05506_gb300 import _lib
    dev = torch.device("cuda", 0)
    bits = mseq.mseq_bits(r, 1)
    pilot, reqs = pk.Pilot(bits, device=dev), _requests(r, bits.size, r)
    for rows, kl_max in ((64, 70), (29, 64)):    # rows without a request behind the last one, or not
        buf = torch.zeros((len(reqs) + 1) * C.sizeof(_lib.ReqDesc), dtype=torch.uint8).pin_memory()
        arr = (_lib.ReqDesc * (len(reqs) + 1)).from_address(buf.data_ptr())
        off = 0
        for d, (M, K, L, Y, H) in zip(arr, reqs):
            d.Y, d.H, d.M, d.K, d.L, d.row_offset = Y.data_ptr(), H.data_ptr(), M, K, L, off
            off += M
            H[:-1] = 0
        ws = torch.empty(pk.grouped_workspace_size(rows, bits.size, kl_max, dtype), dtype=torch.uint8, device=dev)
        pk.estimate_grouped(pilot, buf.data_ptr(), len(reqs) + 1, rows, kl_max, dtype, ws)
        torch.cuda.synchronize()
        assert pk.get_status(dev) == 0
        _check(pk, pilot, reqs, dtype)


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("r", sorted(FEW))
def test_native_loop(r, dtype):
    import paper_2206_05506_gb300 as pk
    from paper_2206_05506_gb300 import serve
    dev = torch.device("cuda", 0)
    N = (1 << r) - 1
    reqs = _requests(r, N, r + 50)
    nat = serve.NativeServer(lambda n: mseq.mseq_bits(n.bit_length(), 1), device=dev, dtype=dtype, slots=2,
                             max_batch_rows=256)
    st = nat.run([serve.Request(i, 0.0, M, N, K, L, Y.data_ptr(), H.data_ptr())
                  for i, (M, K, L, Y, H) in enumerate(reqs)])
    assert st["failed"] == 0 and st["batches"] < len(reqs)
    _check(pk, nat.pilot(N), reqs, dtype)
