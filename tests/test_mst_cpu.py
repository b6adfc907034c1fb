"""Tables of the fast m-sequence transform kernel, on the CPU: for every degree the kernel
takes, the tables drive a numpy model of its data movement (slots, register passes, lags) and
the result is the correlation; slots are a permutation within bounds, and every half-warp
access meets 16 different bank pairs.  Pilots that are no m-sequence, and other lengths, get
no tables."""
import ctypes as C

import numpy as np
import pytest

from synth import mseq


def _tables(bits):
    import paper_2206_05506_gb300 as pk
    lib = pk.lib()
    N = bits.size
    size = lib._ZN4pnce15mst_table_bytesEi
    size.restype, size.argtypes = C.c_size_t, [C.c_int]
    build = lib._ZN4pnce16mst_build_tablesEPKjiPt
    build.restype, build.argtypes = C.c_bool, [C.c_void_p, C.c_int, C.c_void_p]
    n = size(N)
    if n == 0:
        return None
    words = mseq.pack_bits(bits)
    out = np.zeros(n // 2, dtype=np.uint16)
    return out if build(words.ctypes.data, N, out.ctypes.data) else None


def _banks_ok(slots):
    """slots [..., 16] of the lanes of half-warps: 16 different bank pairs each"""
    return np.all(np.sort(slots % 16, axis=-1) == np.arange(16))


@pytest.mark.parametrize("r", range(7, 15))
def test_tables_drive_the_transform(r):
    bits = mseq.mseq_bits(r, seed=r % 2)
    N, S = bits.size, 1 << r
    le = 6 if r >= 11 else 5 if r >= 9 else 4 if r == 8 else 3
    lg = r - le
    E, G = 1 << le, 1 << lg
    tab = _tables(bits)
    in_slot = tab[:S].reshape(E // 8, G, 8).transpose(0, 2, 1).reshape(S)      # by sample n
    out_slot = tab[S:2 * S].reshape(E // 8, G, 8).transpose(0, 2, 1).reshape(E, G)
    lag_slot = tab[2 * S:3 * S]
    col = tab[3 * S:].view(np.uint8).reshape(E // 8, G, 4)
    col = np.stack([col & 15, col >> 4], axis=-1).reshape(E // 8, G, 8)
    col = col.transpose(0, 2, 1).reshape(E, G)                                 # [k][t]
    # in: sample n to its slot, register k of thread t reads its entry k G + t
    assert np.array_equal(np.sort(in_slot), np.arange(S))
    assert _banks_ok(in_slot.reshape(-1, 16))
    rng = np.random.default_rng(r)
    y = rng.standard_normal(N)
    buf = np.zeros(S)
    buf[in_slot[:N]] = y
    k, t = np.arange(E)[:, None], np.arange(G)[None, :]
    rd = k * G + (t & ~15) + col
    assert _banks_ok(rd.reshape(-1, 16))
    x = buf[rd]                                                              # entry k G + t
    assert x[0, 0] == 0.0
    w = x.reshape(S).copy()
    for b in range(r):
        v = w.reshape(-1, 2, 1 << b)
        w = np.stack([v[:, 0] + v[:, 1], v[:, 0] - v[:, 1]], axis=1).reshape(S)
    # out: register k of thread t of the second pass holds entry s
    s = (t + ((k >> lg) << lg) << lg | (k & (G - 1))) if lg <= le else (t << le | k)
    assert np.array_equal(np.sort(s.reshape(-1)), np.arange(S))
    assert np.array_equal(np.sort(out_slot.reshape(-1)), np.arange(S))
    assert _banks_ok(out_slot.reshape(-1, 16)) and _banks_ok(lag_slot.reshape(-1, 16))
    buf[out_slot] = w[s]
    h = buf[lag_slot[:N]] / N
    p = 1.0 - 2.0 * bits
    want = np.fft.ifft(np.fft.fft(y) * np.conj(np.fft.fft(p))).real / N
    assert np.allclose(h, want, rtol=0, atol=1e-12)


def test_other_pilots_get_no_tables():
    bits = mseq.mseq_bits(9, 0)
    flipped = bits.copy()
    flipped[17] ^= 1
    assert _tables(flipped) is None
    assert _tables(np.zeros(511, dtype=np.uint8)) is None
    assert _tables(np.ones(127, dtype=np.uint8)) is None
    for n in (63, 126, 500, 512, 32767):        # below, above and beside the degrees taken
        assert _tables(np.resize(bits, n)) is None
