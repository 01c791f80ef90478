"""The push's fast path and the two ways it hands out tiles.

CPU: the integers and offsets that the fast path takes from a rounded-down
add (FP32, 1.5 2^23) and from the bits (FP64) against floor(), with what it must
refuse.  GPU: the contiguous shares (few tiles per block) and the tickets
(many) give the same FP32 state bit for bit, over discharges of uneven size
with empty species and part-filled tiles."""
import math
import struct
from fractions import Fraction

import numpy as np
import pytest

from paper_0705_0495_gb300 import inputs


def _add_down(x, m, bits):
    """x + m rounded towards minus infinity to `bits` mantissa bits"""
    s = Fraction(x) + Fraction(m)
    if s == 0:
        return 0.0
    e = math.floor(math.log2(abs(float(s))))
    ulp = Fraction(2) ** (e - bits + 1)
    return float(math.floor(s / ulp) * ulp)


def _positions(rng, dtype):
    v = [0.0, 0.5, 1.0, -1.0, np.nextafter(dtype(1), dtype(0)), np.nextafter(dtype(1), dtype(2)),
         -np.finfo(dtype).tiny, np.finfo(dtype).tiny, -1e-9, 1e-9, 4095.999, -4096.0, 4194303.5, -4194303.5]
    v += list(rng.uniform(-3.0, 3.0, 200)) + list(rng.uniform(-5000, 5000, 200))
    return [dtype(x) for x in v]


def test_fp32_fast_floor_is_floor():
    rng = np.random.default_rng(3)
    M = 12582912.0
    for on in _positions(rng, np.float32):
        t = np.float32(_add_down(float(on), M, 24))
        k = struct.unpack("<i", struct.pack("<f", t))[0] - 0x4B400000
        assert k == math.floor(float(on)), on
        fl = np.float32(t - np.float32(M))
        assert float(fl) == math.floor(float(on)), on
        assert np.float32(on - fl) == np.float32(on - np.float32(math.floor(float(on)))), on


def test_fp32_fast_path_refuses_what_is_far_off():
    """beyond |on| < 2^22 the integer read from the bits, added to a cell,
    never lies on a grid (compared as unsigned), whatever its sign does"""
    far = [4194304.0, -4194305.0, 7e6, -7e6, 1.2582911e7, -1.2582911e7, -12582912.0, -12582913.0, -1.3e7,
           -2.4e7, -3e7, 1e9, -1e9, 1e30, -1e30, math.inf, -math.inf]
    for on in far:
        t = np.float32(on) if math.isinf(on) else np.float32(_add_down(float(np.float32(on)), 12582912.0, 24))
        for zero in ((0.0, -0.0) if t == 0 else (t,)):
            k = struct.unpack("<i", struct.pack("<f", np.float32(zero)))[0] - 0x4B400000
            for c in (0, 1, 4095):
                cn = (c + k) & 0xFFFFFFFF
                assert cn >= 4096, (on, c, cn)
    for nan in (0x7FC00000, 0xFFC00000, 0x7FFFFFFF, 0xFFFFFFFF):
        for c in (0, 4095):
            assert ((c + nan - 0x4B400000) & 0xFFFFFFFF) >= 4096


def _words(x):
    u = struct.unpack("<Q", struct.pack("<d", x))[0]
    return u >> 32, u & 0xFFFFFFFF


def _floor_bits(on):
    """the FP64 fast path's floor from the bits of |on| < 64"""
    hi, lo = _words(on)
    a = hi & 0x7FFFFFFF
    e = max((a >> 20) - 1023, -1)
    ip = ((a & 0xFFFFF) | 0x100000) >> (20 - e)
    frac = e < 0 or (((a << (12 + e)) & 0xFFFFFFFF) | lo) != 0
    return -(ip + (1 if frac else 0)) if hi >> 31 else ip


def test_fp64_fast_floor_is_floor():
    rng = np.random.default_rng(4)
    v = _positions(rng, np.float64) + [np.float64(k + d) for k in range(-63, 64) for d in (0.0, 2.0 ** -46, -2.0 ** -46, 0.5)]
    v += [np.nextafter(np.float64(k), np.float64(s)) for k in range(-63, 64) for s in (-100.0, 100.0)]
    for on in v:
        on = float(on)
        if not abs(on) < 64.0:
            assert _words(on)[0] & 0x7FFFFFFF >= 0x40500000  # sent to the general path
            continue
        if on == 0.0 and math.copysign(1.0, on) < 0:
            assert _floor_bits(on) == -1  # offset 1: sent to the general path
            continue
        assert _floor_bits(on) == math.floor(on), on


def test_fp64_energy_bin_from_the_fp32_estimate():
    """the estimate, from values cut to 24 bits, decides the bin except within
    64 units of the last place of an edge; its error stays below 12 units"""
    rng = np.random.default_rng(9)

    def cut(x):
        hi, lo = _words(abs(x))
        if hi < 0x38100000:
            return np.float32(0)
        b = (((hi - 0x38000000) << 3) | (lo >> 29)) & 0xFFFFFFFF
        return struct.unpack("<f", struct.pack("<I", b))[0]

    for _ in range(3000):
        v = rng.normal(0, 1, 3) * 10.0 ** rng.uniform(-4, 2)
        ke = 10.0 ** rng.uniform(-6, 2)
        K = ke * (v[0] * v[0] + v[1] * v[1] + v[2] * v[2])
        f = [np.float32(cut(x)) for x in v]
        Kf = np.float32(np.float32(cut(ke)) * np.float32(f[0] * f[0] + f[1] * f[1] + f[2] * f[2]))
        bits = struct.unpack("<I", struct.pack("<f", Kf))[0]
        exact = struct.unpack("<I", struct.pack("<f", np.float32(K)))[0]
        assert abs(bits - exact) < 13, (v, ke)
        if ((bits + 64) & 0x1FFFFF) >= 128:
            hi = _words(K)[0]
            assert (bits >> 21) - 4 * 127 == 4 * ((hi >> 20) - 1023) + ((hi >> 18) & 3)


def test_fp64_weight_from_one_add():
    rng = np.random.default_rng(4)
    # rn(off 2^40) read from off + 2^12
    for off in list(rng.uniform(0.0, 1.0, 300)) + [0.0, 2.0 ** -41, 3 * 2.0 ** -41, math.nextafter(1.0, 0.0)]:
        got = struct.unpack("<q", struct.pack("<d", off + 4096.0))[0] - struct.unpack("<q", struct.pack("<d", 4096.0))[0]
        assert got == round(off * 2.0 ** 40), off


def test_fp64_uniform_from_bits_is_exact():
    """1 + (w + 1/2) 2^-32 written as a bit pattern, minus 1"""
    rng = np.random.default_rng(6)
    for w in [0, 1, 0xFFF, 0x1000, 0x7FFFFFFF, 0x80000000, 0xFFFFFFFF] + [int(x) for x in rng.integers(0, 2 ** 32, 300)]:
        hi, lo = 0x3FF00000 | (w >> 12), ((w << 20) & 0xFFFFFFFF) | 0x80000
        got = struct.unpack("<d", struct.pack("<Q", (hi << 32) | lo))[0] - 1.0
        assert got == (w + 0.5) / 4294967296.0, w


def test_fp64_charge_words_stay_exact():
    """a cell's sum in 14, 13 and 13-bit words of 32 bits, at the most
    particles a block adds before it flushes, each of the largest weight"""
    most, one = 256 * 1024, 1 << 40
    for w1 in (one, one - 1, 0x5555555555, 1):
        words = (w1 & 0x3FFF, (w1 >> 14) & 0x1FFF, w1 >> 27)
        assert all(most * x < 2 ** 32 for x in words), w1
        assert sum((most * x) << b for x, b in zip(words, (0, 14, 27))) == most * w1
    # 128 particles at once (a warp's sum, in two halves of 24 and 18 bits)
    assert 32 * 4 * ((one - 1) & 0xFFFFFF) < 2 ** 32 and 32 * ((4 * one) >> 24) < 2 ** 32


@pytest.mark.gpu
@pytest.mark.parametrize("sizes", [(1_400_001, 2, 33_333), (700_000, 0, 1, 1_023, 1_500_000)])
def test_shares_and_tickets_give_the_same_state(sizes):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_0705_0495_gb300 import o2pic
    ds = [inputs.cfg1(fp64=False, n_op=n, n_cells=100 + 57 * k, seed=3 + k, diag_every=2)
          for k, n in enumerate(sizes)]
    states = []
    for blocks in ("most", 1):  # one block per SM: many tiles per block, so tickets
        sim = o2pic.Simulation(ds, inputs.xs_tables())
        if blocks == 1:
            sim.set_launch(1)
        sim.step(13)
        states.append([sim.get_state(d, s) for d in range(len(ds)) for s in range(3)]
                      + [{k: sim.diagnostics(d)[k] for k in ("events", "absorbed", "eedf", "iedf", "fm", "dens_sum")}
                         for d in range(len(ds))])
        sim.close()
    for a, b in zip(*states):
        for k in a:
            assert np.array_equal(a[k], b[k]), k
