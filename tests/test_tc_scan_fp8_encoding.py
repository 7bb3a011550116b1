"""The encoding of the tensor-core scan, restated on the CPU with the constants
read from the kernel: e4m3 of the nibbles 0 .. 15 and their split by two byte
permutes, the one-hot row of a code (e4m3 1.0 shifted into one of four words),
and the sum 16 high + low + 2^23, whose low bits are the table sum, exact for
every number of subspaces the scan takes and any order of its FP32 additions."""
import os
import re

import numpy as np

import oracle

SRC = open(os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_03298_gb300", "csrc",
                        "scan_tc.cu")).read()


def e4m3(b):
    s, e, m = -1.0 if b & 0x80 else 1.0, (b >> 3) & 15, b & 7
    return s * (m / 8 * 2.0 ** -6 if e == 0 else (1 + m / 8) * 2.0 ** (e - 7))


def prmt(a, b, sel):
    """Byte permute of two words: byte k of the result is byte sel[4k .. 4k+2] of (a, b)."""
    by = [(a >> (8 * k)) & 255 for k in range(4)] + [(b >> (8 * k)) & 255 for k in range(4)]
    return sum(by[(sel >> (4 * k)) & 7] << (8 * k) for k in range(4))


def f8_table():
    words = re.search(r"uint4 f8 = make_uint4\(([^)]*)\)", SRC).group(1)
    return [int(w.strip().rstrip("u"), 16) for w in words.split(",")]


def test_nibbles_are_e4m3():
    for v, w in enumerate(f8_table()):
        assert [e4m3((w >> (8 * k)) & 255) for k in range(4)] == [4 * v + k for k in range(4)]


def lut16x8(w, t):
    s0 = w & 0x77777777
    k0 = ((w >> 1) & 0x44444444) | 0x32103210
    lo = prmt(prmt(t[0], t[1], s0), prmt(t[2], t[3], s0), k0)
    hi = prmt(prmt(t[0], t[1], s0 >> 16), prmt(t[2], t[3], s0 >> 16), k0 >> 16)
    return lo, hi


def test_table_bytes_split_into_nibbles():
    t = f8_table()
    sel = [int(x, 16) for x in re.findall(r"(?:lo|hi)\[k\] = prmt\(a, b, (0x\w+)u\)", SRC)]
    assert len(sel) == 2
    rng = np.random.default_rng(1)
    for T in list(rng.integers(0, 256, size=(200, 4))) + [[0, 255, 15, 240]]:
        w = sum(int(v) << (8 * k) for k, v in enumerate(T))
        a, b = lut16x8(w, t)
        lo, hi = prmt(a, b, sel[0]), prmt(a, b, sel[1])
        assert [e4m3((lo >> (8 * k)) & 255) for k in range(4)] == [int(v) & 15 for v in T]
        assert [e4m3((hi >> (8 * k)) & 255) for k in range(4)] == [int(v) >> 4 for v in T]


def test_one_hot_rows():
    rot = re.search(r"rot = \((\d+) \* \(lane & 7\) - (\d+)\) & 31", SRC).groups()
    one = int(re.search(r'"r"\((0x\w+)u\), "r"\(c8 - 32u \* i\)', SRC).group(1), 16)
    assert e4m3(one) == 1.0
    rng = np.random.default_rng(2)
    for word in rng.integers(0, 1 << 32, size=50, dtype=np.uint64):
        for lane in range(8):
            code = (int(word) >> (4 * lane)) & 15
            r = (int(rot[0]) * lane - int(rot[1])) & 31
            c8 = ((int(word) >> r) | (int(word) << (32 - r))) & 0xffffffff & 0x78
            row = b""
            for i in range(4):
                sh = (c8 - 32 * i) & 0xffffffff  # shl of 32 and more gives zero
                row += ((one << sh) & 0xffffffff if sh < 32 else 0).to_bytes(4, "little")
            assert [e4m3(v) for v in row] == [1.0 if e == code else 0.0 for e in range(16)]


def test_sums_are_the_scan_sums():
    rng = np.random.default_rng(3)
    for M in (1, 8, 50, 128):
        codes = rng.integers(0, 16, size=(48, M)).astype(np.uint8)
        T = rng.integers(0, 256, size=(M, 16)).astype(np.uint8)
        T[:, 15] = 255
        codes[0] = 15
        parts = []
        for nib in (T >> 4, T & 15):
            terms = nib[np.arange(M)[None], codes].astype(np.float32)
            acc = np.zeros(len(codes), np.float32)
            for j in rng.permutation(M):
                acc = acc + terms[:, j]
            assert acc.max() < 2 ** 12
            parts.append(acc)
        s = np.float32(16) * parts[0] + (parts[1] + np.float32(8388608.0))  # one rounding each, none needed
        got = s.view(np.uint32) & 0xffff
        ref = np.array([oracle.int_dist(T, 0, c) for c in codes])
        np.testing.assert_array_equal(got, ref)
        np.testing.assert_array_equal((s - np.float32(8388608.0)).astype(np.int64), ref)
