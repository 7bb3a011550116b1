"""The bound of the exact re-rank's U8 pass, restated: the FP32 sums of squared
differences in the U8 pass's order (8 lanes of 16-element chunks, packed pairs)
and in the FP32 pass's order (32 lanes of 4-element chunks) differ by at most
2^-17 (2 s (1 + 2^-16)) (1 + 2^-10), s the U8 pass's value, up to 1024
dimensions, on random rows and on rows built so that every rounding goes the
same way.
"""
import numpy as np
import pytest

F = np.float32


def _fma(a, b, c):
    return F(np.float64(a) * np.float64(b) + np.float64(c))  # one rounding (53 bits hold a b + c of FP32 to 1 ulp)


def _tree(v, offs):
    v = list(v)
    for o in offs:
        v = [F(v[i] + v[i ^ o]) for i in range(len(v))]
    return v[0]


def u8_pass(q, x):
    lanes = []
    for j in range(8):
        a = [F(0), F(0)]
        for t0 in range(16 * j, len(q), 128):
            for t in range(t0, t0 + 16):
                e = F(q[t] - x[t])
                a[t & 1] = _fma(e, e, a[t & 1])
        lanes.append(F(a[0] + a[1]))
    return _tree(lanes, (4, 2, 1))


def fp32_pass(q, x):
    lanes = [F(0)] * 32
    for ln in range(32):
        for t0 in range(4 * ln, len(q), 128):
            for t in range(t0, min(t0 + 4, len(q))):
                e = F(q[t] - x[t])
                lanes[ln] = _fma(e, e, lanes[ln])
    return _tree(lanes, (16, 8, 4, 2, 1))


def _rows(d, kind, rng):
    x = rng.integers(0, 256, d).astype(F)
    if kind == "random":
        return (x + rng.normal(0, 40, d)).astype(F), x
    if kind == "far":
        return (x + rng.choice([-1, 1], d) * 1e6 * rng.random(d)).astype(F), x
    # every difference rounds up by almost half an ulp, every addition too
    q = (x + F(3.0) + F(2.0) ** -18 * rng.integers(1, 7, d).astype(F)).astype(F)
    return q, x


def _ratio(d, kind, seed):
    q, x = _rows(d, kind, np.random.default_rng(seed))
    s, f = u8_pass(q, x), fp32_pass(q, x)
    e = 2.0 ** -17 * 2 * float(s) * (1 + 2.0 ** -16) * (1 + 2.0 ** -10)
    return abs(float(s) - float(f)) / e if e else float(s != f)


@pytest.mark.parametrize("d", [16, 144, 784, 1024])
@pytest.mark.parametrize("kind", ["random", "far", "aligned"])
def test_bound(d, kind):
    assert max(_ratio(d, kind, s) for s in range(6)) <= 1.0


def test_roundings_on_a_path():
    """At most 64 + 1 + 3 additions and two for the difference on either path, at 2^-24 each."""
    steps = max(2 + 1024 // 16 + 1 + 3, 2 + 1024 // 32 + 5)
    assert (1 + 2.0 ** -24) ** steps - 1 < 2.0 ** -17
