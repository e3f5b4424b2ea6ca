"""The resampler's output counts #{j : T_j < S} = ceil(S Np / Q - u 2^-32) from
32-bit fixed point (FastCount, with the exact form where the fixed-point
value lies within 8 units of a whole number), against exact integers: every
decided value equals the exact count, on boundaries drawn at random and on
both sides of thresholds, for the smallest and largest Np and Q."""
import numpy as np
import pytest

M32 = (1 << 32) - 1


def _rz32(x):
    """x (float64) rounded to FP32 toward zero."""
    f = np.float32(x)
    return np.nextafter(f, np.float32(0)) if abs(float(f)) > abs(x) else f


class FastCount:
    """The kernel's constants and estimate, step by step."""

    def __init__(self, Q, Np, u):
        p = (Np - 1).bit_length()
        self.f = 30 - p
        self.mask = (1 << self.f) - 1
        self.uo = u >> (p + 2)
        self.sh = Q.bit_length() - 32
        q32 = Q >> self.sh
        num = Np << (62 - p)
        r = np.float32(1.0 / float(np.float32(q32)))
        m0 = int(_rz32(float(_rz32(float(_rz32(num >> 32)) * 4294967296.0)) * float(r)))
        rem = num - m0 * q32
        self.m = m0 + int(_rz32(float(np.float32(rem)) * float(r)))

    def v(self, S):
        return (((S >> self.sh) * self.m) >> 32) - self.uo

    def count(self, S, Q, Np, u):
        v = self.v(S)
        if ((v + 8) & self.mask) >= 16:
            return (v + self.mask) >> self.f, True
        n = (v + 8) >> self.f
        if n < 0:
            return 0, False
        return (n if (S * Np << 32) <= Q * ((n << 32) | u) else n + 1), False


def _exact(S, Q, Np, u):
    return max(0, -((u * Q - (S * Np << 32)) // (Q << 32)))


@pytest.mark.parametrize("Np", [1, 2, 3, 31, 256, 1000, 4095, 16384, 65535, 65536, (1 << 20) - 1, 1 << 20])
def test_counts_equal_exact_integers(Np):
    rng = np.random.default_rng(Np)
    decided = 0
    for _ in range(60):
        lo, hi = 1 << 40, Np << 40
        Q = min(hi, max(lo, int(lo * (hi / lo) ** rng.random()) + int(rng.integers(0, 1 << 20))))
        if rng.random() < 0.15:
            Q = (lo, hi)[int(rng.integers(0, 2))]
        u = int(rng.choice([0, 1, 7, M32, M32 - 5, int(rng.integers(0, 1 << 32)), int(rng.integers(0, 1 << 32))]))
        fc = FastCount(Q, Np, u)
        S = [0, Q, 1, Q - 1] + [int(Q * rng.random()) for _ in range(20)]
        for _ in range(20):  # the thresholds T_j and their neighbours
            j = int(rng.integers(0, Np))
            T = (((j << 32) + u) * Q // Np) >> 32
            S += [min(Q, max(0, T + d)) for d in (-1, 0, 1)]
        for s in S:
            got, fast = fc.count(s, Q, Np, u)
            want = _exact(s, Q, Np, u)
            assert got == want, (Np, Q, u, s, got, want, fast)
            decided += fast
    assert decided > 0
