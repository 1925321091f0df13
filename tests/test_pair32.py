"""The FP32 pair arithmetic of the complex64 products' sparse parts (pair32.cuh), restated in
numpy float32 with one rounding per operation: sums of FP32 numbers times FP64 coefficients held
as hi + lo, against exact FP64.  A pair carries 2^-48 of the largest term per operation."""
import numpy as np

F = np.float32


class P32:
    def __init__(self):
        self.s, self.c = F(0), F(0)

    def add(self, v):
        t = F(self.s + v)
        b = F(t - self.s)
        self.c = F(self.c + F(F(self.s - F(t - b)) + F(v - b)))
        self.s = t

    def fma(self, h, l, v):
        p = F(h * v)
        e = F(np.float64(h) * np.float64(v) - np.float64(p))   # the product of two FP32 numbers is exact in FP64
        e = F(np.float64(l) * np.float64(v) + np.float64(e))
        self.c = F(self.c + e)
        self.add(p)


def test_pair_sums():
    rng = np.random.default_rng(7)
    worst = 0.0
    for n in (1, 3, 12, 40):
        for _ in range(50):
            x = rng.standard_normal(n) * 10.0 ** rng.uniform(-6, 6, n)
            v = rng.standard_normal(n).astype(F)
            h = x.astype(F)
            lo = (x - h.astype(np.float64)).astype(F)
            a = P32()
            for i in range(n):
                a.fma(h[i], lo[i], v[i])
            got = np.float64(a.s) + np.float64(a.c)
            ref = float(np.sum(x.astype(np.longdouble) * v.astype(np.longdouble)))
            worst = max(worst, abs(got - ref) / (n * np.max(np.abs(x * v))))
            assert abs(F(got) - F(ref)) <= 2.0 ** -23 * abs(ref) + n * 2.0 ** -47 * np.max(np.abs(x * v))
    assert worst <= 2.0 ** -46
