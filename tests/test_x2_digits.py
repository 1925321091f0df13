"""The arithmetic of the FP64-accurate tensor-core product, restated in numpy float32
with one rounding per operation: the seven digits of a scaled float pair, exact integer
sums of one level, and the product's error against exact FP64."""
import numpy as np

F = np.float32


def digits(hi, lo, e):
    """As the kernel: t = hi 2^e; digit = t rounded to an integer; t = (t - digit) 256; the low part joins the fourth."""
    def rnd(t):
        return ((t + F(12582912.0)).astype(F) - F(12582912.0)).astype(F)
    t = F(hi) * F(2.0 ** e)
    d = []
    for i in range(7):
        d.append(rnd(t))
        t = (t - d[i]).astype(F)
        if i == 3:
            l = (F(lo) * F(2.0 ** (e + 24))).astype(F)
            p = rnd(l)
            d[i] = (d[i] + p).astype(F)
            t = (t + (l - p).astype(F)).astype(F)
        t = (t * F(256.0)).astype(F)
    return np.stack(d)


def split(v):
    hi = v.astype(F)
    return hi, (v - hi).astype(F)


def exponent(v):
    return 6 - int(np.floor(np.log2(np.max(np.abs(v.astype(F))))))


def test_digits_reconstruct_and_products():
    rng = np.random.default_rng(4)
    for spread in (0.0, 4.0, 12.0):  # decades between the entries of a segment
        a = rng.standard_normal(128) * 10.0 ** (-spread * rng.random(128)) * 1e-9
        b = rng.standard_normal(128) * 10.0 ** (-spread * rng.random(128)) * 3.0
        ea, eb = exponent(a), exponent(b)
        da, db = digits(*split(a), ea), digits(*split(b), eb)
        for v, d, e in ((a, da, ea), (b, db, eb)):
            assert np.all(np.abs(d) <= 256) and np.all(d == np.rint(d))
            back = sum(np.float64(d[i]) * 2.0 ** (-8 * i) for i in range(7)) * 2.0 ** -e
            assert np.max(np.abs(back - v)) <= 2.0 ** -48 * np.max(np.abs(v))
        total = 0.0
        for level in range(7):
            s = sum(np.float64(da[i]) * np.float64(db[level - i]) for i in range(level + 1))
            assert np.sum(np.abs(s)) < 2 ** 24  # exact in FP32 whatever the order
            total += np.sum(s) * 2.0 ** (-8 * level)
        exact = float(np.sum(a.astype(np.longdouble) * b.astype(np.longdouble)))
        assert abs(total * 2.0 ** (-ea - eb) - exact) <= 128 * 2.0 ** -47 * np.max(np.abs(a)) * np.max(np.abs(b))
