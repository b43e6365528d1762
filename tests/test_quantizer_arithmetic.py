"""Arithmetic of the NVFP4 quantizer that is not written as the division it stands for, checked on the CPU."""
import numpy as np


def test_product_with_a_sixth_and_its_remainder_is_the_division_by_six():
    """fl32(x / 6) as q = fl32(x r), fma(fma(-6, q, x), r, q) with r = fl32(1/6): every significand, in the lowest and the
    highest binade that the kernel's comment names and one between.  Extended precision holds both fused sums exactly (x - 6 q has few bits)."""
    f, ext = np.float32, np.longdouble
    assert np.finfo(ext).nmant >= 63
    r = f(0.16666667163372040)
    significands = np.arange(1 << 23, 1 << 24, dtype=np.int64).astype(f)
    for exponent in (-100, 0, 103):
        x = np.ldexp(significands, exponent - 24)               # [2^(exponent - 1), 2^exponent)
        q = x * r
        remainder = (ext(x) - 6 * q.astype(ext)).astype(f)
        got = (remainder.astype(ext) * ext(r) + q.astype(ext)).astype(f)
        assert np.array_equal(got, x / f(6))
