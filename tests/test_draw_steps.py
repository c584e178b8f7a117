"""The exact steps of the Gaussian draw that avoid integer conversions, for every value of
the 23 bits that a word gives: the same uniform, mantissa, exponent, remainder and quadrant
as by integer arithmetic.  Equality, no tolerance: each step is exact in binary32."""
import numpy as np

K = np.arange(1 << 23, dtype=np.uint32)  # w >> 9
NUM = (2 * K + 1).astype(np.int64)


def _bits(x):
    return x.view(np.uint32)


def _from_bits(b):
    return b.astype(np.uint32).view(np.float32)


def test_uniform():
    u = _from_bits(np.uint32(0x3F800000) | K) - np.float32(0.999999940395355224609375)
    assert np.array_equal(u.astype(np.float64), NUM * 2.0 ** -24)


def test_mantissa_and_exponent():
    u = (NUM * 2.0 ** -24).astype(np.float32)
    b = _bits(u)
    over = b - np.uint32(0x3F3504F4)  # modulo 2^32
    f = _from_bits(b - (over & np.uint32(0xFF800000)))
    e = over.view(np.int32) >> 23
    ef = _from_bits(np.uint32(0x4B400000) + e.view(np.uint32)) - np.float32(12582912.0)
    e0 = ((b >> 23) & 0xFF).astype(np.int32) - 127
    f0 = _from_bits((b & np.uint32(0x7FFFFF)) | np.uint32(0x3F800000))
    high = f0 > np.float32(1.41421356237309504880)
    assert np.array_equal(f, np.where(high, f0 * np.float32(0.5), f0))
    assert np.array_equal(e, e0 + high)
    assert np.array_equal(ef, e.astype(np.float32))


def test_quadrant_and_remainder():
    u4 = _from_bits(np.uint32(0x40800000) | K) - np.float32(3.9999997615814208984375)
    qm = u4 + np.float32(12582912.0)
    f = u4 - (qm - np.float32(12582912.0))
    q = (NUM + (1 << 21)) >> 22
    assert np.array_equal(_bits(qm) & 3, q & 3)
    assert np.array_equal(f.astype(np.float64), (NUM - (q << 22)) * 2.0 ** -22)
