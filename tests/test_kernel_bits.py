"""CPU model of f32_to_f64 (fpbits.cuh): the widening of a binary32 from its bit
fields on 32-bit words against the exact conversion, at the edges of every
range it distinguishes."""
import numpy as np


def widen(u):
    """The kernel's integer steps on uint32 patterns; None where it takes the conversion."""
    a = u & np.uint32(0x7fffffff)
    normal = ((a.astype(np.int64) - 0x00800000) % 2 ** 32 < 0x7f000000) | (a == 0)
    hi = np.where(a != 0, (a >> np.uint32(3)) + np.uint32(0x38000000), np.uint32(0)) | (u & np.uint32(0x80000000))
    lo = (u.astype(np.uint64) << np.uint64(29)) & np.uint64(0xffffffff)
    return normal, (hi.astype(np.uint64) << np.uint64(32)) | lo


def test_f32_to_f64_words():
    rng = np.random.default_rng(5)
    edge = np.array([0, 1, 0x007fffff, 0x00800000, 0x00800001, 0x3f800000, 0x7f7fffff, 0x7f800000, 0x7fc00000],
                    dtype=np.uint32)
    u = np.concatenate([edge, edge | np.uint32(0x80000000), rng.integers(0, 2 ** 32, 200000, dtype=np.uint32)])
    normal, bits = widen(u)
    f = u.view(np.float32)
    with np.errstate(invalid="ignore"):
        want = f.astype(np.float64).view(np.uint64)
    is_normal = (np.isfinite(f) & (np.abs(f) >= np.finfo(np.float32).tiny)) | (f == 0)
    assert (normal == is_normal).all()
    assert (bits[normal] == want[normal]).all()
