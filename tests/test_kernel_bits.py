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


def test_upwind_signs():
    """The upwinding's integer sign tests against the comparisons, NaN, infinities and signed zeros included."""
    edge = np.array([0.0, -0.0, 5e-324, -5e-324, 1.0, -1.0, 1e308, -1e308, np.inf, -np.inf, np.nan, -np.nan])
    with np.errstate(invalid="ignore", over="ignore"):
        uL, uR = (a.ravel() for a in np.meshgrid(edge, edge))
        s = uL + uR
        one, sg, inf = np.uint64(1), np.uint64(1 << 63), np.uint64(0x7ff0000000000000)
        pos = lambda x, flip: ((x.view(np.uint64) ^ flip) - one) < inf
        left = pos(uL, np.uint64(0)) & pos(s, np.uint64(0))
        right = ~left & pos(uR, sg) & pos(s, sg)
        want_left = (uL > 0) & (uL + uR > 0)
        want_right = ~want_left & (uR < 0) & (uL + uR < 0)
    assert (left == want_left).all() and (right == want_right).all()
