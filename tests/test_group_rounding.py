"""The FP64 product-sum's grouped rounding, checked in IEEE arithmetic on the
CPU: adding a group of products in one FP32 sum that is rounded to the result's
last place after each product, then added once, gives the same bits as
Algorithm 2's one FP64 addition per product.  The steps restate the kernel's
(code bytes, rounding constants, start value); the reference is plain FP64
addition in order."""
import numpy as np
import pytest

KEEP, EACH, MAX_BITS = 0, 1, 20
F = np.float32


def codes_of(H):
    """Code of each element for unit u = 1 (g = 2^n), as the kernel forms it."""
    bits = H.view(np.uint64)
    n = ((bits >> np.uint64(52)) & np.uint64(0x7FF)).astype(np.int64) - 1075
    top = (bits >> np.uint64(32)) & np.uint64(0xFFFFF)
    edge = ((n >= 0) & (top == 0xFFFFF)) | ((n > 0) & (top == 0)) | (n > MAX_BITS)
    odd = (bits & np.uint64(1)).astype(np.int64) << 7
    return np.where(edge, EACH, np.where(n > 0, (n + 48) | odd, KEEP))


def round_to(x, code):
    m = np.ldexp(F(1), (code & 0x7F) - 25).astype(F)
    r = (np.abs(x) + m).astype(F) - m
    return np.copysign(r.astype(F), x)


def start_of(code):
    return np.where(code & 0x80, np.ldexp(F(1), (code & 0x7F) - 48), F(0)).astype(F)


def grouped(H, P):
    """H <- the products P[0], P[1], ... (integers below 2^20 in magnitude) as one group."""
    code = codes_of(H)
    each = code == EACH
    hi = np.zeros(H.shape, F)
    V = H.copy()
    for i, p in enumerate(P):
        hi = (hi + p.astype(F)).astype(F)                    # exact below 2^24
        if i == len(P) - 1:
            break
        V = np.where(each, V + hi.astype(np.float64), V)
        hi = np.where(each, F(0), hi).astype(F)
        if i == 0:
            hi = (hi + start_of(code)).astype(F)
        hi = round_to(hi, code)
    return V + (hi - start_of(code)).astype(F).astype(np.float64)


def test_rounding_constants_round_to_nearest_even():
    vals = np.array(sorted({s * (2 ** k + d) for k in range(24) for d in (-1, 0, 1) for s in (1, -1)} | {0}), np.int64)
    rng = np.random.default_rng(0)
    vals = np.concatenate([vals, rng.integers(-2 ** 24 + 1, 2 ** 24, 200000)])
    vals = vals[np.abs(vals) < 2 ** 24]
    x = vals.astype(F)
    assert np.array_equal(round_to(x, np.full(vals.shape, KEEP)), x)
    for n in range(1, MAX_BITS + 1):
        got = round_to(x, np.full(vals.shape, n + 48)).astype(np.int64)
        q, r = np.divmod(vals, 1 << n)
        half = 1 << (n - 1)
        want = (q + ((r > half) | ((r == half) & (q & 1 == 1)))) << n
        assert np.array_equal(got, want), n


@pytest.mark.parametrize("nprod", [2, 4, 6])
@pytest.mark.parametrize("scale", [40, 53, 54, 60, 70, 73, 80])
def test_grouped_products_equal_one_addition_each(nprod, scale):
    """H of magnitude about 2^scale u: nothing to round, a few bits, past MAX_BITS."""
    rng = np.random.default_rng(100 * nprod + scale)
    size = 200000
    H = np.rint(np.ldexp(rng.random(size) + 0.25, scale))     # integers, odd and even multiples of the last place
    # next to powers of two, where the last place changes
    k = size // 4
    H[:k] = np.ldexp(1.0, rng.integers(max(scale - 8, 1), scale + 1, k)) + np.rint(np.ldexp(rng.integers(-3, 4, k), max(scale - 52, 0)))
    H *= rng.choice([-1.0, 1.0], size)
    H[-1] = 0.0
    P = [rng.integers(-2 ** 20, 2 ** 20, size) >> rng.integers(0, 20) for _ in range(nprod)]
    P[0][::7] = 2 ** 17                                         # powers of two, and exact cancellation
    P[1][::14] = -2 ** 17
    want = H.copy()
    for p in P:
        want = want + p.astype(np.float64)
    got = grouped(H, P)
    assert np.array_equal(got, want)
