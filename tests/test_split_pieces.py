"""The FP64 speculative split's FP32 pieces, restated in IEEE FP32 on the CPU:
slices of whole operands equal the oracle's (Eq. (fp64split) in FP64) for
entries at ties, powers of two, all-ones significands and wide exponent ranges,
for the levels v^(r) = v^(0) - 8r that the pass assumes."""
import numpy as np
import pytest

import oracle

F, U64 = np.float32, np.uint64


def pieces(x, v0):
    """Slices (FP32 values) of x as the kernel's fast form computes them."""
    b = x.view(U64)
    E = ((b >> U64(52)) & U64(0x7FF)).astype(np.int64)
    M = (b & U64((1 << 52) - 1)) | np.where(E > 0, U64(1 << 52), U64(0))
    neg = (b >> U64(63)).astype(bool)
    t = v0 + 1023 - E
    U = M << U64(10)
    sh = np.minimum(t + 12, 63).astype(U64)
    X = U >> sh
    X = np.where(t + 12 > 63, U64(0), X)
    X |= ((X << sh) != U).astype(U64)
    Xh, Xl = (X >> U64(28)).astype(np.int64), (X & U64(0xFFFFFFF)).astype(np.int64)
    y = (Xh + np.where(Xl > 0, 0.5, 0.0)).astype(F) * np.where(neg, F(-1), F(1))
    out = []

    def level(y, grid, unit_exp):
        C = np.where(y < 0, F(6291456) * F(grid), F(12582912) * F(grid)).astype(F)
        z = ((y + C).astype(F) - C).astype(F)
        out.append(np.ldexp(z.astype(np.float64), unit_exp))
        return (y - z).astype(F)

    y = level(y, 2 ** 15, v0 - 22)
    y = level(y, 2 ** 7, v0 - 22)
    r = (y - np.where(Xl > 0, F(0.5), F(0)) * np.where(neg, F(-1), F(1))).astype(np.int64)
    sX = np.where(neg, -Xl, Xl)
    Yh, Yl = (r << 15) + (sX >> 13), sX & 0x1FFF
    p = np.where(Yl > 0, F(0.5), F(0)).astype(F)
    y = (Yh.astype(F) + p).astype(F)
    y = level(y, 2 ** 14, v0 - 37)
    y = level(y, 2 ** 6, v0 - 37)
    y = ((y - p).astype(np.float64) * 8192 + Yl).astype(F)
    y = level(y, 2 ** 11, v0 - 50)
    level(y, 2 ** 3, v0 - 50)
    return np.stack(out)


@pytest.mark.parametrize("v0", [-78, -20, 0, 1, 60, 127])
@pytest.mark.parametrize("kind", ["uniform", "few bits", "ones", "powers", "wide"])
def test_pieces_equal_the_oracle(v0, kind):
    rng = np.random.default_rng(v0 + 100)
    n = 60000
    m = rng.integers(0, 1 << 52, n, dtype=np.int64).astype(U64)
    if kind == "few bits":
        m &= rng.integers(0, 1 << 52, n, dtype=np.int64).astype(U64) & rng.integers(0, 1 << 52, n, dtype=np.int64).astype(U64)
    if kind == "ones":
        m |= rng.integers(0, 1 << 52, n, dtype=np.int64).astype(U64) | rng.integers(0, 1 << 52, n, dtype=np.int64).astype(U64)
    if kind == "powers":
        m[:] = 0
    span = 45 if kind in ("powers", "wide") else 10
    x = np.ldexp(1.0 + m.astype(np.float64) * 2.0 ** -52, v0 - 1 - rng.integers(0, span, n))
    x *= rng.choice([-1.0, 1.0], n)
    x[:1000] = 0.0
    # entries that pin the six levels to steps of 8
    pin = np.ldexp(np.abs(rng.random(2000)) * 0.5 + 0.5, v0)
    x = np.concatenate([x, pin])
    want, v, flags = oracle.split_f64(x[None, :].copy())
    v = np.asarray(v).ravel()
    assert np.array_equal(v, v0 - 8 * np.arange(6)), v
    if flags:
        pytest.skip("slices below the BF16 range (v0 near the domain's end)")
    w = np.asarray(want).view(np.uint16).reshape(6, -1).astype(np.uint32) << 16
    got = pieces(x, v0).astype(F).view(np.uint32)
    got = np.where(got == 0x80000000, 0, got)
    assert np.array_equal(got, w)
