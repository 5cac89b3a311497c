"""GPU: the split products' epilogue at the edges of its 128 x 64 and 128 x 32 tiles. Even columns of
the result are converted on the integer units and odd ones on the FP64 unit, so a column that stands
twice side by side in B has to come out twice bit for bit; a power of two on the operands has to come
out as that power of two."""
import numpy as np
import pytest

from test_gpu_f64_tiles import _product, ctx  # noqa: F401 (ctx is a fixture)

pytestmark = pytest.mark.gpu


# rows: inside one warp's 32, at and over its edge, over a tile; K: the short (<= 160) and the chunked
# level sums, more than one chunk (640); columns: inside, at and over 8, 32 and 64
@pytest.mark.parametrize("m,k,n", [(1, 3, 1), (31, 40, 7), (32, 160, 8), (33, 161, 9), (96, 200, 31), (127, 640, 33),
                                   (128, 641, 63), (129, 300, 64), (257, 1300, 65), (200, 130, 129)])
@pytest.mark.parametrize("prec", ["split_bf16", "split_f16"])
def test_columns_twice_and_powers_of_two(ctx, m, k, n, prec):  # noqa: F811
    rng = np.random.default_rng(m * 10007 + k * 101 + n)
    A = rng.standard_normal((m, k)) * 10.0 ** rng.uniform(-9, 9, (m, 1))
    B = np.repeat(rng.standard_normal((k, n)) * 10.0 ** rng.uniform(-9, 9, n), 2, axis=1)
    B[:, 2 * (n // 2):2 * (n // 2) + 2] = 0.0          # a column of zeros
    base = _product(ctx, A, B, prec)
    assert np.array_equal(base[:, 0::2], base[:, 1::2])
    assert not base[:, 2 * (n // 2)].any()
    # entries rounded 41 bits below their row's (column's) largest, levels below 2^-42 dropped, over K
    # balancing that may move up to the spread of a column of A (standard normal: a factor of 16)
    bound = 2.0 ** -34 * k * np.outer(np.max(np.abs(A), axis=1), np.max(np.abs(B), axis=0))
    assert np.all(np.abs(base - A @ B) <= bound)
    for p, q in ((-300, -200), (300, 400), (-520, -500)):
        # entries are at most 2^66 in size: 2^(p+q) leaves the operands normal and the result finite
        got = _product(ctx, np.ldexp(A, p), np.ldexp(B, q), prec)
        assert np.array_equal(got[:, 0::2], got[:, 1::2])
        want = np.ldexp(base, p + q)
        # a result below the normal range is stored as zero, everything else is exact
        assert np.array_equal(got, np.where(np.abs(want) < 2.0 ** -1022, 0.0, want))
