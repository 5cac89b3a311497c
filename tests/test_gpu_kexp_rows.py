"""GPU: split products whose A has columns of very different scale, at row and K counts around the
K-balancing kernel's passes (one CTA or a cluster of CTAs per 32 K indices) and the slicing kernel's
row groups and K tiles per warp, against numpy."""
import numpy as np
import pytest

from test_gpu_f64_tiles import _product, ctx  # noqa: F401 (ctx is a fixture)

pytestmark = pytest.mark.gpu


# K: one to five tiles per warp (32, 64 | 256, 512 | 600), ragged; M: below and above 96 rows, one
# pass of a cluster and more, a group of 8 rows short and over
@pytest.mark.parametrize("m,k,n", [(1, 33, 5), (7, 64, 9), (97, 40, 65), (129, 256, 8), (513, 257, 64), (1500, 100, 33),
                                   (60, 512, 70), (130, 600, 40), (260, 1100, 24)])
@pytest.mark.parametrize("prec", ["split_bf16", "split_f16"])
def test_columns_of_different_scale(ctx, m, k, n, prec):  # noqa: F811
    rng = np.random.default_rng(m * 10007 + k * 101 + n)
    A = rng.standard_normal((m, k)) * 10.0 ** rng.uniform(-9, 9, k)
    B = rng.standard_normal((k, n)) * 10.0 ** rng.uniform(-3, 3, k)[:, None]
    A[rng.random((m, k)) < 0.1] = 0.0
    got = _product(ctx, A, B, prec)
    # operands balanced by the exponent of A's column maxima, each entry then rounded 41 bits below
    # its row's (column's) largest, levels below 2^-42 dropped: 2^-38 leaves a factor of four
    # (a column of A without a nonzero entry is not shifted)
    top = np.max(np.abs(A), axis=0)
    e = np.floor(np.log2(np.where(top > 0, top, 1.0)))
    row = np.max(np.abs(A * 2.0 ** -e), axis=1)
    col = np.max(np.abs(B * 2.0 ** e[:, None]), axis=0)
    assert np.all(np.abs(got - A @ B) <= 2.0 ** -38 * k * np.outer(row, col))
