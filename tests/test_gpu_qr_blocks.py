"""GPU: the pivoted QR on columns in shared memory (k_qr.cu) through the SVD, at the sizes where it can go
wrong, against the CPU oracle: one slot and a column more, long thin blocks (up to and past what shared
memory holds), more slots than the GPU holds at once (the step-by-step kernel), tied and zero columns."""
import numpy as np
import pytest

from oracle.symtensor import IN, OUT, Bond as OB, BlockTensor
from test_gpu_linalg import SYM, _check_svd, ctx  # noqa: F401 (ctx is a fixture)
from test_gpu_svd_blocks import _plain

pytestmark = pytest.mark.gpu


# 24: three full slots; 25: one column more; 3210 / 3211 rows: the longest column whose slot fits
# shared memory lies below 3211 (9 columns of 8 bytes per entry in 226 KB)
@pytest.mark.parametrize("m,n", [(24, 24), (25, 40), (512, 16), (3100, 20), (3300, 20), (20, 3300)])
def test_shapes(ctx, m, n):  # noqa: F811
    rng = np.random.default_rng(m * 1000 + n)
    _check_svd(ctx, _plain(rng.standard_normal((m, n)) * 10.0 ** (-4.0 * np.arange(n) / n)), 1)


def test_more_slots_than_resident(ctx):  # noqa: F811
    """700 charge blocks of 17 x 17: 2100 slots, more than fit at once."""
    rng = np.random.default_rng(8)
    secs = [((q,), 17) for q in range(700)]
    T = BlockTensor([OB.make(IN, secs, SYM), OB.make(OUT, secs, SYM)])
    for q in T.keys():
        T.blocks[q] = rng.standard_normal(T.block_shape(q))
    _check_svd(ctx, T, 1, keepdim=9000)


def test_tied_and_zero_columns(ctx):  # noqa: F811
    """Columns of equal norm (an orthogonal matrix, scaled) beside zero columns."""
    rng = np.random.default_rng(9)
    q, _ = np.linalg.qr(rng.standard_normal((40, 30)))
    M = np.concatenate([q, np.zeros((40, 6))], axis=1)
    M[:, 15:30] *= 0.5
    _check_svd(ctx, _plain(M), 1, keepdim=30)
