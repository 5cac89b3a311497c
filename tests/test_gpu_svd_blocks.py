"""GPU: the Jacobi sweeps on column blocks (k_jacobi.cu) at the sizes where they can go wrong, against
the CPU oracle: blocks around the column-block and warp widths, one long enough for narrower column
blocks, more slots than the GPU holds at once, rank-deficient blocks, entries far from 1."""
import numpy as np
import pytest

from oracle.symtensor import IN, OUT, Bond as OB, BlockTensor
from test_gpu_linalg import SYM, _check_svd, ctx  # noqa: F401 (ctx is a fixture)

pytestmark = pytest.mark.gpu


def _plain(M):
    m, n = M.shape
    return BlockTensor([OB.make(0, [((), m)]), OB.make(0, [((), n)])], {(0, 0): M})


# 16: the smallest block with QR; 17, 33, 49: a column block more; 31 .. 65: whole and ragged
# warps; 897: too long for two blocks of 8 vectors in shared memory
@pytest.mark.parametrize("m,n", [(16, 16), (17, 20), (31, 31), (33, 32), (49, 70), (64, 65), (97, 97), (900, 897)])
def test_block_sizes(ctx, m, n):  # noqa: F811
    rng = np.random.default_rng(m * 1000 + n)
    _check_svd(ctx, _plain(rng.standard_normal((m, n)) * 10.0 ** (-6.0 * np.arange(n) / n)), 1)


def test_more_slots_than_resident(ctx):  # noqa: F811
    """400 charge blocks of 17 .. 24 vectors: every CTA runs several slots, round by round."""
    rng = np.random.default_rng(3)
    secs = [((q,), 17 + q % 8) for q in range(400)]
    T = BlockTensor([OB.make(IN, secs, SYM), OB.make(OUT, secs, SYM)])
    for q in T.keys():
        T.blocks[q] = rng.standard_normal(T.block_shape(q))
    _check_svd(ctx, T, 1, keepdim=5000)


def test_rank_deficient(ctx):  # noqa: F811
    """Equal, zero and dependent columns: singular values at and below rounding, orthonormal factors."""
    rng = np.random.default_rng(4)
    M = rng.standard_normal((50, 40))
    M[:, 7] = M[:, 3]
    M[:, 11] = 0.0
    M[:, 20:30] = M[:, :10] @ rng.standard_normal((10, 10))
    _check_svd(ctx, _plain(M), 1, keepdim=28)


@pytest.mark.parametrize("scale", [1e-120, 1e120])
def test_entries_far_from_one(ctx, scale):  # noqa: F811
    rng = np.random.default_rng(5)
    _check_svd(ctx, _plain(rng.standard_normal((60, 45)) * scale), 1)
