"""GPU: what the kernels of the SVD owe to their own synchronisation: more charge blocks of one slot than
CTAs of the Jacobi sweeps (a CTA goes from slot to slot without a wait in the first round)."""
import numpy as np
import pytest

from oracle.symtensor import IN, OUT, Bond as OB, BlockTensor
from test_gpu_linalg import SYM, _check_svd, ctx  # noqa: F401 (ctx is a fixture)

pytestmark = pytest.mark.gpu


def test_more_single_slot_blocks_than_ctas(ctx):  # noqa: F811
    """1000 charge blocks of 2 .. 16 vectors, one slot each, beside one of 40 (at most 5 CTAs of 384 threads
    fit on an SM, so at most 760 run): a block is finished after a sweep that met no pair above the
    tolerance, so a slot that loses that flag leaves its block after the first sweep, with singular
    vectors far from orthogonal."""
    rng = np.random.default_rng(0)
    secs = [((q,), 40 if q == 500 else 2 + q % 15) for q in range(1001)]
    T = BlockTensor([OB.make(IN, secs, SYM), OB.make(OUT, secs, SYM)])
    for q in T.keys():
        T.blocks[q] = rng.standard_normal(T.block_shape(q))
    _check_svd(ctx, T, 1)
