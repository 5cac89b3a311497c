"""GPU: the SVD of blocks whose squared norms lie at or beyond the end of the FP64 range, and of blocks with
an infinity or a NaN: a singular value is right or not finite, and other charge blocks are untouched; and
columns at the length that the QR's shared memory ends at."""
import numpy as np
import pytest

import paper_2401_01921_gb300 as tnx
from oracle.symtensor import IN, OUT, Bond as OB, BlockTensor
from test_gpu_linalg import SYM, _check_svd, ctx, to_lib  # noqa: F401 (ctx is a fixture)
from test_gpu_svd_blocks import _plain

pytestmark = pytest.mark.gpu


def _values(ctx, T):  # noqa: F811
    U, S, V, terr, dw = tnx.svd_truncate(to_lib(ctx, T), 1)
    return [np.diag(b) for _, b in sorted(S.block_dict().items())]


# 32 rows: one entry per lane, so that no lane's own square or sum overflows, only the sum over the warp;
# 20 columns: the QR in shared memory; 1e152: the squared norms are finite
@pytest.mark.parametrize("scale,finite", [(1e154, False), (1e152, True)])
def test_norms_beyond_the_range(ctx, scale, finite):  # noqa: F811
    rng = np.random.default_rng(11)
    M = rng.uniform(0.9, 1.0, (32, 20)) * rng.choice([-1.0, 1.0], (32, 20)) * scale
    (s,) = _values(ctx, _plain(M))
    if finite:
        assert np.max(np.abs(s - np.linalg.svd(M, compute_uv=False))) <= 1e-12 * s[0]
    else:
        assert not np.any(np.isfinite(s))


def test_one_column_at_the_end_of_the_range(ctx):  # noqa: F811
    """|x|^2 = 1.1e308 is finite, |x|^2 + |x_0| |x| (of the reflector) is not."""
    rng = np.random.default_rng(12)
    M = rng.standard_normal((32, 20)) * 1e100
    M[:, 4] = rng.standard_normal(32) * 1e150
    M[0, 4] = 1.05e154
    (s,) = _values(ctx, _plain(M))
    n0 = 1.05e154 * np.sqrt(1.0 + np.sum((M[1:, 4] / 1.05e154) ** 2))
    assert abs(s[0] - n0) <= 1e-12 * n0
    # the others see that column only through its direction, up to (1e100 / 1e154)^2
    u = M[:, 4] / n0
    rest = np.delete(M, 4, axis=1)
    ref = np.linalg.svd(rest - np.outer(u, u @ rest), compute_uv=False)
    assert np.max(np.abs(s[1:] - ref)) <= 1e-12 * ref[0]


@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_an_entry_that_is_no_number_stays_in_its_block(ctx, value):  # noqa: F811
    rng = np.random.default_rng(13)
    secs = [((0,), 24), ((1,), 20), ((2,), 33)]
    T = BlockTensor([OB.make(IN, secs, SYM), OB.make(OUT, secs, SYM)])
    for q in T.keys():
        T.blocks[q] = rng.standard_normal(T.block_shape(q))
    T.blocks[(1, 1)][3, 5] = value
    got = _values(ctx, T)
    assert [len(s) for s in got] == [24, 20, 33]
    assert not np.any(np.isfinite(got[1]))
    for s, q in ((got[0], (0, 0)), (got[2], (2, 2))):
        ref = np.linalg.svd(T.blocks[q], compute_uv=False)
        assert np.max(np.abs(s - ref)) <= 1e-12 * ref[0]


# a slot of the QR holds nine columns, padded to 32 entries: 9 * 8 * 3200 bytes and its few words of state
# fit 226 KB, 9 * 8 * 3232 do not (the step-by-step QR takes them)
@pytest.mark.parametrize("rows", [3169, 3200, 3201])
def test_longest_columns_in_shared_memory(ctx, rows):  # noqa: F811
    holds = tnx.lib()._Z20tnx_qr_block_columnsi
    assert holds(rows) == (8 if rows <= 3200 else 0)
    rng = np.random.default_rng(rows)
    _check_svd(ctx, _plain(rng.standard_normal((rows, 20)) * 10.0 ** (-4.0 * np.arange(20) / 20)), 1)


# blocks of fewer than 16 vectors: no QR, the sweeps run on the block itself
@pytest.mark.parametrize("scale", [1e-140, 1e-75, 1e-70, 1e70, 1e75, 1e140])
def test_small_blocks_far_from_one(ctx, scale):  # noqa: F811
    rng = np.random.default_rng(14)
    secs, secs2 = [((0,), 9), ((1,), 2), ((2,), 15)], [((0,), 12), ((1,), 3), ((2,), 4)]
    T = BlockTensor([OB.make(IN, secs, SYM), OB.make(OUT, secs2, SYM)])
    for q in T.keys():
        T.blocks[q] = rng.standard_normal(T.block_shape(q)) * scale
    for s, q in zip(_values(ctx, T), sorted(T.keys())):
        ref = np.linalg.svd(T.blocks[q], compute_uv=False)
        assert np.max(np.abs(s - ref)) <= 1e-13 * ref[0]
