"""GPU: FP64 and FP32 products at the edges of their tiles, and the skinny (K <= 16) products with rows
shared by several threads, against numpy."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2401_01921_gb300 as tnx
    from paper_2401_01921_gb300 import build
    build.build()
    return tnx.Context(0)


def _product(ctx, A, B, prec):
    import paper_2401_01921_gb300 as tnx
    (m, k), n = A.shape, B.shape[1]
    bond = lambda d: tnx.Bond(ctx, tnx.BD_REG, [((), d)])
    ta, tb = tnx.Tensor(ctx, [bond(m), bond(k)]), tnx.Tensor(ctx, [bond(k), bond(n)])
    ta.upload(A)
    tb.upload(B)
    net = tnx.Network(ctx, "A: i, k\nB: k, j\nTOUT: i, j\n")
    net.put("A", ta)
    net.put("B", tb)
    net.set_precision(prec)
    return net.launch([ta.bonds[0], tb.bonds[1]]).download().reshape(m, n)


# 8 x 8 tiles: one row / column short and over, K at and beside the staged 32; 2060 x 2060: 16 x 16 tiles;
# K <= 16: skinny, 1 to 200 rows (1 to 128 threads' worth), few and many columns
@pytest.mark.parametrize("m,k,n", [(7, 17, 9), (8, 32, 8), (9, 33, 7), (1, 31, 65), (64, 64, 64), (130, 65, 3),
                                   (2060, 19, 2060), (1, 1, 1), (3, 16, 130), (33, 5, 64), (65, 16, 7), (200, 11, 9)])
@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_product(ctx, m, k, n, prec):
    rng = np.random.default_rng(m * 10007 + k * 101 + n)
    A, B = rng.standard_normal((m, k)), rng.standard_normal((k, n))
    B[rng.random((k, n)) < 0.3] = 0.0
    got = _product(ctx, A, B, prec)
    # a k-term sum of rounded products, operands rounded first in FP32 (K <= 16 stays FP64)
    eps = 2.0 ** -53 if prec == "f64" or k <= 16 else 2.0 ** -24
    assert np.all(np.abs(got - A @ B) <= (k + 3) * 2 * eps * (np.abs(A) @ np.abs(B)))
