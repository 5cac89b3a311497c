"""GPU: the fused MPO step with a warp per tile (many small bands): a batch large enough for it gives the
bits that each instance's own launch gives with its kernel, bands of one row to several tiles, in the
tree that scatters into the last operand and the one that writes the rows out; and a single apply."""
import numpy as np
import pytest

import paper_2401_01921_gb300 as tnx
import tnx_inputs as I

from gpu_harness import lib_heff, oracle_heff, rel_fro
from test_gpu_fused_rows import ctx  # noqa: F401 (a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", ["(L,((psi,R),(W1,W2)))", "(((psi,R),(W1,W2)),L)"])
@pytest.mark.parametrize("prec,tol", [("f64", 1e-12), ("split_bf16", 1e-10)])
def test_batch_with_a_warp_per_tile(ctx, order, prec, tol):  # noqa: F811
    wls = [I.hubbard_workload(c, seed_base=2000 + 4 * i) for i, c in enumerate([64, 150, 333, 700])]
    built = [lib_heff(ctx, wl, prec=prec, order=order) for wl in wls]
    outs = [tnx.Tensor(ctx, B["psi"]) for _, _, B in built]
    batch = tnx.Batch(ctx, [n for n, _, _ in built])
    batch.launch_into(outs)
    for (net, T, B), o, wl in zip(built, outs, wls):
        onet, _ = oracle_heff(wl, order=order)
        assert rel_fro(o.block_dict(), onet.launch()) <= tol
        assert np.array_equal(o.download(), net.launch(B["psi"]).download())


def test_apply_with_a_warp_per_tile(ctx):  # noqa: F811
    wl = I.hubbard_workload(601)
    order = "(L,(((psi,R),W2),W1))"
    net, T, B = lib_heff(ctx, wl, order=order)
    onet, _ = oracle_heff(wl, order=order)
    assert rel_fro(net.launch(B["psi"]).block_dict(), onet.launch()) <= 1e-12
