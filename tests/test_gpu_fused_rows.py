"""GPU: the fused MPO step on full tiles, two rows to a lane (ragged last tiles, an odd number of rows):
FP64 applies of the Heisenberg H_eff, against the oracle, in the tree that scatters into the last
operand and the one that writes the rows out."""
import pytest

import tnx_inputs as I

from gpu_harness import lib_heff, oracle_heff, rel_fro

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2401_01921_gb300 as tnx
    from paper_2401_01921_gb300 import build
    build.build()
    return tnx.Context(0)


@pytest.mark.parametrize("chi,n,order", [(1301, 33, "(L,((psi,R),(W1,W2)))"), (1597, 35, "(((psi,R),(W1,W2)),L)")])
def test_apply_with_full_tiles(ctx, chi, n, order):
    wl = I.heisenberg_workload(chi, n)
    net, T, B = lib_heff(ctx, wl, order=order)
    onet, _ = oracle_heff(wl, order=order)
    assert rel_fro(net.launch(B["psi"]).block_dict(), onet.launch()) <= 1e-12
