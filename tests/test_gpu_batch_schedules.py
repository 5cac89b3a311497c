"""GPU: the launch schedules that the autotuning of a batch chooses from are four different ones."""
import ctypes as C

import numpy as np
import pytest

import paper_2401_01921_gb300 as tnx
import tnx_inputs as I

from gpu_harness import lib_heff
from test_gpu_serve import ctx  # noqa: F401 (a fixture)

pytestmark = pytest.mark.gpu


def _shape(batch, step, choice):
    f = tnx.lib()._Z21tnx_batch_split_shapePK9tnx_batchiiPiS2_
    f.argtypes, f.restype = [C.c_void_p, C.c_int, C.c_int, C.POINTER(C.c_int), C.POINTER(C.c_int)], None
    n, g = C.c_int(), C.c_int()
    f(batch.h, step, choice, C.byref(n), C.byref(g))
    return n.value, g.value


@pytest.mark.parametrize("prec", ["split_bf16", "tf32"])
def test_schedules(ctx, prec):  # noqa: F811
    wls = [I.hubbard_workload(600 + 20 * i, seed_base=1000 + 4 * i) for i in range(8)]
    built = [lib_heff(ctx, wl, prec=prec, order="(L,(((psi,R),W2),W1))") for wl in wls]
    batch = tnx.Batch(ctx, [net for net, _, _ in built])
    step = max(range(4), key=lambda k: _shape(batch, k, 0)[0])   # four contractions, the MPO's have no split tiles
    tiles, grid = _shape(batch, step, 0)
    assert tiles > 456 and grid == 0                 # one CTA per tile
    assert _shape(batch, step, 304) == (tiles, 304) and _shape(batch, step, 456) == (tiles, 456)
    padded, grid = _shape(batch, step, 152)          # equal lists for 152 CTAs, the shorter ones with holes
    assert grid == 152 and padded >= tiles and padded % 152 == 0
    outs = [tnx.Tensor(ctx, B["psi"]) for _, _, B in built]
    batch.launch_into(outs)
    first = [o.download() for o in outs]
    assert batch.autotune(outs) in (0, 152, 304, 456)   # leaves the last candidate's outputs
    assert all(np.array_equal(o.download(), x) for o, x in zip(outs, first))
    batch.launch_into(outs)
    assert all(np.array_equal(o.download(), x) for o, x in zip(outs, first))
