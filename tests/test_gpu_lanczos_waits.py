"""GPU: the waits inside a Lanczos step (its CTAs wait for one another: a cluster up to 20480 entries, a
resident grid above), with other work on the GPU that delays some of them."""
import numpy as np
import pytest

import paper_2401_01921_gb300 as tnx
import tnx_inputs as I

from gpu_harness import lib_heff
from test_gpu_serve import ctx  # noqa: F401 (a fixture)

pytestmark = pytest.mark.gpu


def test_solves_side_by_side(ctx):  # noqa: F811
    """Clusters and resident grids of several solves on streams of their own: the eigenvalues and Ritz
    vectors of each are the bits that it gives alone (the order of every sum is fixed)."""
    wls = [I.heisenberg_workload(c, 20) for c in (64, 128, 200, 400, 512)]   # the last two: grids
    wls += [I.hubbard_workload(64, seed_base=2000), I.hubbard_workload(350, seed_base=3000)]
    nets = [lib_heff(ctx, wl, symmetric=True) for wl in wls]
    alone = []
    for net, T, B in nets:
        evec = tnx.Tensor(ctx, B["psi"])
        lam, k = tnx.lanczos(net, "psi", T["psi"], 15, evec)
        alone.append((lam, k, evec.download()))
    srv = tnx.Server(ctx, max_slots=len(nets))
    for _ in range(4):
        outs = [tnx.Tensor(ctx, B["psi"]) for _, _, B in nets]
        ids = [srv.submit(net, "psi", T["psi"], tnx.REQ_LANCZOS, 15, o) for (net, T, B), o in zip(nets, outs)]
        for (lam, k, x), rid, o in zip(alone, ids, outs):
            ev, mv, _ = srv.wait(rid, 60000)
            assert (ev, mv) == (lam, k)
            assert np.array_equal(o.download(), x)
    srv.close()
    ctx.sync()
