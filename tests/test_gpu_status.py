"""GPU: the outcome of a bounded device wait reaches the call whose kernels made it.  The status word of a
network is set by the host here, as a kernel does when a wait runs out; no wait runs out."""
import ctypes as C
import gc

import pytest

import paper_2401_01921_gb300 as tnx
import tnx_inputs as I

from gpu_harness import lib_heff
from test_gpu_serve import ctx  # noqa: F401 (a fixture)

pytestmark = pytest.mark.gpu


def _expire(net, site):
    f = tnx.lib()._Z18tnx_network_statusP11tnx_network
    f.argtypes, f.restype = [C.c_void_p], C.POINTER(C.c_int32)
    f(net.h)[0] = site


def test_a_served_request_reports_its_own_wait(ctx):  # noqa: F811
    nets = [lib_heff(ctx, I.heisenberg_workload(c, 10), symmetric=True) for c in (64, 96)]
    alone = [tnx.lanczos(net, "psi", T["psi"], 10) for net, T, B in nets]
    srv = tnx.Server(ctx, max_slots=2)
    outs = [tnx.Tensor(ctx, B["psi"]) for _, _, B in nets]
    submit = lambda i, kind: srv.submit(nets[i][0], "psi", nets[i][1]["psi"], kind, 10, outs[i])
    for kind in (tnx.REQ_LANCZOS, tnx.REQ_APPLY):
        _expire(nets[0][0], 43)
        ids = [submit(0, kind), submit(1, tnx.REQ_LANCZOS)]
        with pytest.raises(tnx.TnxError) as e:
            srv.wait(ids[0], 60000)
        assert e.value.name == "TNX_ERR_TIMEOUT" and "site 43" in str(e.value)
        assert srv.wait(ids[1], 60000)[:2] == alone[1]   # the other request is not blamed
        ctx.sync()                                       # nor is what comes next
        assert srv.wait(submit(0, tnx.REQ_LANCZOS), 60000)[:2] == alone[0]
    srv.close()


def test_a_direct_call_reports_and_clears(ctx):  # noqa: F811
    net, T, B = lib_heff(ctx, I.heisenberg_workload(64, 10), symmetric=True)
    alone = tnx.lanczos(net, "psi", T["psi"], 10)
    for call in (lambda: tnx.lanczos(net, "psi", T["psi"], 10), ctx.sync):
        _expire(net, 41)
        with pytest.raises(tnx.TnxError) as e:
            call()
        assert e.value.name == "TNX_ERR_TIMEOUT" and "site 41" in str(e.value)
        ctx.sync()
        assert tnx.lanczos(net, "psi", T["psi"], 10) == alone
    # a network destroyed with an unread code leaves it to the next synchronisation
    # ... not to the network that is created next
    _expire(net, 42)
    del net, call, e
    gc.collect()
    net, T, B = lib_heff(ctx, I.heisenberg_workload(64, 10), symmetric=True)
    srv = tnx.Server(ctx, max_slots=1)
    assert srv.wait(srv.submit(net, "psi", T["psi"], tnx.REQ_LANCZOS, 10), 60000)[:2] == alone
    srv.close()
    with pytest.raises(tnx.TnxError) as e:
        ctx.sync()
    assert "site 42" in str(e.value)
    ctx.sync()
