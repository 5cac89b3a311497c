"""GPU: the one-launch Lanczos step at the sizes where it changes shape (a cluster of eight CTAs up to
20480 entries, a resident grid above) and with the Gram-Schmidt pass in both, against the oracle."""
import numpy as np
import pytest

import tnx_inputs as I

from gpu_harness import lib_heff
from test_gpu_lanczos_oracle import _check_solve, _oracle_solve, ctx  # noqa: F401 (ctx is a fixture)

pytestmark = pytest.mark.gpu

# entries: 36 (most CTAs without any), 514, 18620 (the cluster's largest), 24648 (25 CTAs), 34632 (34), 77384 (76)
SIZES = [("dense", 3, 10), ("hubbard", 20, 15), ("heisenberg", 200, 20), ("heisenberg", 230, 20), ("hubbard", 350, 20),
         ("heisenberg", 400, 20)]


def _workload(model, chi):
    return {"dense": I.dense_workload, "hubbard": I.hubbard_workload,
            "heisenberg": lambda c: I.heisenberg_workload(c, 20)}[model](chi)


@pytest.mark.parametrize("model,chi,nsteps", SIZES)
def test_step_against_oracle(ctx, model, chi, nsteps):  # noqa: F811
    _check_solve(ctx, _workload(model, chi), "f64", None, nsteps, 1e-12, 1e-8)


@pytest.mark.parametrize("model,chi", [("heisenberg", 200), ("hubbard", 350), ("heisenberg", 400)])
def test_pass_in_every_step(ctx, model, chi):  # noqa: F811
    """FP32 products are no symmetric operator to FP64 accuracy, so every step takes the pass: the basis
    stays orthonormal to FP64 rounding (one pass leaves about sqrt(n) eps |w| before over after, here
    below 1e-11), so the Ritz vector has unit norm; without the pass it would lose about 1e-7."""
    import paper_2401_01921_gb300 as tnx
    wl = _workload(model, chi)
    net, T, B = lib_heff(ctx, wl, symmetric=True, prec="f32")
    evec = tnx.Tensor(ctx, B["psi"])
    lam, k = tnx.lanczos(net, "psi", T["psi"], 20, evec)
    olam, _, ok, _ = _oracle_solve(wl, None, 20)
    assert k == ok == 20
    assert abs(np.linalg.norm(evec.download()) - 1.0) <= 1e-11
    # the operator is off by at most K eps32 of the product of norms, K <= 4000
    assert abs(lam - olam) <= 4000 * 2.0 ** -24 * abs(olam)
