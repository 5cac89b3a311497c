"""GPU: what the kernels of the SVD owe to their own synchronisation: more charge blocks of one slot than
CTAs of the Jacobi sweeps (a CTA goes from slot to slot without a wait in the first round), and the
kernels behind a wait that ran out (the status word is set by the host here; no wait runs out)."""
import ctypes as C

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


N = 16   # vectors of the one block below, and their entries


class _Launches:
    """The launchers of the library (C++ names), on device arrays for one 16 x 16 block."""

    def __init__(self, ctx, status):
        import torch

        import paper_2401_01921_gb300 as tnx
        self.lib, self.torch = tnx.lib(), torch
        rng = np.random.default_rng(6)
        self.keep = {}
        f = lambda n, v: self._dev(n, np.asarray(v, dtype=np.float64))
        i = lambda n, v: self._dev(n, np.asarray(v, dtype=np.int32))
        x, eye = rng.standard_normal((N, N)), np.eye(N)
        ptr = [f("X", x), f("tau", np.zeros(N)), f("u0", np.ones(N)), i("perm", np.arange(N)), f("nrm", np.zeros(2 * N)),
               i("pos", np.zeros(2 * N)), f("Xr", x), f("Jr", eye), f("Xf", np.full((N, N), 7.0)),
               f("J", np.full((N, N), 7.0)), f("sigma", np.full(N, 7.0))]
        d = f("D", np.tile([1.0, 1.0, 0.0, 0.0], (N, 1)))
        struct = lambda n, p, w, tail=(): self._dev(n, np.concatenate(
            [np.array(p, dtype=np.int64).view(np.uint8), np.array(w, dtype=np.int32).view(np.uint8),
             np.array(tail, dtype=np.int64).view(np.uint8)]))
        self.q = struct("q", ptr, [N, N, N, 0], [d])
        self.svd = struct("svd", [ptr[6], ptr[7], ptr[10]], [N, N])
        # one pair of column blocks of eight vectors: one slot
        jb = [ptr[6], ptr[7], d, i("ver", [0, 0])], [N, N, 2, 8]
        self.jb = struct("jb", *jb)
        self.jb_host = np.concatenate([np.array(jb[0], dtype=np.int64).view(np.uint8),
                                       np.array(jb[1], dtype=np.int32).view(np.uint8)])
        self.vecs = i("vecs", [[0, p] for p in range(N)])
        self.pairs = i("pairs", [[0, p] for p in range(N // 2)])
        self.slots = i("slots", [[0, 0]])
        self.words = i("words", np.zeros(1024))   # zeroed counters, flags and maxima
        self.stat = i("stat", [status, 0])
        self.before = {n: self.get(n) for n in ("Xr", "Jr", "Xf", "J", "sigma", "D")}

    def _dev(self, name, a):
        self.keep[name] = self.torch.from_numpy(np.ascontiguousarray(a)).cuda()
        return self.keep[name].data_ptr()

    def get(self, name):
        self.torch.cuda.synchronize()
        return self.keep[name].cpu().numpy().copy()

    def changed(self):
        return {n for n, a in self.before.items() if not np.array_equal(a, self.get(n))}

    def run(self, which):
        p, w = C.c_void_p, lambda k: C.c_void_p(self.words + 4 * k)
        st, sweeps = p(self.stat), p(self.stat + 4)
        if which == "gather":
            code = self.lib._Z22tnx_launch_qr_gather_rPK5SvdQriiPKiP11CUstream_st(p(self.q), 1, N, st, None)
        elif which == "apply":
            code = self.lib._Z19tnx_launch_qr_applyPK5SvdQrPK4int2iiPKiP11CUstream_st(p(self.q), p(self.vecs), N, N, st,
                                                                                     None)
        elif which == "sweeps in shared memory":
            code = self.lib._Z23tnx_launch_jacobi_blockPK7JbGroupS1_iPK4int2iidPiPjS5_S5_P11CUstream_st(
                p(self.jb), self.jb_host.ctypes.data_as(p), 1, p(self.slots), 1, 60, C.c_double(1e-13), w(0), w(64), st,
                sweeps, None)
        else:
            code = self.lib._Z22tnx_launch_jacobi_coopPK8SvdGroupPK4int2iiiidPyS5_PiS6_P11CUstream_st(
                p(self.svd), p(self.pairs), N // 2, N, N, 60, C.c_double(1e-13), w(128), w(512), st, sweeps, None)
        assert code == 0


@pytest.mark.parametrize("which,writes", [("gather", {"Xr"}), ("apply", {"Xf", "J", "sigma"}),
                                          ("sweeps in shared memory", {"Xr", "Jr", "D"}), ("sweeps", {"Xr", "Jr"})])
def test_nothing_runs_behind_a_wait_that_ran_out(ctx, which, writes):  # noqa: F811
    """With the status word set (an expired QR has written only a part of its permutation) the kernels
    behind it touch nothing; with it clear they do their work."""
    for status in (1, 0):
        k = _Launches(ctx, status)
        k.run(which)
        assert k.changed() == (set() if status else writes)
        assert k.get("stat")[0] == status
