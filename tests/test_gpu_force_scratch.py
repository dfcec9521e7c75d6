"""The force gives the same numbers whatever scratch its plaquette matrices get.

All time slices at once, ranges of slices that share a ring with the slices on
either side, or no scratch: each link's sums run over the same matrices in the
same order, so the gradients agree bit for bit.  The limits are set through an
internal symbol of the library (force_scratch_limit, csrc/api.cu), which also makes
a context's larger allocations fail as they do when memory is short.
"""
import ctypes

import numpy as np
import pytest

from oracle import force as of
from paper_2407_08092_gb300 import synth

from .gpu_util import Pair

pytestmark = pytest.mark.gpu


def scratch_limit(ctx, limit, refuse=-1):
    """Sets the context's scratch limits in bytes and returns the slices in use before."""
    from paper_2407_08092_gb300 import lqdd
    f = lqdd.library()._ZN2lq19force_scratch_limitEP6lq_ctxxx
    f.argtypes = [ctypes.c_void_p, ctypes.c_longlong, ctypes.c_longlong]
    f.restype = ctypes.c_int
    return f(ctx, limit, refuse)


class Force:
    def __init__(self, L, t_bc=-1):
        self.p = Pair(L, eps=0.4, seed=1800 + sum(L), m0=0.07, csw=1.0, t_bc=t_bc)
        self.slice = 5184 * (self.p.V // L[3])
        self.X, self.Y = synth.gaussian_spinor(self.p.V, 71), synth.gaussian_spinor(self.p.V, 72)
        self.dX, self.dY = self.p.dev(self.X), self.p.dev(self.Y)

    def __call__(self):
        G = self.p.torch.full_like(self.p.dU, float("nan"))
        self.p.lqdd.lq_force(self.p.ctx, self.dX, self.dY, G)
        return self.p.host(G)

    def oracle(self):
        return of.bilinear_grad(self.p.L, self.p.U, self.X, self.Y, self.p.lat.m0, self.p.lat.csw, self.p.lat.t_bc)


@pytest.mark.parametrize("L", [(4, 2, 2, 2), (4, 4, 2, 4), (6, 4, 2, 6), (2, 4, 6, 10)], ids=lambda L: "x".join(map(str, L)))
def test_force_is_the_same_with_any_scratch(L):
    f = Force(L)
    try:
        whole = f()
        want = f.oracle()
        assert np.abs(whole - want).max() < 1e-12 * np.abs(want).max()
        assert scratch_limit(f.p.ctx, 0) == L[3]
        # none, and rings of 3 slices (ranges of one) up to all but one, remainders among them
        for slots in [0] + list(range(3, L[3] + 1)):
            scratch_limit(f.p.ctx, slots * f.slice + f.slice // 2)
            for _ in range(2):   # the second time in a scratch that holds the first's matrices
                assert np.array_equal(f(), whole), slots
            assert scratch_limit(f.p.ctx, -1) == slots
        # fewer slices than a ring needs
        scratch_limit(f.p.ctx, min(2, L[3] - 1) * f.slice)
        assert np.array_equal(f(), whole)
        assert scratch_limit(f.p.ctx, -1) == 0
    finally:
        f.p.close()


def test_force_when_its_scratch_cannot_be_had():
    f = Force((4, 4, 4, 10))
    try:
        whole = f()
        for most in (9, 5, 3, 2, 0):   # slices that an allocation may have
            scratch_limit(f.p.ctx, -1, most * f.slice)
            for _ in range(2):
                assert np.array_equal(f(), whole), most
            # what could be had is kept: 10 -> 5 -> 3 -> none
            assert scratch_limit(f.p.ctx, -1) == (5 if most >= 5 else 3 if most >= 3 else 0)
    finally:
        f.p.close()


def test_force_scratch_is_given_back_when_memory_is_short():
    f = Force((4, 4, 4, 10))
    lqdd = f.p.lqdd
    try:
        first = f()
        x = f.p.torch.zeros_like(f.dX)
        # workspaces beyond 4 MB cannot be had: 257 FP64 fields (16 MB), 65 x 8 FP32 fields (16 MB)
        def solve():
            prm = lqdd.make_params(solver=lqdd.LQ_SOLVER_GMRES, prec=lqdd.LQ_F64, tol=1e-10, restart=256, max_restarts=2)
            lqdd.lq_solve(f.p.ctx, prm, f.dX, x)

        def batch():
            b = f.dX.unsqueeze(0).repeat(8, 1, 1, 1)
            lqdd.lq_solve_batch(f.p.ctx, lqdd.make_batch_params(tol=1e-10, restart=64), 8, b, f.p.torch.zeros_like(b))

        for call in (solve, batch):
            scratch_limit(f.p.ctx, -1, 4 << 20)
            assert np.array_equal(f(), first)        # 10 slices, 3.3 MB
            with pytest.raises(lqdd.LqError) as err:
                call()
            assert err.value.status == lqdd.LQ_ERR_OOM
            assert np.array_equal(f(), first)
            assert scratch_limit(f.p.ctx, -1) == 5   # half of what it had
            call()                                    # and with memory enough it runs
    finally:
        f.p.close()
