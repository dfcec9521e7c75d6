"""FP32 and BF16 operators on either side of the switch to the kernels of small
lattices (20480 sites a parity), where the twelve-thread kernel runs several waves
of blocks.  Tolerances are those of the parity and BF16 tests."""
import pytest

import oracle
from paper_2407_08092_gb300 import synth

from .gpu_util import Pair, rel

pytestmark = pytest.mark.gpu

TOL = {1: 1e-5, 3: 1e-2}   # LQ_F32, LQ_BF16


@pytest.fixture(scope="module", params=[(16, 16, 10, 16), (14, 18, 10, 18)], ids=["20480", "22680"])
def pair(request):
    p = Pair(request.param, eps=0.25, seed=1900 + sum(request.param), m0=0.05, csw=1.0, t_bc=-1)
    yield p
    p.close()


@pytest.mark.parametrize("prec", [1, 3], ids=["f32", "bf16"])
def test_operators_and_sweep(pair, prec):
    from paper_2407_08092_gb300 import lqdd
    full = synth.gaussian_spinor(pair.V, 65)
    half = full[:pair.Vh]
    assert rel(pair.apply(lqdd.LQ_OP_SCHUR, prec, half), pair.lat.schur(half)) < TOL[prec]
    assert rel(pair.apply(lqdd.LQ_OP_SCHUR_DAG, prec, half), pair.lat.schur_dag(half)) < TOL[prec]
    omega = 0.8 / 5.2
    p = lqdd.make_params(smoother=lqdd.LQ_SMOOTH_RICHARDSON, smooth_n=3, omega=omega, inner_prec=prec, prec=lqdd.LQ_F64)
    e = pair.torch.empty((pair.V, 4, 3), dtype=pair.torch.complex128, device="cuda")
    lqdd.lq_smooth(pair.ctx, p, pair.dev(full), e)
    assert rel(pair.host(e), oracle.smoother(pair.lat, full, "richardson", 3, omega=omega)) < TOL[prec]
