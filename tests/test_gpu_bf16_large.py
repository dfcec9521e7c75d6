"""The BF16 Richardson sweep by the kernel of larger lattices (one thread a site);
the 8^4 lattices of the other BF16 tests take twelve threads a site.  Tolerances
are those of the 8^4 tests."""
import numpy as np
import pytest

import oracle
from paper_2407_08092_gb300 import synth

from .gpu_util import Pair, rel

pytestmark = pytest.mark.gpu

OMEGA = 0.8 / 5.2


@pytest.fixture(scope="module")
def pair():
    p = Pair((18, 10, 14, 22), eps=0.25, seed=1700, m0=0.05, csw=1.0, t_bc=-1)   # 27720 sites a parity
    yield p
    p.close()


@pytest.mark.parametrize("outer", [0, 2], ids=["f64", "df64"])
def test_bf16_richardson_smoother_against_oracle(pair, outer):
    from paper_2407_08092_gb300 import lqdd
    r = synth.gaussian_spinor(pair.V, 62)
    prm = lqdd.make_params(prec=outer, smoother=lqdd.LQ_SMOOTH_RICHARDSON, smooth_n=5, omega=OMEGA,
                           inner_prec=lqdd.LQ_BF16)
    out = pair.torch.empty_like(pair.dev(r))
    lqdd.lq_smooth(pair.ctx, prm, pair.dev(r), out)
    assert rel(pair.host(out), oracle.smoother(pair.lat, r, "richardson", 5, omega=OMEGA)) < 1e-2


def test_fgmres_with_bf16_richardson_reaches_1e10(pair):
    from paper_2407_08092_gb300 import lqdd
    b = synth.gaussian_spinor(pair.V, 63)
    x = pair.torch.zeros_like(pair.dev(b))
    prm = lqdd.make_params(solver=lqdd.LQ_SOLVER_FGMRES, prec=lqdd.LQ_DF64, tol=1e-10, restart=10, max_restarts=50,
                           smoother=lqdd.LQ_SMOOTH_RICHARDSON, smooth_n=5, omega=OMEGA, inner_prec=lqdd.LQ_BF16)
    status, _ = lqdd.lq_solve(pair.ctx, prm, pair.dev(b), x)
    assert status == lqdd.LQ_OK
    assert np.linalg.norm(b - pair.lat.dirac(pair.host(x))) / np.linalg.norm(b) <= 1e-10
