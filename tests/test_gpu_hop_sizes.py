"""The two forms of the hopping kernels and their natural output, against the oracle.

Small lattices run twelve threads a site (blocks of 32 sites), larger ones one
thread a site (blocks of 128, of 32 in FP64).  The shapes: 144 sites a parity,
four and a half blocks of the first form; 27720, past the switch in every
precision, whose last warp and last block are partial and whose extents are no
powers of two.  Every hop mode runs: the operators (K1, K2, FULL, both gamma_5
ends), the smoother (PREP, RICH, RECON) and a solve (RES, RECON_RES).
Tolerances are those of the parity and BF16 tests.
"""
import numpy as np
import pytest

import oracle
from paper_2407_08092_gb300 import synth

from .gpu_util import Pair, rel

pytestmark = pytest.mark.gpu

TOL = {0: 1e-12, 1: 1e-5, 2: 1e-12, 3: 1e-2}   # LQ_F64, LQ_F32, LQ_DF64, LQ_BF16


@pytest.fixture(scope="module", params=[(6, 4, 2, 6), (18, 10, 14, 22)], ids=lambda L: "x".join(map(str, L)))
def pair(request):
    p = Pair(request.param, eps=0.25, seed=1400 + sum(request.param), m0=0.05, csw=1.0, t_bc=-1)
    yield p
    p.close()


@pytest.mark.parametrize("prec", [0, 1, 2, 3], ids=["f64", "f32", "df64", "bf16"])
def test_operators_write_natural_fields(pair, prec):
    from paper_2407_08092_gb300 import lqdd
    lat = pair.lat
    full = synth.gaussian_spinor(lat.V, 2100 + lat.V)
    half = full[:lat.Vh]
    assert rel(pair.apply(lqdd.LQ_OP_SCHUR, prec, half), lat.schur(half)) < TOL[prec]
    assert rel(pair.apply(lqdd.LQ_OP_SCHUR_DAG, prec, half), lat.schur_dag(half)) < TOL[prec]
    if prec != 3:
        assert rel(pair.apply(lqdd.LQ_OP_FULL, prec, full), lat.dirac(full)) < TOL[prec]
    # in place: the input is read before the output is written
    x = pair.dev(half)
    lqdd.lq_apply(pair.ctx, lqdd.LQ_OP_SCHUR, prec, x, x)
    assert rel(pair.host(x), lat.schur(half)) < TOL[prec]


@pytest.mark.parametrize("prec", [0, 2], ids=["f64", "df64"])
def test_smoother_and_solve(pair, prec):
    from paper_2407_08092_gb300 import lqdd
    lat = pair.lat
    r = synth.gaussian_spinor(lat.V, 6100 + lat.V)
    omega = 0.8 / 5.2
    for inner, tol in ((prec, TOL[prec]), (1, TOL[1])):
        p = lqdd.make_params(smoother=lqdd.LQ_SMOOTH_RICHARDSON, smooth_n=3, omega=omega, inner_prec=inner, prec=prec)
        e = pair.torch.empty((lat.V, 4, 3), dtype=pair.torch.complex128, device="cuda")
        lqdd.lq_smooth(pair.ctx, p, pair.dev(r), e)
        assert rel(pair.host(e), oracle.smoother(lat, r, "richardson", 3, omega=omega)) < tol
    x = pair.torch.zeros((lat.V, 4, 3), dtype=pair.torch.complex128, device="cuda")
    prm = lqdd.make_params(solver=lqdd.LQ_SOLVER_GMRES, prec=prec, tol=1e-10, restart=30, max_restarts=200)
    status, st = lqdd.lq_solve(pair.ctx, prm, pair.dev(r), x)
    assert status == lqdd.LQ_OK
    true = np.linalg.norm(r - lat.dirac(pair.host(x))) / np.linalg.norm(r)
    assert true <= 1.001e-10 and abs(st.rel_resid_true - true) <= 1e-13


@pytest.mark.parametrize("prec", [0, 1, 2, 3], ids=["f64", "f32", "df64", "bf16"])
def test_point_source(pair, prec):
    """Zeros of either sign take a route of their own into df64 and FP32."""
    from paper_2407_08092_gb300 import lqdd
    x = np.zeros((pair.Vh, 4, 3), dtype=np.complex128)
    x[::3] = complex(-0.0, -0.0)
    x[pair.Vh // 2, 1, 2] = 1.0
    assert rel(pair.apply(lqdd.LQ_OP_SCHUR, prec, x), pair.lat.schur(x)) < TOL[prec]


def test_batch_matches_oracle(pair):
    """Preparation, residuals and reconstruction of several right-hand sides in one launch."""
    from paper_2407_08092_gb300 import lqdd
    n = 3
    b = np.stack([synth.gaussian_spinor(pair.V, 7100 + r) for r in range(n)])
    x = pair.torch.zeros((n, pair.V, 4, 3), dtype=pair.torch.complex128, device="cuda")
    status, stats = lqdd.lq_solve_batch(pair.ctx, lqdd.make_batch_params(tol=1e-10, restart=16), n, pair.dev(b), x)
    assert status == lqdd.LQ_OK
    got = pair.host(x)
    for r in range(n):
        true = np.linalg.norm(b[r] - pair.lat.dirac(got[r])) / np.linalg.norm(b[r])
        assert true <= 1.001e-10 and abs(stats[r].rel_resid_true - true) <= 1e-13


@pytest.mark.parametrize("prec", [0, 1, 2, 3], ids=["f64", "f32", "df64", "bf16"])
def test_apply_replayed_from_a_graph(pair, prec):
    """The overlapped launches of one call, captured and replayed on another input."""
    import torch
    from paper_2407_08092_gb300 import lqdd
    s = torch.cuda.Stream()
    ctx = lqdd.lq_create(lqdd.make_lattice(pair.L, -1, 0.05, 1.0), s.cuda_stream)
    try:
        lqdd.lq_set_gauge(ctx, pair.dU)
        x = pair.dev(synth.gaussian_spinor(pair.Vh, 81))
        out = torch.empty_like(x)
        torch.cuda.synchronize()
        lqdd.lq_apply(ctx, lqdd.LQ_OP_SCHUR, prec, x, out)   # workspaces and links of this precision
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            lqdd.lq_apply(ctx, lqdd.LQ_OP_SCHUR, prec, x, out)
        y = synth.gaussian_spinor(pair.Vh, 82)
        x.copy_(pair.dev(y))
        for _ in range(2):
            g.replay()
        torch.cuda.synchronize()
        assert rel(out.cpu().numpy(), pair.lat.schur(y)) < TOL[prec]
    finally:
        lqdd.lq_destroy(ctx)


@pytest.mark.parametrize("n,m", [(2, 0), (1, 1)])
@pytest.mark.parametrize("block", [(4, 4, 4, 4), (2, 2, 4, 2)])
def test_sap_few_steps(n, m, block):
    """The shortest chains of the block solve's loads ahead: no and one Minimal Residual step."""
    from oracle import sap as osap
    from paper_2407_08092_gb300 import lqdd
    p = Pair((8, 8, 4, 8), eps=0.25, seed=1500, m0=0.05, csw=1.0, t_bc=-1)
    try:
        r = synth.gaussian_spinor(p.V, 93)
        out = p.torch.empty_like(p.dev(r))
        prm = lqdd.make_params(smoother=lqdd.LQ_SMOOTH_SAP, smooth_n=n, smooth_m=m, inner_prec=lqdd.LQ_F32,
                               prec=lqdd.LQ_DF64, sap_block=block)
        lqdd.lq_smooth(p.ctx, prm, p.dev(r), out)
        assert rel(p.host(out), osap.sap(p.lat, r, n, m, block)) < 1e-5
    finally:
        p.close()
