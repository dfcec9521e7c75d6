"""Child process of test_gpu_bounds_large: loads the index-checked library (the
LQ_LIBRARY environment variable names it), runs the library's calls on a lattice
beyond every switch to the small lattices' hopping kernels and on one below, every
caller field surrounded by canary values, compares with the oracle, and prints one
JSON line as bounds_child does."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402
import torch  # noqa: E402

import oracle  # noqa: E402
from paper_2407_08092_gb300 import lqdd, synth  # noqa: E402
from tests.bounds_child import Padded, rel  # noqa: E402

# 27720 sites a parity: the last warp, the last block of 32, 64 and 128 sites and
# the last layout tile are partial; 144: four and a half blocks of the small form
SHAPES = [(18, 10, 14, 22), (6, 4, 2, 6)]
TOL = {lqdd.LQ_F64: 1e-12, lqdd.LQ_F32: 1e-5, lqdd.LQ_DF64: 1e-12, lqdd.LQ_BF16: 1e-2}
OMEGA = 0.8 / 5.2


def main():
    torch.cuda.set_device(0)
    stream = torch.cuda.current_stream().cuda_stream
    errs, failed, fields = {}, [], []

    def check(name, got, want, tol):
        errs[name] = rel(got, want)
        if not errs[name] < tol:
            failed.append(name)

    for L in SHAPES:
        name = "x".join(map(str, L))
        U = synth.gauge_links(L, 0.25, 1600 + sum(L))
        lat = oracle.Lattice(L, U, m0=0.05, csw=1.0, t_bc=-1)
        V, Vh = lat.V, lat.Vh

        def padded(what, shape, init=None):
            p = Padded(shape, init)
            fields.append((f"{name}:{what}", p))
            return p

        ctx = lqdd.lq_create(lqdd.make_lattice(L, -1, 0.05, 1.0), stream)
        try:
            dU = padded("U", (V, 4, 3, 3), U)
            lqdd.lq_set_gauge(ctx, dU.t)
            full = synth.gaussian_spinor(V, 31)
            half = full[:Vh]
            ref = {lqdd.LQ_OP_SCHUR: lat.schur(half), lqdd.LQ_OP_SCHUR_DAG: lat.schur_dag(half),
                   lqdd.LQ_OP_FULL: lat.dirac(full)}
            # the operators, natural output of one parity and of both
            for prec, tol in TOL.items():
                for op, want in ref.items():
                    if prec == lqdd.LQ_BF16 and op == lqdd.LQ_OP_FULL:
                        continue
                    v = full if op == lqdd.LQ_OP_FULL else half
                    x, y = padded("x", v.shape, v), padded("y", v.shape)
                    lqdd.lq_apply(ctx, op, prec, x.t, y.t)
                    check(f"{name}:op{op}:{prec}", y.t.cpu().numpy(), want, tol)
            b, e = padded("b", (V, 4, 3), full), padded("e", (V, 4, 3))
            # smoothers: (outer, inner) precision; df64 around FP32 takes FP32 ends and
            # writes each parity's natural rows by itself
            want = oracle.smoother(lat, full, "richardson", 3, omega=OMEGA)
            for outer, inner in ((lqdd.LQ_DF64, lqdd.LQ_F32), (lqdd.LQ_DF64, lqdd.LQ_BF16),
                                 (lqdd.LQ_DF64, lqdd.LQ_DF64), (lqdd.LQ_F64, lqdd.LQ_F64), (lqdd.LQ_F64, lqdd.LQ_F32)):
                p = lqdd.make_params(smoother=lqdd.LQ_SMOOTH_RICHARDSON, smooth_n=3, omega=OMEGA, inner_prec=inner,
                                     prec=outer)
                e.t.zero_()
                lqdd.lq_smooth(ctx, p, b.t, e.t)
                check(f"{name}:richardson:{outer}:{inner}", e.t.cpu().numpy(), want, max(TOL[outer], TOL[inner]))
            # solves: the residual of the reconstruction included
            for prec in (lqdd.LQ_DF64, lqdd.LQ_F64):
                e.t.zero_()
                prm = lqdd.make_params(solver=lqdd.LQ_SOLVER_GMRES, prec=prec, tol=1e-10, restart=30, max_restarts=200)
                st, _ = lqdd.lq_solve(ctx, prm, b.t, e.t)
                check(f"{name}:solve:{prec}", lat.dirac(e.t.cpu().numpy()), full, 1.001e-10)
                if st != lqdd.LQ_OK:
                    failed.append(f"{name}:solve:{prec}:status")
            # several right-hand sides in one launch
            nb = 3
            hb = np.stack([synth.gaussian_spinor(V, 40 + r) for r in range(nb)])
            B, X = padded("B", (nb, V, 4, 3), hb), padded("X", (nb, V, 4, 3))
            st, _ = lqdd.lq_solve_batch(ctx, lqdd.make_batch_params(tol=1e-10, restart=16), nb, B.t, X.t)
            got = X.t.cpu().numpy()
            for r in range(nb):
                check(f"{name}:batch:{r}", lat.dirac(got[r]), hb[r], 1.001e-10)
            # the force; its values are tested elsewhere
            G = padded("G", (V, 4, 3, 3))
            lqdd.lq_force(ctx, b.t, e.t, G.t)
            if not torch.isfinite(torch.view_as_real(G.t)).all():
                failed.append(f"{name}:force")
        finally:
            lqdd.lq_destroy(ctx)
    bad = [n for n, f in fields if not f.intact()]
    status, checked, violations, first = lqdd.lq_bounds_check()
    print(json.dumps({"checked": checked, "status": status, "violations": violations, "first_code": first,
                      "bad_canaries": bad, "failed": failed, "max_err": errs}), flush=True)


if __name__ == "__main__":
    main()
