"""The work that a program gives this library, as cases to be timed.

A program that uses the library holds one context per lattice and gauge field
and calls the C ABI through ``lqdd``: it loads a gauge field, applies the
operator, smooths, solves for one or many right-hand sides and takes the
fermion force.  The cases go from the 8^4 test lattice, where a call is a few
launches long, to the 32^3 x 64 benchmark lattice, over the four precisions,
with the sizes of the tests and the benchmark and with extents that are no
power of two.  Inputs are those of ``synth``: near-unit SU(3) links
exp(i eps sum_k a_k lambda_k) with a_k ~ N(0, 1) (drawn on the GPU here), and
Gaussian spinors or the point sources of a propagator.

Fields cross the boundary as complex doubles whatever the precision inside.
A smoother's correction is computed in single precision and goes into the
next single-precision step, so those cases take it as complex64.

``exact`` restates each operation in complex double torch, from the operator's
formula alone.
"""
from __future__ import annotations

import math

import torch

from paper_2407_08092_gb300 import lqdd

F64, F32, DF64, BF16 = lqdd.LQ_F64, lqdd.LQ_F32, lqdd.LQ_DF64, lqdd.LQ_BF16
PREC = {"f64": F64, "f32": F32, "df64": DF64, "bf16": BF16}
OPS = {"full": lqdd.LQ_OP_FULL, "schur": lqdd.LQ_OP_SCHUR, "schur_dag": lqdd.LQ_OP_SCHUR_DAG}
OMEGA = 0.8 / 5.2          # Richardson weight of the tests
TOL = 1e-10                # relative residual of every solve


def _case(kind, L, m0=0.05, eps=0.25, **more):
    return dict(kind=kind, Lx=L[0], Ly=L[1], Lz=L[2], Lt=L[3], m0=m0, eps=eps, csw=1.0, t_bc=-1, **more)


def listed():
    return [
        # the outer operator on the smallest lattice in use: a call is its launches
        dict(_case("apply", (8, 8, 8, 8), op="schur", prec="df64"), name="apply_df64_8x4"),
        # the inner operator at the benchmark's size
        dict(_case("apply", (32, 32, 32, 64), m0=0.02, op="schur", prec="f32"), name="apply_f32_32x64"),
        # the adjoint, as normal equations take it, on extents that are no power of two
        dict(_case("apply", (18, 10, 14, 22), op="schur_dag", prec="df64"), name="dagger_df64_18x10x14x22"),
        # a residual of the full system in native double precision
        dict(_case("apply", (16, 16, 16, 32), op="full", prec="f64"), name="full_f64_16x32"),
        # the operator in half-width storage
        dict(_case("apply", (24, 24, 24, 48), op="schur", prec="bf16"), name="apply_bf16_24x48"),
        # a new configuration: links and clover term in, then the residual's operator in df64
        dict(_case("gauge", (24, 24, 24, 48)), name="new_gauge_24x48"),
        # one smoother call of a multigrid or preconditioned solver, both kinds
        dict(_case("smooth", (24, 24, 24, 48), smoother="richardson", n=5, m=1), name="richardson_24x48"),
        dict(_case("smooth", (24, 24, 24, 48), smoother="sap", n=3, m=4), name="sap_24x48"),
        # the propagator of a point: twelve spin-colour sources on two lattices together
        dict(_case("group", (16, 16, 16, 32), rhs=12, Lx2=8, Ly2=8, Lz2=8, Lt2=8, rhs2=12), name="group_12rhs_16x32_8x4"),
        # a mixed-precision solve at the benchmark's size
        dict(_case("solve", (32, 32, 32, 64), m0=0.02), name="solve_32x64"),
        # molecular dynamics: the force of given fields, and action with gradient on a small lattice
        dict(_case("force", (24, 24, 24, 48)), name="force_24x48"),
        dict(_case("action", (8, 8, 8, 8)), name="action_backward_8x4"),
    ]


def _extents(rng, vmax, step=2, least=4):
    """Four extents, multiples of `step`, whose volume is spread over its logarithm up to vmax."""
    target = math.exp(rng.uniform(math.log(least ** 4), math.log(vmax)))
    side = target ** 0.25
    L = []
    for mu in range(4):
        v = side * math.exp(rng.uniform(-0.35, 0.35)) * (1.5 if mu == 3 else 0.87)
        L.append(max(least, step * round(v / step)))
    while L[0] * L[1] * L[2] * L[3] > vmax:
        k = max(range(4), key=lambda i: L[i])
        L[k] -= step
    return tuple(L)


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "gauge", "smooth", "smooth", "group", "solve", "force", "action"])
    big = 24 ** 3 * 48
    if kind == "apply":
        prec = rng.choice(["f64", "f32", "df64", "bf16"])
        op = rng.choice(["schur", "schur_dag"] + ([] if prec == "bf16" else ["full"]))
        return _case("apply", _extents(rng, 32 ** 3 * 64 if prec != "f64" else big), op=op, prec=prec)
    if kind == "smooth":
        if rng.random() < 0.5:
            return _case("smooth", _extents(rng, big), smoother="richardson", n=rng.randint(1, 6), m=1)
        return _case("smooth", _extents(rng, big, step=8, least=8), smoother="sap", n=rng.randint(1, 4), m=rng.randint(1, 6))
    if kind == "group":
        L2 = _extents(rng, 8 ** 4)
        return _case("group", _extents(rng, 12 ** 3 * 24), rhs=rng.randint(1, 12), Lx2=L2[0], Ly2=L2[1], Lz2=L2[2],
                     Lt2=L2[3], rhs2=rng.randint(1, 12))
    if kind == "action":
        return _case("action", _extents(rng, 8 ** 4))
    return _case(kind, _extents(rng, big))


def _ext(case):
    return (case["Lx"], case["Ly"], case["Lz"], case["Lt"])


def _ext2(case):
    return (case["Lx2"], case["Ly2"], case["Lz2"], case["Lt2"])


def _volume(L):
    return L[0] * L[1] * L[2] * L[3]


# ---- inputs -----------------------------------------------------------------------

def _mul(a, b):
    """Products of 3x3 matrices [..., 3, 3]."""
    return (a.unsqueeze(-1) * b.unsqueeze(-3)).sum(-2)


def _links(L, eps, gen):
    """exp(i eps sum_k a_k lambda_k), a_k ~ N(0, 1): U[V, 4, 3, 3] complex128."""
    V = _volume(L)
    out = torch.empty((4 * V, 3, 3), dtype=torch.complex128, device="cuda")
    eye = torch.eye(3, dtype=torch.complex128, device="cuda")
    chunk = 1 << 20
    for lo in range(0, 4 * V, chunk):
        n = min(chunk, 4 * V - lo)
        a = torch.randn((n, 8), dtype=torch.float64, device="cuda", generator=gen) * eps
        H = torch.zeros((n, 3, 3), dtype=torch.complex128, device="cuda")
        for k, (i, j) in ((0, (0, 1)), (3, (0, 2)), (5, (1, 2))):   # lambda_1,2 lambda_4,5 lambda_6,7
            z = torch.complex(a[:, k], -a[:, k + 1])
            H[:, i, j], H[:, j, i] = z, z.conj()
        s = a[:, 7] / math.sqrt(3.0)
        H[:, 0, 0], H[:, 1, 1], H[:, 2, 2] = a[:, 2] + s, s - a[:, 2], -2 * s
        X = H * (1j / 16)
        E = eye + X / 12
        for q in range(11, 0, -1):          # Taylor sum to order 12 of X = iH/16
            E = eye + _mul(X, E) / q
        for _ in range(4):
            E = _mul(E, E)
        out[lo:lo + n] = E
    return out.view(V, 4, 3, 3)


def _gauss(shape, gen):
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), dtype=torch.float64, device="cuda", generator=gen))


def _points(L, n, gen):
    """Point sources of a propagator, one spin and colour after the other, at one site."""
    V = _volume(L)
    b = torch.zeros((n, V, 4, 3), dtype=torch.complex128, device="cuda")
    x = int(torch.randint(V, (1,), generator=gen, device="cuda"))
    for r in range(n):
        b[r, x, r % 4, (r // 4) % 3] = 1.0
    return b


def _inputs(case, seed):
    """Everything drawn from the seed, in one order for prepare() and exact()."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    L, kind = _ext(case), case["kind"]
    V = _volume(L)
    d = {"U": _links(L, case["eps"], gen)}
    if kind == "apply":
        d["x"] = _gauss((V if case["op"] == "full" else V // 2, 4, 3), gen)
    elif kind == "force":
        d["X"], d["Y"] = _gauss((V, 4, 3), gen), _gauss((V, 4, 3), gen)
    elif kind == "group":
        d["b"] = _points(L, case["rhs"], gen)
        d["U2"] = _links(_ext2(case), case["eps"], gen)
        d["b2"] = _points(_ext2(case), case["rhs2"], gen)
    else:
        d["x"] = _gauss((V, 4, 3), gen)
    return d


class _Held:
    """What a program keeps: contexts, fields and parameters."""

    def __init__(self):
        self.ctxs, self.grp = [], None

    def context(self, case, L, U):
        ctx = lqdd.lq_create(lqdd.make_lattice(L, case["t_bc"], case["m0"], case["csw"]),
                             torch.cuda.current_stream().cuda_stream)
        self.ctxs.append(ctx)
        if U is not None:
            lqdd.lq_set_gauge(ctx, U)
        return ctx

    def __del__(self):
        if self.grp is not None:
            lqdd.lq_group_destroy(self.grp)
        for ctx in self.ctxs:
            lqdd.lq_destroy(ctx)


def _mixed():
    """The mixed solve of the benchmark: df64 FGMRES(10) around FP32 GMRES(8) to 1e-5."""
    return lqdd.make_params(solver=lqdd.LQ_SOLVER_FGMRES, prec=DF64, tol=TOL, restart=10, max_restarts=20,
                            smoother=lqdd.LQ_SMOOTH_GMRES, smooth_n=40, smooth_m=8, smooth_tol=1e-5, inner_prec=F32)


def prepare(case, seed):
    kind, L = case["kind"], _ext(case)
    s = _Held()
    s.kind = kind
    s.__dict__.update(_inputs(case, seed))
    if kind == "action":
        from paper_2407_08092_gb300.autograd import FermionAction
        s.action = FermionAction(L, case["m0"], case["csw"], t_bc=case["t_bc"], params=_mixed())
        s.U.requires_grad_(True)
        return s
    s.ctx = s.context(case, L, None if kind == "gauge" else s.U)
    if kind == "apply":
        s.op, s.prec, s.out = OPS[case["op"]], PREC[case["prec"]], torch.empty_like(s.x)
    elif kind == "gauge":
        s.out = torch.empty_like(s.x)
    elif kind == "smooth":
        sap = case["smoother"] == "sap"
        s.params = lqdd.make_params(prec=DF64, inner_prec=F32, omega=OMEGA, smooth_n=case["n"], smooth_m=case["m"],
                                    smoother=lqdd.LQ_SMOOTH_SAP if sap else lqdd.LQ_SMOOTH_RICHARDSON)
        s.out = torch.empty_like(s.x)
    elif kind == "solve":
        s.params, s.out = _mixed(), torch.empty_like(s.x)
    elif kind == "group":
        ctx2 = s.context(case, _ext2(case), s.U2)
        s.params = lqdd.make_batch_params(tol=TOL)
        s.grp = lqdd.lq_group_create([s.ctx, ctx2], torch.cuda.current_stream().cuda_stream)
        s.out, s.out2 = torch.empty_like(s.b), torch.empty_like(s.b2)
    elif kind == "force":
        s.out = torch.empty_like(s.U)
    return s


def _solved(status):
    if status != lqdd.LQ_OK:
        raise RuntimeError(lqdd.lq_status_string(status))


def run(s):
    if s.kind == "apply":
        lqdd.lq_apply(s.ctx, s.op, s.prec, s.x, s.out)
        return s.out
    if s.kind == "gauge":
        lqdd.lq_set_gauge(s.ctx, s.U)
        lqdd.lq_apply(s.ctx, lqdd.LQ_OP_FULL, DF64, s.x, s.out)
        return s.out
    if s.kind == "smooth":
        lqdd.lq_smooth(s.ctx, s.params, s.x, s.out)
        return s.out.to(torch.complex64)
    if s.kind == "solve":
        s.out.zero_()
        _solved(lqdd.lq_solve(s.ctx, s.params, s.x, s.out)[0])
        return s.out
    if s.kind == "group":
        s.out.zero_()
        s.out2.zero_()
        _solved(lqdd.lq_solve_group(s.grp, s.ctx, s.params, [s.b, s.b2], [s.out, s.out2])[0])
        return [s.out, s.out2]
    if s.kind == "force":
        lqdd.lq_force(s.ctx, s.X, s.Y, s.out, coef=-2.0)
        return s.out
    S = s.action(s.U, s.x)
    G, = torch.autograd.grad(S, s.U)
    return [S.detach(), G]


# ---- the work of one pass --------------------------------------------------------------

# bytes of a link and of a site's clover pair as the library stores them, and flops of
# one parity's hops with its clover term (1320 for the hops, 552 for the blocks, 24 for a sum)
_LINK = {"f64": 144, "df64": 144, "f32": 48, "bf16": 24}
_CLOVER = {"f64": 576, "df64": 576, "f32": 288, "bf16": 288}


def _one_operator(prec, V):
    """Links and both clover fields of one application, and its flops, on V sites."""
    return V * (4 * _LINK[prec] + _CLOVER[prec]), V // 2 * 3768


def work(case):
    kind, L = case["kind"], _ext(case)
    V = _volume(L)
    full = 192 * V                                   # a full spinor of complex doubles
    if kind == "apply":
        b, f = _one_operator(case["prec"], V)
        return {"bytes": b + (2 if case["op"] == "full" else 1) * full, "flops": f}
    if kind == "gauge":
        # links in; df64 and FP32 links, clover blocks and the odd inverses out; the operator's fields.
        # Field strengths from plaquettes: three and two times two 3x3 products (198) a plane.
        return {"bytes": V * 576 + V * (4 * 192 + 864) + V // 2 * 864 + 2 * full,
                "flops": V * 6 * 1206 + V // 2 * 3000 + V // 2 * 3768}
    if kind == "smooth":
        b, f = _one_operator("f32", V)
        n = case["n"] if case["smoother"] == "richardson" else case["n"] * (case["m"] + 1)
        return {"bytes": b + full + 96 * V, "flops": f * (n + 1)}
    if kind == "solve":
        # source and solution once; about 30 applications of the FP32 operator, whose vectors
        # (in, intermediate written and read, in again, out: 480 bytes an even site) cannot stay on the chip
        b, f = _one_operator("f32", V)
        return {"bytes": 30 * (b + 240 * V) + 3 * full, "flops": 33 * f}
    if kind == "group":
        t = {"bytes": 0.0, "flops": 0.0}
        for Lm, n in ((L, case["rhs"]), (_ext2(case), case["rhs2"])):
            b, f = _one_operator("f32", _volume(Lm))
            t["bytes"] += 30 * (b + n * 240 * _volume(Lm)) + 3 * n * 192 * _volume(Lm)
            t["flops"] += 33 * n * f
        return t
    # the gradient: 4 links in and out, two spinors in; per plane and link eight leaf terms that share
    # their products between neighbours (about four 3x3 products each plane and link end)
    force = {"bytes": V * 2 * 576 + 2 * full, "flops": V * (12 * 4 * 198 + 4 * 672)}
    if kind == "force":
        return force
    b, f = _one_operator("f32", V)
    return {"bytes": force["bytes"] + 60 * (b + 240 * V), "flops": force["flops"] + 66 * f}


# ---- the same in complex double torch ------------------------------------------------

_PLANES = ((0, 1), (0, 2), (1, 2), (0, 3), (1, 3), (2, 3))


def _gammas():
    s = torch.tensor([[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]], dtype=torch.complex128)
    g = torch.zeros((4, 4, 4), dtype=torch.complex128)
    for k in range(3):
        g[k, :2, 2:], g[k, 2:, :2] = -1j * s[k], 1j * s[k]
    g[3, :2, 2:] = g[3, 2:, :2] = torch.eye(2)
    return g.cuda()


def _dag(m):
    return m.conj().transpose(-1, -2)


class _Exact:
    """D = C - 1/2 sum_mu [(1 - g_mu) U_mu(x) delta_{x+mu} + (1 + g_mu) U_mu(x-mu)^+ delta_{x-mu}]."""

    def __init__(self, case, L, U):
        self.L, self.U, self.V = L, U, _volume(L)
        self.g, self.eye = _gammas(), torch.eye(4, dtype=torch.complex128, device="cuda")
        self.bc = case["t_bc"]
        dev = U.device
        c, r = [], torch.arange(self.V, device=dev)
        for mu in range(4):
            c.append(r % L[mu])
            r = r // L[mu]
        self.c = c
        self.parity = (c[0] + c[1] + c[2] + c[3]) & 1
        self.even, self.odd = torch.nonzero(self.parity == 0)[:, 0], torch.nonzero(self.parity == 1)[:, 0]
        F = {}
        for mu, nu in _PLANES:
            um, un = U[:, mu], U[:, nu]
            dn = lambda x, *k: self._shift(x, k, -1)  # noqa: E731  the value at x - mu
            up = lambda x, k: self._shift(x, (k,), +1)  # noqa: E731
            P = _mul(_mul(um, up(un, mu)), _dag(_mul(un, up(um, nu))))
            Q2 = _mul(_mul(un, _dag(up(dn(um, mu), nu))), _mul(_dag(dn(un, mu)), dn(um, mu)))
            Q3 = _mul(_dag(_mul(dn(un, mu, nu), dn(um, mu))), _mul(dn(um, mu, nu), dn(un, nu)))
            Q4 = _mul(_mul(_dag(dn(un, nu)), dn(um, nu)), _mul(up(dn(un, nu), mu), _dag(um)))
            Q = P + Q2 + Q3 + Q4
            F[(mu, nu)] = (Q - _dag(Q)) / 8
        # C as two 6x6 blocks (spins 0,1 and 2,3; colour fastest)
        C = torch.zeros((2, self.V, 2, 3, 2, 3), dtype=torch.complex128, device=dev)
        for (mu, nu), f in F.items():
            sig = 0.5j * (self.g[mu] @ self.g[nu] - self.g[nu] @ self.g[mu])
            for b in range(2):
                sb = sig[2 * b:2 * b + 2, 2 * b:2 * b + 2]
                C[b] = C[b] + case["csw"] * 0.5j * torch.einsum("st,vab->vsatb", sb, f)
        self.C = C.reshape(2, self.V, 6, 6) + (4 + case["m0"]) * torch.eye(6, dtype=torch.complex128, device=dev)
        self.Cinv = None

    def _shift(self, x, mus, s):
        """x at the neighbour s steps along each of mus (s = +1: the value at x + mu)."""
        L = self.L
        y = x.reshape((L[3], L[2], L[1], L[0]) + x.shape[1:])
        for mu in mus:
            y = torch.roll(y, -s, 3 - mu)
        return y.reshape(x.shape)

    def hop(self, p, keep=None):
        """sum over the eight neighbours; keep[(mu, s)]: which sites take that neighbour."""
        out = torch.zeros_like(p)
        for mu in range(4):
            for s in (+1, -1):
                h = p if s > 0 else (self.U[:, mu].conj().unsqueeze(1) * p.unsqueeze(-1)).sum(-2)  # U^+ at the source
                h = self._shift(h, (mu,), s)
                if s > 0:
                    h = (self.U[:, mu].unsqueeze(1) * h.unsqueeze(-2)).sum(-1)
                h = torch.einsum("st,vta->vsa", self.eye - s * self.g[mu], h)
                if mu == 3 and self.bc < 0:
                    edge = self.c[3] == (self.L[3] - 1 if s > 0 else 0)
                    h = torch.where(edge[:, None, None], -h, h)
                if keep is not None:
                    h = h * keep[(mu, s)][:, None, None]
                out = out + h
        return out

    def site(self, C, p):
        y = [(C[b] * p[:, 2 * b:2 * b + 2].reshape(-1, 1, 6)).sum(-1).reshape(-1, 2, 3) for b in range(2)]
        return torch.cat(y, 1)

    def D(self, p):
        return self.site(self.C, p) - 0.5 * self.hop(p)

    def inv(self, p):
        if self.Cinv is None:
            self.Cinv = torch.linalg.inv(self.C)
        return self.site(self.Cinv, p)

    def on(self, which, p):
        return p * (self.parity == which)[:, None, None]

    def schur(self, xe):
        """D_S on a full-lattice field that vanishes on the odd sites."""
        t = self.inv(self.on(1, -0.5 * self.hop(xe)))
        return self.site(self.C, xe) + self.on(0, 0.5 * self.hop(t))

    def prepare(self, r):
        return self.on(0, r) + self.on(0, 0.5 * self.hop(self.inv(self.on(1, r))))

    def reconstruct(self, r, xe):
        return xe + self.inv(self.on(1, r) + self.on(1, 0.5 * self.hop(xe)))

    def solve(self, b):
        """D x = b by BiCGStab on the Schur system to 1e-15."""
        bh = self.prepare(b)
        x = torch.zeros_like(bh)
        r, r0 = bh.clone(), bh.clone()
        rho = al = om = 1.0
        v = p = torch.zeros_like(bh)
        stop = 1e-15 * float(bh.norm())
        for _ in range(400):
            rho1 = torch.vdot(r0.reshape(-1), r.reshape(-1))
            p = r + (rho1 / rho) * (al / om) * (p - om * v)
            v = self.schur(p)
            al = rho1 / torch.vdot(r0.reshape(-1), v.reshape(-1))
            q = r - al * v
            t = self.schur(q)
            om = torch.vdot(t.reshape(-1), q.reshape(-1)) / torch.vdot(t.reshape(-1), t.reshape(-1))
            x = x + al * p + om * q
            r, rho = q - om * t, rho1
            if float(r.norm()) <= stop:
                break
        return self.reconstruct(b, x)

    def sap(self, b, n, m):
        """SAP(n, m) from zero with 4^4 blocks (2 where the extent is 2), Algorithm 1."""
        B = [4 if length % 4 == 0 else 2 for length in self.L]
        blk, colour, mult = 0, 0, 1
        for mu in range(4):
            k = self.c[mu] // B[mu]
            blk, colour, mult = blk + mult * k, colour + k, mult * (self.L[mu] // B[mu])
        keep = {}
        for mu in range(4):
            for s in (+1, -1):
                pos = self.c[mu] % B[mu]
                inside = pos != (B[mu] - 1 if s > 0 else 0)
                keep[(mu, s)] = inside if self.L[mu] > B[mu] else torch.ones_like(inside)

        def dot(a, c):
            w = (a.conj() * c).reshape(self.V, 12).sum(1)
            return torch.zeros(mult, dtype=w.dtype, device=w.device).index_add_(0, blk, w)

        def schur(v):
            return self.site(self.C, v) + self.on(0, 0.5 * self.hop(self.inv(self.on(1, -0.5 * self.hop(v, keep))), keep))

        x = torch.zeros_like(b)
        for _ in range(n):
            for col in (0, 1):
                r = (b - self.D(x)) * ((colour & 1) == col)[:, None, None]
                q = self.on(0, r) + self.on(0, 0.5 * self.hop(self.inv(self.on(1, r)), keep))
                e = torch.zeros_like(b)
                for _ in range(m):
                    p = schur(q)
                    pp = dot(p, p).real
                    al = torch.where(pp > 0, dot(p, q) / pp.clamp(min=1e-300), torch.zeros_like(dot(p, q)))[blk]
                    e = e + al[:, None, None] * q
                    q = q - al[:, None, None] * p
                e = e + self.inv(self.on(1, r) + self.on(1, 0.5 * self.hop(e, keep)))
                x = x + e
        return x


def exact(case, seed):
    kind, L = case["kind"], _ext(case)
    V = _volume(L)
    if (kind == "solve" and V > 20000) or (kind == "group" and V > 20000):
        return None                                   # tens of seconds of double-precision iterations
    d = _inputs(case, seed)
    if kind == "force" or kind == "action":
        d["U"].requires_grad_(True)
    if kind == "group":
        outs = []
        for Lm, U, b in ((L, d["U"], d["b"]), (_ext2(case), d["U2"], d["b2"])):
            e = _Exact(case, Lm, U)
            outs.append(torch.stack([e.solve(v) for v in b]))
        return outs
    if kind == "force":
        e = _Exact(case, L, d["U"])
        b = (d["Y"].conj() * e.D(d["X"])).sum().real
        return -2.0 * torch.autograd.grad(b, d["U"])[0]
    if kind == "action":
        with torch.no_grad():
            e = _Exact(case, L, d["U"])
            g5 = torch.tensor([1.0, 1, -1, -1], dtype=torch.float64, device="cuda")[None, :, None]
            Y = g5 * e.solve(g5 * d["x"])
            X = e.solve(Y)
        e = _Exact(case, L, d["U"])
        b = (Y.conj() * e.D(X)).sum().real
        return [(Y.abs() ** 2).sum(), -2.0 * torch.autograd.grad(b, d["U"])[0]]
    e = _Exact(case, L, d["U"])
    x = d["x"]
    if kind == "gauge":
        return e.D(x)
    if kind == "solve":
        return e.solve(x)
    if kind == "smooth":
        if case["smoother"] == "sap":
            return e.sap(x, case["n"], case["m"])
        bh = e.prepare(x)
        xe = OMEGA * bh
        for _ in range(1, case["n"]):
            xe = xe + OMEGA * (bh - e.schur(xe))
        return e.reconstruct(x, xe)
    if case["op"] == "full":
        return e.D(x)
    g5 = torch.tensor([1.0, 1, -1, -1], dtype=torch.float64, device="cuda")[None, :, None]
    f = torch.zeros((V, 4, 3), dtype=torch.complex128, device="cuda")
    f[e.even] = x if case["op"] == "schur" else g5 * x
    y = e.schur(f)[e.even]
    return y if case["op"] == "schur" else g5 * y
