"""The work that a user of this framework has it do, as cases that can be timed and compared.

The framework solves Carreau Stokes systems with FGMRES and the multilevel GDSW preconditioner.
A program sets a context up once per mesh and partition and then calls it: products with the
operator, evaluations of the nonlinear residual, preconditioner applies inside a Krylov method of
its own, whole solves, Newton steps; or it hands whole problems to the solve server, or solves by
the multigrid whose coarse solver is the GDSW method.  Each of these is a kind of case here:

  spmv    one product with the assembled operator (gdsw_spmv)
  picard  the nonlinear residual at a state: u_k from x, nu(u_k), assembly, lifting, b - A x
  apply   one preconditioner apply in FP64 (gdsw_apply), for a Krylov method of the caller's
  solve   assembly, lifting and one FGMRES solve with FP32 or BF16 local factors.  Mixed-precision
          applies are measured here, inside the FP64 iteration that makes up for their rounding
  newton  one Newton step from a state (gdsw_newton_step), FP32 local factors
  serve   a batch of requests through the solve server: set-up and solve of problems never seen
  mg      one multigrid-preconditioned solve over three grids

`exact` evaluates the same finite-element problem with its own quadrature, matrix-free or as a
dense matrix, in 64 bits; sizes whose dense solution would take longer have no exact value.
"""
import math

import numpy as np
import torch

from paper_2606_01433_gb300 import gdsw, inputs

F64 = torch.float64


def listed():
    return [
        # the smallest product: the 8^3 problem of the tests, a few microseconds, launch-bound
        dict(name="spmv_8", kind="spmv", shape="box", nx=8, ny=8, nz=8, pressure="q1"),
        # the benchmark's channel with obstacles (751 thousand dofs): the operator fills memory
        dict(name="spmv_channel32", kind="spmv", shape="channel", nx=32, ny=32, nz=32, pressure="q1"),
        # nonlinear residual on a small ragged box, as a line search calls it again and again
        dict(name="picard_12x7x9", kind="picard", shape="box", nx=12, ny=7, nz=9, pressure="q1"),
        # the same at the benchmark's size: the re-assembly of every Picard step
        dict(name="picard_channel32", kind="picard", shape="channel", nx=32, ny=32, nz=32, pressure="q1"),
        # one Newton step on the 8^3 problem: Jacobian, small mixed-precision solve, update
        dict(name="newton_8", kind="newton", shape="box", nx=8, ny=8, nz=8, pressure="q1", parts="2x2x2", groups="",
             precision="fp32", tol=1e-12),
        # smallest FP64 apply, two levels: latency of the launch chain
        dict(name="apply64_8", kind="apply", shape="box", nx=8, ny=8, nz=8, pressure="q1", parts="2x2x2", groups=""),
        # FP64 apply on a ragged box with the discontinuous pressure, parts that do not divide the
        # mesh, three levels
        dict(name="apply64_p1disc", kind="apply", shape="box", nx=17, ny=14, nz=12, pressure="p1disc", parts="4x3x3",
             groups="2x2x2"),
        # smallest whole solve of the serving mix, FP32 factors
        dict(name="solve_8", kind="solve", shape="box", nx=8, ny=8, nz=8, pressure="q1", parts="2x2x2", groups="",
             precision="fp32", tol=1e-12),
        # irregular parts: the die on a quarter of its mesh, recursive bisection into 64 parts,
        # BF16 level-1 factors
        dict(name="solve_die_bf16", kind="solve", shape="die", nx=32, ny=32, nz=64, pressure="q1", parts="64",
             groups="8", precision="bf16", tol=1e-10),
        # the benchmark step: channel with obstacles, 4x4x4 parts, three levels, FP32 factors
        dict(name="solve_channel32", kind="solve", shape="channel", nx=32, ny=32, nz=32, pressure="q1", parts="4x4x4",
             groups="2x2x2", precision="fp32", tol=1e-10),
        # four requests of the serving mix at once through the server: set-up bound
        dict(name="serve_8_16", kind="serve", sizes="16,8,12,14", slots=4, tol=1e-10),
        # multigrid on 32^3 with the GDSW coarse solver on 8^3, symmetric V(2,2), FP32 smoothing
        dict(name="mg_32", kind="mg", nx=32, parts="4x4x4", groups="2x2x2,2x2x2", nu=2, tol=1e-10),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _parts_of(n, rng):
    """Boxes per axis: parts of three to six elements, two at least."""
    return max(2, min(4, n // rng.choice((3, 4, 5, 6))))


def draw(rng):
    kind = rng.choice(("spmv", "picard", "newton", "apply", "solve", "solve", "serve", "mg"))
    if kind == "serve":
        sizes = [rng.randint(8, 15) for _ in range(rng.randint(1, 4))]
        return dict(kind=kind, sizes=",".join(map(str, sizes)), slots=rng.choice((2, 4)), tol=1e-10)
    if kind == "mg":
        m = 4 * rng.randint(4, 7)
        return dict(kind=kind, nx=m, parts="2x2x2", groups="", nu=rng.choice((2, 3)), tol=1e-10)
    c = dict(kind=kind, shape="box")
    if kind in ("spmv", "picard"):
        if rng.random() < 0.3:
            m = rng.randint(12, 31)
            c.update(shape="channel", nx=m, ny=m, nz=m)
        else:
            c.update({k: _log_int(rng, 5, 30) for k in ("nx", "ny", "nz")})
        c["pressure"] = rng.choice(("q1", "q1", "p1disc"))
        return c
    if kind == "solve" and rng.random() < 0.25:
        m = 2 * rng.randint(8, 14)
        return dict(c, shape="die", nx=m, ny=m, nz=2 * m, pressure="q1", parts="32", groups="4",
                    precision=rng.choice(("fp32", "bf16")), tol=1e-10)
    hi = dict(newton=14, apply=14, solve=22)[kind]
    c.update({k: _log_int(rng, 6, hi) for k in ("nx", "ny", "nz")})
    p = [_parts_of(c[k], rng) for k in ("nx", "ny", "nz")]
    c["parts"] = "x".join(map(str, p))
    c["groups"] = "2x2x2" if min(p) > 2 else ""
    c["pressure"] = "q1" if kind == "newton" else rng.choice(("q1", "q1", "p1disc"))
    if kind != "apply":
        c["precision"] = rng.choice(("fp32", "fp32", "bf16"))
        c["tol"] = 1e-12 if _dense(c) else 1e-10
    return c


# ---------------------------------------------------------------------------- problems
def _triple(t):
    return tuple(int(v) for v in t.split("x"))


def _problem(case, seed):
    """The problem of a case; the seed gives the frozen velocity and the Carreau exponent."""
    n = 0.3 + 0.6 * np.random.default_rng(seed).random()
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if case["shape"] == "die":
        gr = [int(v) for v in case["groups"].split(",")]
        return inputs.die(nx, ny, nz, nparts=int(case["parts"]), per_group=gr[0], levels=2 + len(gr), seed=seed, n=n)
    parts = _triple(case.get("parts", "1x1x1"))
    groups = tuple(_triple(g) for g in case.get("groups", "").split(",") if g)
    if case["shape"] == "channel":
        p = inputs.channel(nx, parts=parts, groups=groups, levels=2 + len(groups), seed=seed, n=n)
        p.pressure = case["pressure"]
        return p
    return inputs.box_problem(nx, ny, nz, parts, groups=groups, levels=2 + len(groups), form="symmetric", seed=seed,
                              uk_seed=seed, lam=1.0, n=n, nu_inf=1e-3, pressure=case["pressure"])


def _randn(n, seed):
    return torch.randn(n, dtype=F64, device="cuda", generator=torch.Generator("cuda").manual_seed(seed))


def _state_vector(p, seed):
    """A state in the order of the free dofs: the frozen velocity, a small random pressure."""
    m = _Mesh(p, "cpu")
    x = np.zeros(m.n)
    x[:m.nu] = p.uk[m.vnode.numpy()].ravel()
    x[m.nu:] = 0.1 * np.random.default_rng(seed + 1).standard_normal(m.n - m.nu)
    return torch.from_numpy(x).cuda()


def _serve_problems(case, seed):
    rng = np.random.default_rng(seed)
    return [inputs.carreau_cube(int(m), float(rng.uniform(0.3, 1.0)), float(10.0 ** -rng.uniform(1.0, 4.0)),
                                int(rng.integers(0, 2 ** 31 - 1))) for m in case["sizes"].split(",")]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        return dict(kind=kind, server=gdsw.Server(mem_budget_bytes=64 << 30, max_slots=case["slots"]),
                    probs=_serve_problems(case, seed), tol=case["tol"])
    if kind == "mg":
        groups = tuple(_triple(g) for g in case["groups"].split(",") if g)
        probs = inputs.mg_hierarchy(case["nx"], 3, parts=_triple(case["parts"]), groups=groups,
                                    levels=2 + len(groups), seed=seed)
        g = gdsw.Multigrid(probs, pre=case["nu"], post=case["nu"], smoother="fp32", coarse_tol=1e-1, tol=case["tol"],
                           symmetric=True)
        b = _randn(g.n, seed)
        return dict(kind=kind, mg=g, b=b, x=torch.zeros_like(b))
    p = _problem(case, seed)
    if kind in ("spmv", "picard"):
        ctx = gdsw.Context(p, levels=1)
    elif kind == "apply":
        ctx = gdsw.Context(p)
    else:
        ctx = gdsw.Context(p, precision=(case["precision"], "fp32", "fp32"), phi_precision="fp32", tol=case["tol"])
    s = dict(kind=kind, ctx=ctx)
    if kind in ("spmv", "apply"):
        s["x"] = _randn(ctx.n, seed)
        s["y"] = torch.empty_like(s["x"])
    elif kind in ("picard", "newton"):
        s["x0"] = _state_vector(p, seed)
        s["x"], s["b"], s["r"] = (torch.empty_like(s["x0"]) for _ in range(3))
    else:
        s["b"] = torch.empty(ctx.n, dtype=F64, device="cuda")
        s["x"] = torch.empty_like(s["b"])
    return s


def run(state):
    s, kind = state, state["kind"]
    if kind == "spmv":
        s["ctx"].gdsw_spmv(s["x"], s["y"])
        return s["y"]
    if kind == "apply":
        s["ctx"].gdsw_apply(s["x"], s["y"])
        return s["y"]
    if kind == "picard":
        c = s["ctx"]
        c.gdsw_picard_update(s["x0"])
        c.gdsw_reassemble()
        c.gdsw_rhs_lift(s["b"])
        c.gdsw_residual(s["b"], s["x0"], s["r"])
        return s["b"], s["r"]
    if kind == "newton":
        s["x"].copy_(s["x0"])
        s["ctx"].gdsw_picard_update(s["x"])
        s["ctx"].newton_step(s["x"])
        return s["x"]
    if kind == "solve":
        c = s["ctx"]
        c.gdsw_reassemble()
        c.gdsw_rhs_lift(s["b"])
        s["x"].zero_()
        c.gdsw_solve(s["b"], s["x"])
        return s["b"], s["x"]
    if kind == "serve":
        t = [s["server"].gdsw_server_submit(p, tol=s["tol"]) for p in s["probs"]]
        return [s["server"].gdsw_server_wait(q)[1] for q in t]
    s["x"].zero_()
    s["mg"].solve(s["b"], s["x"])
    return s["x"]


# ---------------------------------------------------------------------------- work
_BLOCKS = 512    # 3x3 velocity blocks per element: 125 + 3 * 75 + 3 * 45 + 27 over its own eight nodes
_FILL = dict(box=1.0, channel=0.955, die=0.33)   # fluid share of the voxel box


def _operator(elements):
    """Bytes and flops of one product: values of A and B once, x and y once."""
    n = 25 * elements
    return (72 * _BLOCKS + 24 * 125) * elements + 16 * n, (18 * _BLOCKS + 12 * 125) * elements


def _factors(p):
    """(local dofs, factor entries) of all Schwarz levels; a symmetric inverse is read by half."""
    z = gdsw.Context(p, analyze_only=True).sizes
    return float(sum(z.local_dofs)), float(sum(z.factor_entries))


def _steps(tol, levels):
    return (3.2 if levels == 2 else 7.0) * -math.log10(tol)


def work(case):
    kind = case["kind"]
    if kind == "serve":
        b = f = 0.0
        for p in _serve_problems(case, 1):
            nl, ent = _factors(p)
            s = ent / (1.4 * nl)          # slab size: 1.4 s^2 stored entries per s dofs
            ob, of = _operator(p.n_elems)
            its = _steps(case["tol"], p.levels)
            b += 4 * ent + its * (2 * ent + ob)
            f += 2 * s * s * nl + its * (2 * ent + of)
        return dict(bytes=b, flops=f)
    if kind == "mg":
        e = case["nx"] ** 3 * 8 / 7
        ob, of = _operator(e)
        cycles = 4.0 * -math.log10(case["tol"])
        sweeps = 2 * case["nu"]           # per sweep every patch inverse (FP32) and the operator once
        return dict(bytes=cycles * (sweeps * (4 * 89 * 89 * e + ob / 2) + ob),
                    flops=cycles * (sweeps * (2 * 89 * 89 * e + of) + of))
    e = _FILL[case["shape"]] * case["nx"] * case["ny"] * case["nz"]
    ob, of = _operator(e)
    if kind == "spmv":
        return dict(bytes=ob, flops=of)
    if kind == "picard":
        # A written and read once; element matrices by sum factorisation
        return dict(bytes=2 * ob, flops=30e3 * e + of)
    p = _problem(case, 1)
    nl, ent = _factors(p)
    if kind == "apply":
        return dict(bytes=4 * ent + 40 * nl, flops=2 * ent)
    size = 2 if case["precision"] == "bf16" else 4
    its = _steps(case["tol"], p.levels)
    return dict(bytes=2 * ob + its * (size * ent / 2 + 20 * nl + ob), flops=30e3 * e + its * (2 * ent + of))


# ---------------------------------------------------------------------------- exact values
class _Mesh:
    """Fluid elements, their nodes and the free dofs of a problem (the order of the C header)."""

    def __init__(self, p, device):
        NX, NY = 2 * p.nx + 1, 2 * p.ny + 1
        e = np.flatnonzero(p.mask)
        ex, ey, ez = e % p.nx, (e // p.nx) % p.ny, e // (p.nx * p.ny)
        a = np.arange(27)
        conn = ((2 * ex)[:, None] + a % 3) + NX * (((2 * ey)[:, None] + (a // 3) % 3)
                                                   + NY * ((2 * ez)[:, None] + a // 9))
        active = np.zeros(p.n_nodes, bool)
        active[conn] = True
        free = active & (p.tags != 1) & (p.tags != 2)
        vnode = np.flatnonzero(free)
        if p.pressure == "q1":
            vert = conn[:, [0, 2, 6, 8, 18, 20, 24, 26]]
            pidx = np.full(p.n_nodes, -1)
            nodes = np.unique(vert)
            pidx[nodes] = np.arange(nodes.size)
            pconn, npres = pidx[vert], nodes.size
        else:
            pconn, npres = np.arange(4 * e.size).reshape(-1, 4), 4 * e.size
        self.vnode = torch.from_numpy(vnode).to(device)
        self.conn = torch.from_numpy(conn).to(device)
        self.pconn = torch.from_numpy(pconn).to(device)
        self.nu, self.n, self.nodes, self.h, self.np = 3 * vnode.size, 3 * vnode.size + npres, p.n_nodes, p.h, npres


def _shape(p, device):
    """Gradients of the Q2 basis (27 points x 27 nodes x 3), pressure basis, weights (27)."""
    g = np.array([-math.sqrt(0.6), 0.0, math.sqrt(0.6)])
    gw = np.array([5.0, 8.0, 5.0]) / 9.0
    v = np.stack([g * (g - 1) / 2, 1 - g * g, g * (g + 1) / 2], 1)
    d = np.stack([g - 0.5, -2 * g, g + 0.5], 1)
    q1 = np.stack([(1 - g) / 2, (1 + g) / 2], 1)

    def prod(x, y, z):   # axes: points (z, y, x), basis (z, y, x); x runs fastest
        return np.einsum("ia,jb,kc->kjicba", x, y, z).reshape(27, -1)

    dphi = np.stack([prod(d, v, v), prod(v, d, v), prod(v, v, d)], -1)
    if p.pressure == "q1":
        psi = prod(q1, q1, q1)
    else:
        z, y, x = np.meshgrid(g, g, g, indexing="ij")
        psi = np.stack([np.ones(27), x.ravel(), y.ravel(), z.ravel()], 1)
    w = np.einsum("i,j,k->kji", gw, gw, gw).ravel()
    return [torch.from_numpy(np.ascontiguousarray(t)).to(device) for t in (dphi, psi, w)]


class _Exact:
    """The operator at a nodal velocity, from its weak form."""

    def __init__(self, p, uk=None):
        self.p, self.m = p, _Mesh(p, "cuda")
        self.dphi, self.psi, self.w = _shape(p, "cuda")
        self.dphi = self.dphi * (2.0 / p.h)
        self.w = self.w * (p.h / 2.0) ** 3
        self.g = torch.from_numpy(np.ascontiguousarray(p.g)).cuda()
        dirichlet = torch.from_numpy(np.isin(p.tags, (1, 2))).cuda()
        self.g = torch.where(dirichlet[:, None], self.g, torch.zeros_like(self.g))
        self.at(torch.from_numpy(p.uk).cuda() if uk is None else uk)

    def grad(self, v):
        return torch.einsum("eac,qal->eqcl", v[self.m.conn], self.dphi)

    def at(self, uk):
        p, gr = self.p, self.grad(uk)
        self.D = 0.5 * (gr + gr.transpose(2, 3))
        t = 1.0 + 2.0 * p.lam ** 2 * (self.D ** 2).sum((2, 3))
        self.visc = p.nu_inf + (p.nu0 - p.nu_inf) * t ** ((p.n_carreau - 1) / 2)
        self.slope = 4.0 * (p.nu0 - p.nu_inf) * (p.n_carreau - 1) * p.lam ** 2 * t ** ((p.n_carreau - 3) / 2)

    def nodal(self, x):
        """Velocity at every node (Dirichlet nodes zero) of a vector of free dofs."""
        v = torch.zeros(self.m.nodes, 3, dtype=F64, device="cuda")
        v[self.m.vnode] = x[:self.m.nu].view(-1, 3)
        return v

    def times(self, v, pres):
        """A (v, p) on the free dofs, v given at every node."""
        m, gr = self.m, self.grad(v)
        pq = torch.einsum("ek,qk->eq", pres[m.pconn], self.psi)
        sig = self.visc[..., None, None] * (gr + gr.transpose(2, 3)) - pq[..., None, None] * torch.eye(3, dtype=F64, device="cuda")
        fe = torch.einsum("eqcl,qal,q->eac", sig, self.dphi, self.w)
        ve = torch.zeros(m.nodes, 3, dtype=F64, device="cuda").index_add_(0, m.conn.reshape(-1), fe.reshape(-1, 3))
        div = gr.diagonal(dim1=2, dim2=3).sum(-1)
        pe = -torch.einsum("eq,qk,q->ek", div, self.psi, self.w)
        po = torch.zeros(m.np, dtype=F64, device="cuda").index_add_(0, m.pconn.reshape(-1), pe.reshape(-1))
        return torch.cat([ve[m.vnode].reshape(-1), po])

    def product(self, x):
        return self.times(self.nodal(x), x[self.m.nu:])

    def lift(self):
        return -self.times(self.g, torch.zeros(self.m.np, dtype=F64, device="cuda"))

    def dense(self, newton=False):
        m, E = self.m, self.m.conn.shape[0]
        eye = torch.eye(3, dtype=F64, device="cuda")
        f = self.visc * self.w
        O = torch.einsum("eq,qal,qbm->ealbm", f, self.dphi, self.dphi)
        K = torch.einsum("ealbl,cd->eacbd", O, eye) + O.permute(0, 1, 4, 3, 2)
        if newton:
            t = torch.einsum("eqcl,qal->eqac", self.D, self.dphi)
            K = K + torch.einsum("eq,eqac,eqbd->eacbd", self.slope * self.w, t, t)
        K = K.reshape(E, 81, 81)
        B = -torch.einsum("q,qk,qbd->kbd", self.w, self.psi, self.dphi).reshape(-1, 81)
        num = torch.full((m.nodes,), -1, dtype=torch.int64, device="cuda")
        num[m.vnode] = torch.arange(m.vnode.numel(), device="cuda")
        vd = num[m.conn]
        vd = torch.where(vd[..., None] >= 0, 3 * vd[..., None] + torch.arange(3, device="cuda"), m.n).reshape(E, 81)
        pd = m.nu + m.pconn
        A = torch.zeros(m.n + 1, m.n + 1, dtype=F64, device="cuda")   # the last row and column take the rest
        A.index_put_((vd[:, :, None].expand_as(K), vd[:, None, :].expand_as(K)), K, accumulate=True)
        Be = B.expand(E, *B.shape)
        A.index_put_((pd[:, :, None].expand_as(Be), vd[:, None, :].expand_as(Be)), Be, accumulate=True)
        Bt = Be.transpose(1, 2)
        A.index_put_((vd[:, :, None].expand_as(Bt), pd[:, None, :].expand_as(Bt)), Bt, accumulate=True)
        return A[:m.n, :m.n]


def _dense(case):
    """Whether the dense solution of a case is a matter of seconds."""
    return case["shape"] == "box" and case["nx"] * case["ny"] * case["nz"] <= 520


def exact(case, seed):
    kind = case["kind"]
    if kind in ("serve", "mg", "apply") or (kind in ("solve", "newton") and not _dense(case)):
        return None   # no independent value within seconds
    p = _problem(case, seed)
    if kind == "spmv":
        return _Exact(p).product(_randn(_Mesh(p, "cpu").n, seed))
    if kind == "solve":
        X = _Exact(p)
        b = X.lift()
        return b, torch.linalg.solve(X.dense(), b)
    x = _state_vector(p, seed)
    X = _Exact(p)
    X.at(X.nodal(x) + X.g)
    b = X.lift()
    r = b - X.product(x)
    if kind == "picard":
        return b, r
    return x + torch.linalg.solve(X.dense(newton=True), r)
