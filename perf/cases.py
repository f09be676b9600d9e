"""The work a program gives this framework, as measurable cases.

A simulation of pressurised cracks repeats a few calls: per load step some Newton
steps; per Newton step one residual (more in the line search), one multigrid
set-up and one GMRES solve; per GMRES iteration one operator apply and one V-cycle
per block.  A gradient adds transposed applies and solves.  The cases are those
calls, one by one, and two whole calls (a GMRES solve, a load step).

Meshes are those of the tests and of the benchmark: (-10, 10)^2, ncx x ncx coarse
cells, ``refine`` global refinements, then ``local`` refinements of the box
|x| <= 2, |y| <= 1 ("box") or of a band around the crack |x| <= 1, y = 0 ("band").
"""
import functools
import math

import torch

import paper_2404_03265_gb300 as pff

HALF = 10.0          # the domain is (-HALF, HALF)^2
NU, GC, KAPPA = 0.2, 1.0, 1e-10


def _case(name, kind, mesh, ncx, refine, local, degree=1, dtype="float64", op="jacobian", modulus=False, block=0):
    c = dict(kind=kind, mesh=mesh, ncx=ncx, refine=refine, local=local, degree=degree, dtype=dtype, op=op,
             modulus=modulus, block=block)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest problem of the test suite (4,293 DoFs): a call is launches and latency
        _case("jacobian-q1-f32-4k", "apply", "box", 4, 3, 2, dtype="float32"),
        # the operator-apply benchmark (4.1M DoFs), FP32: what a mixed-precision Krylov loop calls most
        _case("jacobian-q1-f32-4m", "apply", "box", 16, 6, 2, dtype="float32"),
        # the default GMRES matvec of a crack simulation: FP64 on the band-refined mesh (1.04M DoFs)
        _case("jacobian-q1-f64-1m", "apply", "band", 16, 5, 7),
        # the vector-Jacobian product of the adjoint, with a per-cell modulus, on an odd mesh (197k DoFs)
        _case("transpose-q1-f64-200k", "apply", "box", 7, 5, 2, op="transpose", modulus=True),
        # quadratic elements at the size of the benchmark (16.4M DoFs), FP32
        _case("jacobian-q2-f32-16m", "apply", "box", 16, 6, 2, degree=2, dtype="float32"),
        # quadratic elements, FP64 (267k DoFs, odd band mesh): matvec of a Q2 solve
        _case("jacobian-q2-f64-270k", "apply", "band", 9, 4, 3, degree=2),
        # Newton residual and every line-search trial, on the band mesh (1.04M DoFs)
        _case("residual-q1-1m", "residual", "band", 16, 5, 7),
        # the preconditioner of every GMRES iteration: displacement block of the 1.04M-DoF solve
        _case("vcycle-u-q1-1m", "vcycle", "band", 16, 5, 7, dtype="float32", block=0),
        # the phase-field block, quadratic elements (267k DoFs): many small levels
        _case("vcycle-phi-q2-270k", "vcycle", "band", 9, 4, 3, degree=2, dtype="float32", block=1),
        # what a Newton step does before its linear solve: a new linearisation, the multigrid
        # set-up and the first preconditioner application, on the 1.04M-DoF mesh
        _case("setup-q1-1m", "setup", "band", 16, 5, 7, dtype="float32"),
        # one linear solve of the size of the differentiation workload (65k DoFs)
        _case("gmres-q1-65k", "gmres", "box", 4, 5, 2, dtype="float32"),
        # one load step (Newton, active set, line search, GMRES) of the smallest test problem
        _case("load-step-q1-4k", "step", "box", 4, 3, 2, dtype="float32"),
    ]


# largest DoF count that draw() gives a kind of call (by degree 1, 2): its cost stays below the largest listed one
_MOST = {"apply": 4.0e6, "residual": 1.0e6, "vcycle": 1.0e6, "setup": 3.0e5, "gmres": 6.0e4, "step": 5.0e3}


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "residual", "vcycle", "vcycle", "setup", "gmres", "step"])
    degree = 1 if kind == "step" else rng.choice([1, 1, 2])
    dofs = math.exp(rng.uniform(math.log(3.0e3), math.log(_MOST[kind])))
    ncx = rng.randint(3, 16)
    cells = math.sqrt(dofs / (3.0 * degree * degree))            # cells per side after the global refinements
    refine = max(1, int(math.floor(math.log2(max(cells / ncx, 1.0)))))
    while refine < 2 or (ncx << refine) < 12:
        refine += 1
    ncx = max(3, min(16, int(round(cells / (1 << refine)))))
    mesh = rng.choice(["box", "band"])
    local = rng.randint(1, 2) if mesh == "box" or kind in ("step", "gmres") else rng.randint(1, 5)
    dtype = rng.choice(["float32", "float64"]) if kind == "apply" else "float32"
    op = rng.choice(["jacobian", "transpose"]) if kind in ("apply", "gmres") else "jacobian"
    modulus = kind != "step" and rng.random() < 0.4
    block = rng.randint(0, 1) if kind == "vcycle" else 0
    return _case(None, kind, mesh, ncx, refine, local, degree, dtype, op, modulus, block)


# ---- meshes: built once per program, every solve on them uses the same handle ----

@functools.lru_cache(maxsize=24)
def _mesh(mesh, ncx, refine, local, degree):
    """The mesh handle, and its slots' integer coordinates and flags on the GPU."""
    m = pff.Mesh(-HALF, HALF, -HALF, HALF, ncx, ncx)
    m.refine_global(refine)
    h = math.sqrt(2.0) * 2.0 * HALF / (ncx * 2 ** (refine + local))
    for _ in range(local):
        if mesh == "box":
            m.refine_box(0, -2.0, 2.0, -1.0, 1.0)
        else:
            m.refine_box(1, -1.0 - 2.0 * h, 1.0 + 2.0 * h, -2.0 * h, 2.0 * h)
    m.finalize(degree)
    X, Y, F = (torch.from_numpy(a).cuda() for a in m.slots())
    return m, X, Y, F


def _mesh_of(case):
    return _mesh(case["mesh"], case["ncx"], case["refine"], case["local"], case["degree"])


def _inputs(case, seed):
    """The caller's data in slot layout (FP64): a state near a pressurised crack, and what the call is applied to."""
    m, X, Y, F = _mesh_of(case)
    g = torch.Generator(device="cuda").manual_seed(int(seed))

    def uniform(*shape):
        return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)

    n, info = X.numel(), m.info
    node, boundary, hanging = (F & 1) == 1, (F & 2) == 2, (F & 4) == 4
    x = -HALF + X.double() * (2.0 * HALF / info["x_max"])
    y = -HALF + Y.double() * (2.0 * HALF / info["y_max"])
    eps = 2.0 * info["h_min"]
    s = uniform(8).tolist()
    p = 1e-3 * (1.0 + s[0])
    d = dict(p=p, eps=eps)
    zero = torch.zeros((), dtype=torch.float64, device="cuda")
    if case["kind"] in ("apply", "residual"):
        # a general state: phase field between broken and sound, small displacements
        phi, phit = uniform(n), uniform(n)
        u = 1e-3 * normal(2, n)
        active = uniform(n) < 0.02
    else:
        # the phase field of a crack of half length 1 (profile of width eps, a little uneven), the
        # displacement of its opening
        dist = torch.sqrt(torch.clamp(x.abs() - 1.0, min=0.0) ** 2 + y * y)
        uneven = 1e-3 * (1.0 + torch.sin(3.0 * x + 6.0 * s[1]) * torch.cos(2.0 * y + 6.0 * s[2]))
        phi = torch.clamp(1.0 - (0.93 + 0.05 * s[3]) * torch.exp(-dist / eps) - uneven, 0.0, 1.0)
        phit = torch.clamp(phi + 0.01 * s[4], max=1.0)
        opening = 2.0 * p * torch.sqrt(torch.clamp(1.0 - (x / 1.2) ** 2, min=0.0))
        u = torch.stack([-0.3 * opening * x * torch.exp(-y.abs()),
                         opening * torch.tanh(y / eps) * torch.exp(-y.abs())]) * (0.8 + 0.4 * s[5])
        u = u * (1.0 + 1e-3 * normal(2, n))
        active = (phi < 0.3 + 0.2 * s[6])
    d["phi"], d["phit"] = (torch.where(node, f, zero) for f in (phi, phit))
    d["u"] = torch.where(node & ~boundary, u, zero)
    d["active"] = (active & node & ~hanging).to(torch.uint8)
    d["x"] = torch.where(node, normal(3, n), zero)
    if case["modulus"]:
        d["E"] = torch.exp(0.1 * normal(info["n_leaf_cells"]) - 0.005)
    return d


def prepare(case, seed):
    m = _mesh_of(case)[0]
    d = _inputs(case, seed)
    pb = pff.Problem(m, E=1.0, nu=NU, Gc=GC, eps=d["eps"], kappa=KAPPA, p=d["p"])
    if case["modulus"]:
        pb.set_cell_modulus(d["E"])
    pb.set_state(d["u"], d["phi"], d["phit"])
    pb.set_active(d["active"])
    st = dict(kind=case["kind"], pb=pb, block=case["block"], transpose=case["op"] == "transpose")
    st["op"] = pff.PFF_OP_TRANSPOSE if st["transpose"] else pff.PFF_OP_JACOBIAN
    kind = case["kind"]
    if kind == "apply":
        v = d["x"].to(getattr(torch, case["dtype"]))
        st.update(xu=v[:2].contiguous(), xp=v[2].contiguous())
        st.update(yu=torch.empty_like(st["xu"]), yp=torch.empty_like(st["xp"]))
    elif kind == "residual":
        st.update(u=d["u"], phi=d["phi"], phit=d["phit"], R=torch.empty_like(d["x"]))
    else:
        st["mg"] = pff.MG(pb, pff.PFF_F32 if case["dtype"] == "float32" else pff.PFF_F64)
        if kind == "vcycle":
            st["mg"].setup()
            st["r"] = (d["x"][:2] if case["block"] == 0 else d["x"][2]).contiguous()
            st["z"] = torch.empty_like(st["r"])
        elif kind == "setup":
            st.update(u=d["u"], phi=d["phi"], phit=d["phit"], active=d["active"])
            st.update(ru=d["x"][:2].contiguous(), rp=d["x"][2].contiguous())
            st.update(zu=torch.empty_like(st["ru"]), zp=torch.empty_like(st["rp"]))
        elif kind == "gmres":
            st["mg"].setup()
            st.update(b=d["x"], sol=torch.empty_like(d["x"]))
        else:  # one load step from the state at rest, phi_old the crack of the step before
            st.update(phi_old=d["phi"], u=torch.empty_like(d["u"]), phi=torch.empty_like(d["phi"]),
                      active=torch.empty_like(d["active"]))
    return st


def run(st):
    kind, pb = st["kind"], st["pb"]
    if kind == "apply":
        pb.apply(st["xu"], st["xp"], st["yu"], st["yp"], op=st["op"])
        return [st["yu"], st["yp"]]
    if kind == "residual":
        pb.residual(st["u"], st["phi"], st["phit"], st["R"])
        return [st["R"]]
    if kind == "vcycle":
        st["mg"].vcycle(st["block"], st["r"], st["z"])
        return [st["z"]]
    if kind == "setup":
        pb.set_state(st["u"], st["phi"], st["phit"])
        pb.set_active(st["active"])
        st["mg"].setup()
        st["mg"].vcycle(0, st["ru"], st["zu"])
        st["mg"].vcycle(1, st["rp"], st["zp"])
        return [st["mg"].lam(0), st["mg"].lam(1), st["zu"], st["zp"]]
    if kind == "gmres":
        pff.gmres(pb, st["mg"], st["b"], st["sol"], rtol=1e-6, transpose=st["transpose"])
        return [st["sol"]]
    st["u"].zero_()
    st["phi"].copy_(st["phi_old"])
    st["active"].zero_()
    pff.newton_step(pb, st["mg"], st["u"], st["phi"], st["phi_old"], st["active"])
    return [st["u"], st["phi"], st["active"]]


def work(case):
    """Bytes: vectors and linearisation once, in the call's precision.  Flops: the sum-factorised cell
    loops (about 0.5 kflop per Q1 cell and 3 kflop per Q2 cell for the whole Jacobian)."""
    info = _mesh_of(case)[0].info
    n, cells = info["n_nodes"], info["n_leaf_cells"]
    size = 4 if case["dtype"] == "float32" else 8
    full = (500.0 if case["degree"] == 1 else 3000.0) * cells
    kind = case["kind"]
    if kind == "apply":
        return {"bytes": float(size * (10 * n + (cells if case["modulus"] else 0))), "flops": full}
    if kind == "residual":
        return {"bytes": 8.0 * 7 * n, "flops": 0.7 * full}
    # a V-cycle of one block: six level applies on about 4/3 of the leaf cells
    comps = 2 if case["block"] == 0 else 1
    vbytes, vflops = 16.0 * comps * n + size * (4 + comps) * n * 4 / 3, 6 * 0.3 * comps * full * 4 / 3
    if kind == "vcycle":
        return {"bytes": vbytes, "flops": vflops}
    both_b, both_f = 48.0 * n + size * 11 * n * 4 / 3, 6 * 0.9 * full * 4 / 3
    if kind == "setup":  # twelve applies of the eigenvalue estimate per level and block, then a V-cycle each
        return {"bytes": 32.0 * n + both_b, "flops": 3 * both_f}
    # an iterative solve: its data once; an apply and a V-cycle of both blocks per iteration
    iterations = 15 if kind == "gmres" else 60
    return {"bytes": 80.0 * n, "flops": iterations * (both_f + full)}


# ---- the same results in 64 bits: the weak form of the residual on the leaf cells, its derivatives by autograd ----

def _constraints(m, X, Y, F, degree):
    """Cell nodes (cells, nodes per cell) as slots, and hanging slots with their parents and weights."""
    info = m.info
    lij = torch.from_numpy(m.leaf_cells()).cuda().long()
    lev, ci, cj = lij.unbind(1)
    step = torch.bitwise_left_shift(torch.ones_like(lev), info["finest_level"] - lev)   # node spacing of the cell
    wide = info["x_max"] + 1
    slots = torch.nonzero((F & 1) == 1).flatten()
    keys, order = torch.sort(Y[slots].long() * wide + X[slots].long())
    slots = slots[order]

    def find(xx, yy):
        k = yy * wide + xx
        at = torch.searchsorted(keys, k).clamp(max=keys.numel() - 1)
        return slots[at], keys[at] == k

    k = degree
    nodes = torch.stack([find((ci * k + a) * step, (cj * k + b) * step)[0] for b in range(k + 1) for a in range(k + 1)], 1)
    hang, par, wgt = [], [], []
    # a node halfway between two neighbouring nodes of a cell's edge that the cell does not have hangs on that edge
    half = [([0, 1], 0.5)] if k == 1 else [([0, 1, 2], 0.25), ([0, 1, 2], 0.75)]
    for side in range(4):
        for ids, t in half:
            along = (ci if side < 2 else cj) * k * step + (k * step * int(round(4 * t))) // 4
            across = ((cj if side < 2 else ci) + side % 2) * k * step
            ok = step >= 2
            s, there = find(*((along, across) if side < 2 else (across, along)))
            sel = torch.nonzero(ok & there & ((F[s] & 4) == 4)).flatten()
            w = [1 - t, t] if k == 1 else [2 * (t - .5) * (t - 1), -4 * t * (t - 1), 2 * t * (t - .5)]
            e = side % 2 * k
            cols = [(i + (k + 1) * e) if side < 2 else (e + (k + 1) * i) for i in ids]
            hang.append(s[sel])
            par.append(nodes[sel][:, cols])
            wgt.append(torch.tensor(w, dtype=torch.float64, device="cuda").expand(sel.numel(), k + 1))
    return lev, nodes, torch.cat(hang), torch.cat(par), torch.cat(wgt)


class _Form:
    """A(U)(W): the semilinear form on slot vectors (3, n_slots), U and W extended to the hanging nodes."""

    def __init__(self, case, d):
        self.m, X, Y, self.F = _mesh_of(case)
        k = case["degree"]
        lev, self.nodes, self.hang, self.par, self.wgt = _constraints(self.m, X, Y, self.F, k)
        assert self.hang.unique().numel() == int(((self.F & 4) == 4).sum())
        self.h = (2.0 * HALF / case["ncx"]) * torch.pow(0.5, lev.double())
        t = {1: [0.5 - math.sqrt(1 / 12), 0.5 + math.sqrt(1 / 12)], 2: [0.5 - math.sqrt(0.15), 0.5, 0.5 + math.sqrt(0.15)]}[k]
        w = {1: [0.5, 0.5], 2: [5 / 18, 8 / 18, 5 / 18]}[k]
        if k == 1:
            L, D = [[1 - q, q] for q in t], [[-1.0, 1.0] for q in t]
        else:
            L = [[2 * (q - .5) * (q - 1), -4 * q * (q - 1), 2 * q * (q - .5)] for q in t]
            D = [[4 * q - 3, 4 - 8 * q, 4 * q - 1] for q in t]
        T = functools.partial(torch.tensor, dtype=torch.float64, device="cuda")
        L, D, w = T(L), T(D), T(w)
        nb = (k + 1) ** 2
        self.N = torch.einsum("pa,qb->pqba", L, L).reshape(nb, nb)       # value of basis (b, a) at point (p, q)
        self.Nx = torch.einsum("pa,qb->pqba", D, L).reshape(nb, nb)
        self.Ny = torch.einsum("pa,qb->pqba", L, D).reshape(nb, nb)
        self.JxW = torch.einsum("p,q->pq", w, w).reshape(1, nb) * (self.h * self.h)[:, None]
        self.E = d["E"][:, None] if "E" in d else 1.0
        self.mu, self.lam = 0.5 / (1 + NU), NU / ((1 + NU) * (1 - 2 * NU))
        self.p, self.eps = d["p"], d["eps"]
        self.phit = self.cells(d["phit"][None])[0]
        f = self.F
        node, hanging = (f & 1) == 1, (f & 4) == 4
        self.u_free = node & ~hanging & ((f & 2) == 0)
        self.node = node & ~hanging

    def cells(self, v):
        if self.hang.numel():
            v = v.clone()
            v[:, self.hang] = (v[:, self.par] * self.wgt).sum(-1)
        return v[:, self.nodes]

    def __call__(self, U, W):
        c, t = self.cells(U), self.cells(W)
        ih = 1.0 / self.h[:, None]
        val = lambda f: f @ self.N.T
        dx = lambda f: (f @ self.Nx.T) * ih
        dy = lambda f: (f @ self.Ny.T) * ih
        phi, phit = val(c[2]), val(self.phit)
        e11, e22, g12 = dx(c[0]), dy(c[1]), dy(c[0]) + dx(c[1])
        s11 = self.E * ((2 * self.mu + self.lam) * e11 + self.lam * e22)
        s22 = self.E * ((2 * self.mu + self.lam) * e22 + self.lam * e11)
        s12 = self.E * self.mu * g12
        g = (1 - KAPPA) * phit * phit + KAPPA
        w11, w22, w12, wp = dx(t[0]), dy(t[1]), dy(t[0]) + dx(t[1]), val(t[2])
        a = g * (s11 * w11 + s22 * w22 + s12 * w12) + phit * phit * self.p * (w11 + w22)
        a = a + ((1 - KAPPA) * phi * (s11 * e11 + s22 * e22 + s12 * g12) + 2 * self.p * phi * (e11 + e22)) * wp
        a = a + GC * (self.eps * (dx(c[2]) * dx(t[2]) + dy(c[2]) * dy(t[2])) - (1 - phi) / self.eps * wp)
        return (a * self.JxW).sum()

    def product(self, U, x, transpose):
        """G x or G^T x at U, condensed, on every slot."""
        U = U.clone().requires_grad_(True)
        W = (x.clone() if transpose else torch.zeros_like(x)).requires_grad_(True)
        q = torch.autograd.grad(self(U, W), U, create_graph=not transpose)[0]
        return q.detach() if transpose else torch.autograd.grad((q * x).sum(), W)[0]

    def diagonal(self):
        """About the diagonal (each hanging node's share with squared weights), to precondition with."""
        mo, ih = 2 * self.mu + self.lam, 1.0 / self.h[:, None]
        g = self.E * ((1 - KAPPA) * (self.phit @ self.N.T) ** 2 + KAPPA) * self.JxW * ih * ih
        gx, gy = g @ (self.Nx ** 2), g @ (self.Ny ** 2)
        m = GC * ((self.JxW @ (self.N ** 2)) / self.eps + self.eps * ((self.JxW * ih * ih) @ (self.Nx ** 2 + self.Ny ** 2)))
        out = torch.zeros(3, self.F.numel(), dtype=torch.float64, device="cuda")
        for c, v in enumerate((mo * gx + self.mu * gy, self.mu * gx + mo * gy, m)):
            out[c].index_add_(0, self.nodes.flatten(), v.flatten())
            out[c].index_add_(0, self.par.flatten(), (out[c][self.hang][:, None] * self.wgt ** 2).flatten())
        return out


def _cg(A, b, dinv, free, tol=1e-13, most=4000):
    x, r = torch.zeros_like(b), torch.where(free, b, torch.zeros_like(b))
    z = dinv * r
    p, rz, r0 = z.clone(), (r * z).sum(), r.norm()
    for i in range(most):
        if i % 20 == 0 and r.norm() <= tol * r0:
            break
        q = torch.where(free, A(p), torch.zeros_like(p))
        a = rz / (p * q).sum()
        x, r = x + a * p, r - a * q
        z = dinv * r
        new = (r * z).sum()
        p, rz = z + (new / rz) * p, new
    return x


def exact(case, seed):
    kind = case["kind"]
    # no value but the algorithm's own: a V-cycle (its smoothing ranges are estimates), a load step
    # (its result is where the iteration stops); a GMRES solution only at sizes that plain CG solves in seconds
    if kind in ("vcycle", "setup", "step") or (kind == "gmres" and _mesh_of(case)[0].info["n_nodes"] > 30000):
        return None
    d = _inputs(case, seed)
    f = _Form(case, d)
    U = torch.cat([d["u"], d["phi"][None]])
    zero = torch.zeros((), dtype=torch.float64, device="cuda")
    if kind == "residual":
        W = torch.zeros_like(U).requires_grad_(True)
        R = -torch.autograd.grad(f(U, W), W)[0]
        return [torch.where(torch.stack([f.u_free, f.u_free, f.node]), R, zero)]
    free = torch.stack([f.u_free, f.u_free, f.node & (d["active"] == 0)])
    fixed = torch.stack([(f.F & 3) == 3] * 2 + [f.node & (d["active"] != 0)])
    transpose = case["op"] == "transpose"

    def G(x):
        return torch.where(free, f.product(U, torch.where(free, x, zero), transpose), zero)

    if kind == "apply":
        x = d["x"].to(getattr(torch, case["dtype"])).double()
        y = torch.where(fixed, x, G(x))
        return [y[:2], y[2]]
    # block triangular: the blocks one after the other, the coupling on the right-hand side
    b, diag = d["x"], f.diagonal()
    dinv = torch.where(free & (diag > 0), 1.0 / torch.where(diag > 0, diag, torch.ones_like(diag)), zero)
    blocks = [torch.stack([free[0], free[1], free[2] & False]), torch.stack([free[0] & False, free[1] & False, free[2]])]
    x = torch.zeros_like(b)
    for blk in blocks[::-1] if transpose else blocks:
        x = x + _cg(lambda v: G(torch.where(blk, v, zero)), b - G(x), dinv, blk)
    return [torch.where(fixed, b, x)]
