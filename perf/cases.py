"""The work this solver is measured on: preconditioner cycles, operator applications and whole
solves, over the sizes, precisions and options that its configurations, benchmark and tests use.

A case is a dict of plain values:
  do      "vcycle" (z = V(nu1, nu2) r), "apply" (y = H x), "solve" or "batch" (independent solves at once)
  field   "const" (k = kh (nx - 1)), "bump" (a Gaussian bump of amplitude 0.3 on it), "mp2" or "mp3" (the
          paper's second and third model problem: Dirichlet low edges, ECS layers on the high ones)
  nx ny nz  interior nodes per axis (nz = 0: two dimensions); layer: ECS nodes per layered side
  mg      precision of the cycle, "c64" or "c128"; pc: "csg" or "csl"
  smoother "jacobi", "rbgs" or "ilu"; galerkin; nu1; nu2; levels (0: down to 8 unknowns an axis)
  method  "bicgstab" or "idr" (IDR(4)); sizes: the batch's interior nodes per axis, comma separated
"""
import math

import numpy as np
import torch

import helm_inputs as hi
from paper_0912_0180_gb300.helm import Helm, solve_batch

THETA = 0.5          # ECS angle of the "const" and "bump" grids
AMP, WIDTH2 = 0.3, 0.02
TOL = 1e-11          # solves are run to a reference solution's tolerance
MAXMV = 6000


def _case(name=None, **kw):
    c = dict(do="vcycle", field="bump", nx=0, ny=0, nz=0, layer=16, kh=0.5, mg="c64", pc="csg", smoother="jacobi",
             galerkin=False, nu1=1, nu2=1, levels=0, method="bicgstab", sizes="")
    c.update(kw)
    return c if name is None else dict(name=name, **c)


def listed():
    return [
        # the cycle of the smallest configuration: a chain of tiny levels, all latency
        _case("vcycle-2d-96-c64-rbgs", field="const", nx=64, ny=64, layer=16, kh=20 / 63, smoother="rbgs"),
        # the benchmark's 640^2 grid, both precisions of its cycle
        _case("vcycle-2d-640-c64", nx=512, ny=512, layer=64),
        _case("vcycle-2d-640-c128", nx=512, ny=512, layer=64, mg="c128"),
        # a grid as large as the paper's third problem at r = 150
        _case("vcycle-2d-2304-c64", nx=2048, ny=2048, layer=128),
        # ragged sizes, red-black smoothing, the shifted Laplacian
        _case("vcycle-2d-odd-c128-rbgs", nx=511, ny=383, layer=29, mg="c128", pc="csl", smoother="rbgs"),
        # the paper's second problem with its Galerkin coarse operators
        _case("vcycle-mp2-galerkin-c128", field="mp2", nx=385, ny=385, layer=128, mg="c128", galerkin=True),
        # the paper's own multigrid (ILU(0), Galerkin, V(0,1)) on its third problem
        _case("vcycle-mp3-ilu-c64", field="mp3", nx=513, ny=513, layer=128, smoother="ilu", galerkin=True, nu1=0),
        # the 160^3 benchmark's cycle and operator
        _case("vcycle-3d-160-c64-rbgs", field="const", nx=128, ny=128, nz=128, layer=16, kh=40 / 127, smoother="rbgs",
              levels=4),
        _case("apply-3d-160", do="apply", field="const", nx=128, ny=128, nz=128, layer=16, kh=40 / 127),
        # a served 3D request: ragged, variable k, default depth, the FP64 cycle
        _case("vcycle-3d-odd-c128", nx=95, ny=111, nz=79, layer=17, kh=0.4, mg="c128"),
        # whole calls: the smallest configuration, alone; an uneven batch
        _case("solve-2d-96-c64", do="solve", field="const", nx=64, ny=64, layer=16, kh=20 / 63, smoother="rbgs"),
        _case("batch-2d-8-c64", do="batch", layer=24, kh=0.45, sizes="63,127,255,63,127,255,63,511"),
    ]


def _log(rng, lo, hi_):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi_)))))


def draw(rng):
    what = rng.choice(["vcycle2"] * 5 + ["vcycle3"] * 3 + ["galerkin", "ilu", "apply2", "apply3", "solve2", "solve3", "batch"])
    mg = rng.choice(["c64", "c128"])
    layer = rng.randint(16, 32)
    kh = rng.uniform(0.3, 0.6)
    pc = rng.choice(["csg", "csg", "csl"])
    field = rng.choice(["const", "bump"])
    if what in ("vcycle2", "apply2"):
        n = _log(rng, 63, 2048)
        ny = max(63, min(2048, int(n * rng.uniform(0.6, 1.4))))
        return _case(do="apply" if what == "apply2" else "vcycle", field=field, nx=n, ny=ny,
                     layer=rng.randint(16, max(16, min(128, n // 8))), kh=kh, mg=mg, pc=pc,
                     smoother=rng.choice(["jacobi", "jacobi", "rbgs"]))
    if what in ("vcycle3", "apply3"):
        n = [_log(rng, 40, 128) for _ in range(3)]
        sm = rng.choice(["jacobi", "rbgs"])
        return _case(do="apply" if what == "apply3" else "vcycle", field=field, nx=n[0], ny=n[1], nz=n[2],
                     layer=rng.randint(8, 16), kh=kh, mg=mg, pc=pc, smoother=sm)
    if what == "galerkin":
        n = _log(rng, 129, 1025)
        return _case(field=rng.choice(["mp2", "mp3"]), nx=n, ny=n, layer=max(16, n // 4), mg=mg, pc=pc, galerkin=True)
    if what == "ilu":
        n = _log(rng, 97, 513)
        return _case(field="mp3", nx=n, ny=n, layer=max(16, n // 4), mg=mg, pc=pc, smoother="ilu", galerkin=True, nu1=0)
    if what == "solve3":
        n = [_log(rng, 32, 80) for _ in range(3)]
        return _case(do="solve", field="const", nx=n[0], ny=n[1], nz=n[2], layer=rng.randint(8, 16), kh=kh, mg=mg, pc=pc)
    if what == "batch":
        sizes = ",".join(str(rng.choice([63, 127, 255])) for _ in range(rng.randint(4, 12)))
        return _case(do="batch", layer=layer, kh=kh, mg=mg, pc=pc, sizes=sizes)
    n = _log(rng, 63, 512)
    return _case(do="solve", field=field, nx=n, ny=max(63, int(n * rng.uniform(0.7, 1.1))), layer=layer, kh=kh, mg=mg, pc=pc,
                 method=rng.choice(["bicgstab", "idr"]))


# ---- what a program has in hand ------------------------------------------------------------------

def _precond(c):
    mp = c["field"].startswith("mp")
    sm = {"jacobi": hi.SM_JACOBI, "rbgs": hi.SM_RBGS, "ilu": hi.SM_ILU}[c["smoother"]]
    kind = hi.PC_CSG_UNIFORM if c["pc"] == "csg" else hi.PC_CSL
    theta = math.pi / 20 if mp else 0.3
    shift = 1 + 0.36j if mp else 1 + 0.5j
    return hi.Precond(kind=kind, theta_beta=theta, shift=shift, nu1=c["nu1"], nu2=c["nu2"], smoother=sm, omega=0.5,
                      max_levels=c["levels"] or 32, galerkin=c["galerkin"])


def _problem(c, n=None):
    """The grid (with phi for the model problems) and the bump its context forms on the device."""
    if c["field"] == "mp2":
        return hi.workload_mp2(n_int=c["nx"], n_l=c["layer"], r=50.0 * (c["nx"] - 1) / 384), None
    if c["field"] == "mp3":
        return hi.workload_mp3(r=90.0 * (c["nx"] - 1) / 1024, n_int=c["nx"], n_l=c["layer"]), None
    dim = 3 if c["nz"] else 2
    ni = (c["nx"], c["ny"], c["nz"])[:dim] if n is None else (n, n)
    # square cells: the extents follow the node counts
    p = hi.make_problem(dim, ni, c["layer"], extent=[(m - 1) / (ni[0] - 1) for m in ni], theta_gamma=THETA,
                        k0=c["kh"] * (ni[0] - 1), rhs="zero")
    bump = None
    if c["field"] == "bump":
        bump = dict(amp=AMP, width2=WIDTH2, centre=tuple(0.5 * e for e in p.extent[:dim]))
    return p, bump


def _vector(p, seed):
    """A residual-like field: a wave packet at a seeded place over seeded noise a hundred times smaller."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    rng = np.random.default_rng(seed)
    shape = p.shape[::-1]
    v = torch.randn(*shape, dtype=torch.complex128, device="cuda", generator=g) * 0.01
    r2, ph = 0.0, 0.0
    for a in range(p.dim):
        x = torch.linspace(0, 1, p.shape[a], dtype=torch.float64, device="cuda")
        x = x.reshape([-1 if d == p.dim - 1 - a else 1 for d in range(p.dim)])
        r2 = r2 + (x - rng.uniform(0.2, 0.8)) ** 2
        ph = ph + 0.25 * rng.uniform(-1, 1) * p.shape[a] * x
    return (v + torch.polar(torch.exp(-r2 / 0.05), ph)).reshape(-1).contiguous()


def _source(p, seed):
    """A point source at a seeded interior node."""
    rng = np.random.default_rng(seed)
    idx = [hi.interior_node_index(p, a, int(rng.integers(1, p.n_int[a] - 1))) for a in range(p.dim)]
    b = torch.zeros(*p.shape[::-1], dtype=torch.complex128, device="cuda")
    b[tuple(idx[::-1])] = 1.0
    return b.reshape(-1)


def _instances(c):
    if c["do"] == "batch":  # every other one with the bump
        return [_problem(dict(c, field="bump" if i % 2 else "const"), int(n)) for i, n in enumerate(c["sizes"].split(","))]
    return [_problem(c)]


def prepare(case, seed):
    c = case
    insts = _instances(c)
    hs = [Helm(p, _precond(c), mg_dtype=c["mg"], k_bump=bump) for p, bump in insts]
    st = {"do": c["do"], "h": hs}
    if c["do"] in ("solve", "batch"):
        st["b"] = [_source(p, seed + 1000 * i) for i, (p, _) in enumerate(insts)]
        st["method"] = hi.IDR if c["method"] == "idr" else hi.BICGSTAB
        st["shadow"] = hi.shadow_space(hs[0].n, 4) if c["method"] == "idr" else None
    else:
        st["r"] = _vector(insts[0][0], seed)
    return st


def run(state):
    h = state["h"]
    if state["do"] == "vcycle":
        return h[0].vcycle(state["r"])
    if state["do"] == "apply":
        return h[0].apply(state["r"])
    if state["do"] == "batch":
        return solve_batch(h, state["b"], method=state["method"], tol=TOL, maxmv=MAXMV)[0]
    return h[0].solve(state["b"][0], method=state["method"], s=4, tol=TOL, maxmv=MAXMV, shadow=state["shadow"])[0]


def _unknowns(c):
    if c["do"] == "batch":
        return sum((int(n) + 2 * c["layer"]) ** 2 for n in c["sizes"].split(","))
    if c["field"].startswith("mp"):
        return (c["nx"] - 1 + c["layer"]) ** 2
    return math.prod(n + 2 * c["layer"] for n in (c["nx"], c["ny"], c["nz"]) if n)


def work(case):
    """Input read and output written once, with phi where it varies; the arithmetic of one cycle (a sweep and a
    residual down, a correction and a sweep up, on every level), of one operator row, or, for a solve, of one
    preconditioned matvec: how many a solve takes is the method's affair."""
    n, dim = _unknowns(case), 3 if case["nz"] else 2
    row = 8 * (2 * dim + 1)                                     # a complex row: real products and sums
    cycle = (3 * row + 30) * n * (8 / 7 if dim == 3 else 4 / 3)
    out = 8 if case["do"] == "vcycle" and case["mg"] == "c64" else 16
    flops = {"vcycle": cycle, "apply": row * n}.get(case["do"], cycle + row * n)
    return {"bytes": n * (16 + out + (0 if case["field"] == "const" else 8)), "flops": flops}


# ---- the same numbers in plain torch, 64 bits ----------------------------------------------------

def _axis(n_int, lo, hi_, extent, theta):
    """Mesh widths (complex) and real positions of the unknowns of one axis."""
    h = extent / (n_int - 1)
    w = [h * np.exp(1j * theta)] * (lo + 1 if lo else 0) + [h + 0j] * (n_int - 1) + [h * np.exp(1j * theta)] * (hi_ + 1 if hi_ else 0)
    w = np.array(w)
    first = -lo if lo else 1
    return w, (first + np.arange(len(w) - 1)) * h


def _rows(w):
    """Shortley-Weller rows of -d2/dz2 for the widths w."""
    l, r = w[:-1], w[1:]
    return -2 / (l * (l + r)), 2 / (l * r), -2 / (r * (l + r))


def _grid(p, bump):
    ax = [_axis(p.n_int[a], *p.n_layer[a], p.extent[a], p.theta_gamma) for a in range(p.dim)]
    shape = [len(x) for _, x in ax][::-1]
    if p.phi is not None:
        phi = torch.from_numpy(p.phi).reshape(shape).cuda()
    elif bump:
        r2 = 0.0
        for a in range(p.dim):
            x = torch.from_numpy(ax[a][1]).cuda() - bump["centre"][a]
            r2 = r2 + x.reshape([-1 if d == p.dim - 1 - a else 1 for d in range(p.dim)]) ** 2
        phi = (p.k0 * (1 + bump["amp"] * torch.exp(-r2 / bump["width2"]))) ** 2
    else:
        phi = torch.full(shape, p.k0 ** 2, dtype=torch.float64, device="cuda")
    return [w for w, _ in ax], phi


class _Op:
    """A level operator: {offset (slowest axis first): weights}; the weights of neighbours outside are zero."""

    def __init__(self, st, shape):
        self.st, self.shape, self.zero = st, list(shape), (0,) * len(shape)
        self.diag = st[self.zero].expand(shape) if st[self.zero].shape != tuple(shape) else st[self.zero]

    def apply(self, x, diag=True):
        y = self.diag * x if diag else torch.zeros_like(x)
        for off, wt in self.st.items():
            if off == self.zero:
                continue
            dst = tuple(slice(max(0, -o), n - max(0, o)) for o, n in zip(off, self.shape))
            src = tuple(slice(max(0, o), n - max(0, -o)) for o, n in zip(off, self.shape))
            y[dst] += wt.expand(self.shape)[dst] * x[src]
        return y


def _sw(ws, phi, s):
    d = len(ws)
    st, diag = {}, -s * phi.to(torch.complex128)
    for a in range(d):
        am, a0, ap = (torch.from_numpy(v).cuda().reshape([-1 if k == d - 1 - a else 1 for k in range(d)]) for v in _rows(ws[a]))
        off = [0] * d
        off[d - 1 - a] = 1
        st[tuple(-o for o in off)], st[tuple(off)] = am, ap
        diag = diag + a0
    st[(0,) * d] = diag
    return _Op(st, phi.shape)


def _fw(r):
    """Full weighting, axis by axis: coarse c gathers fine 2c, 2c+1, 2c+2."""
    for a in range(r.dim()):
        r = r.transpose(0, a)
        nc = r.shape[0] // 2 if r.shape[0] > 1 else 1
        e = torch.cat([r, torch.zeros_like(r[:1])])
        r = (0.25 * e[0:2 * nc:2] + 0.5 * e[1:2 * nc + 1:2] + 0.25 * e[2:2 * nc + 2:2]).transpose(0, a)
    return r


def _interp(e, shape):
    for a in range(e.dim()):
        e = e.transpose(0, a)
        n, nc = shape[a], e.shape[0]
        f = torch.zeros((n,) + tuple(e.shape[1:]), dtype=e.dtype, device=e.device)
        f[1:2 * nc:2] = e
        f[0:2 * nc:2] += 0.5 * e
        k = len(range(2, n, 2))
        f[2:n:2] += 0.5 * e[:k]
        e = f.transpose(0, a)
    return e


def _galerkin(A, cshape):
    """R A P (2D, 3 x 3 box) read off nine probing vectors."""
    cj, ci = torch.meshgrid(*(torch.arange(n, device="cuda") for n in cshape), indexing="ij")
    st = {(b, a): torch.zeros(cshape, dtype=torch.complex128, device="cuda") for b in (-1, 0, 1) for a in (-1, 0, 1)}
    for pj in range(3):
        for pi in range(3):
            v = ((cj % 3 == pj) & (ci % 3 == pi)).to(torch.complex128)
            y = _fw(A.apply(_interp(v, A.shape)))
            for (b, a), w in st.items():
                w += torch.where(((cj + b) % 3 == pj) & ((ci + a) % 3 == pi), y, 0)
    for (b, a), w in st.items():  # no weights to neighbours outside
        if b:
            w[0 if b < 0 else -1] = 0
        if a:
            w[:, 0 if a < 0 else -1] = 0
    return _Op(st, cshape)


class _Ilu:
    """ILU(0) in natural order on the pattern of A, and its solves, along the wavefronts i + 2 j."""
    LOW, UP = [(-1, -1), (-1, 0), (-1, 1), (0, -1)], [(0, 1), (1, -1), (1, 0), (1, 1)]

    def __init__(self, A):
        nj, ni = A.shape
        self.pad = lambda: np.zeros((nj + 2, ni + 2), np.complex128)
        f = {}
        for off in self.LOW + [(0, 0)] + self.UP:
            f[off] = self.pad()
            if off in A.st:
                f[off][1:-1, 1:-1] = A.st[off].expand(A.shape).cpu().numpy()
                if off[0]:
                    f[off][1 if off[0] < 0 else nj] = 0
                if off[1]:
                    f[off][:, 1 if off[1] < 0 else ni] = 0
        f[0, 0][f[0, 0] == 0] = 1
        self.f, self.waves = f, []
        for t in range(ni + 2 * (nj - 1)):
            j = np.arange(max(0, -(-(t - ni + 1) // 2)), min(nj - 1, t // 2) + 1)
            self.waves.append((j + 1, t - 2 * j + 1))
        kept = set(A.st)
        for J, I in self.waves:
            for lo in self.LOW:
                if lo not in kept:
                    continue
                L = f[lo][J, I] / f[0, 0][J + lo[0], I + lo[1]]
                f[lo][J, I] = L
                for up in self.UP:
                    to = (lo[0] + up[0], lo[1] + up[1])
                    if up in kept and to in kept:
                        inside = (I + to[1] >= 1) & (I + to[1] <= ni) & (J + to[0] >= 1) & (J + to[0] <= nj)
                        f[to][J, I] -= np.where(inside, L * f[up][J + lo[0], I + lo[1]], 0)

    def solve(self, r):
        y = self.pad()
        y[1:-1, 1:-1] = r.cpu().numpy()
        for J, I in self.waves:
            y[J, I] -= sum(self.f[o][J, I] * y[J + o[0], I + o[1]] for o in self.LOW)
        for J, I in self.waves[::-1]:
            y[J, I] = (y[J, I] - sum(self.f[o][J, I] * y[J + o[0], I + o[1]] for o in self.UP)) / self.f[0, 0][J, I]
        return torch.from_numpy(y[1:-1, 1:-1].copy()).cuda()


def _levels(c, ws, phi):
    beta = np.exp(1j * _precond(c).theta_beta) if c["pc"] == "csg" else 1.0
    s = 1.0 if c["pc"] == "csg" else complex(_precond(c).shift)
    ws = [w * beta for w in ws]
    ops = [_sw(ws, phi, s)]
    while len(ops) < (c["levels"] or 32) and max(phi.shape) > 8 and min(phi.shape) >= 3:
        ws = [np.array([w[2 * k] + w[2 * k + 1] for k in range((len(w) - 1) // 2)] + [w[2 * ((len(w) - 1) // 2):].sum()]) for w in ws]
        phi = phi[tuple(slice(1, 2 * (n // 2), 2) for n in phi.shape)]
        ops.append(_galerkin(ops[-1], phi.shape) if c["galerkin"] else _sw(ws, phi, s))
    return ops


def _cycle(c, ops, l, f):
    A = ops[l]
    if l == len(ops) - 1:
        n = f.numel()
        M = torch.empty(n, n, dtype=torch.complex128, device="cuda")
        M.zero_()
        idx = torch.arange(n, device="cuda").reshape(A.shape)
        for off, wt in A.st.items():
            dst = tuple(slice(max(0, -o), m - max(0, o)) for o, m in zip(off, A.shape))
            src = tuple(slice(max(0, o), m - max(0, -o)) for o, m in zip(off, A.shape))
            M[idx[dst].reshape(-1), idx[src].reshape(-1)] = wt.expand(A.shape)[dst].reshape(-1)
        return torch.linalg.solve(M, f.reshape(-1)).reshape(A.shape)
    if c["smoother"] == "ilu":
        lu = _Ilu(A)
    elif c["smoother"] == "rbgs":
        red = sum(torch.arange(n, device="cuda").reshape([-1 if d == a else 1 for d in range(f.dim())])
                  for a, n in enumerate(A.shape)) % 2 == 0

    def smooth(u):
        if c["smoother"] == "jacobi":
            return u + 0.5 * (f - A.apply(u)) / A.diag
        if c["smoother"] == "ilu":
            return u + lu.solve(f - A.apply(u))
        for m in (red, ~red):
            u = torch.where(m, (f - A.apply(u, diag=False)) / A.diag, u)
        return u

    u = torch.zeros_like(f)
    for _ in range(c["nu1"]):
        u = smooth(u)
    u = u + _interp(_cycle(c, ops, l + 1, _fw(f - A.apply(u))), A.shape)
    for _ in range(c["nu2"]):
        u = smooth(u)
    return u


def _solved(ws, phi, b):
    """H^-1 b: by the axes' eigenvectors where k is constant, else by block elimination along y; refined twice."""
    H = _sw(ws, phi, 1.0)
    d = b.dim()
    if float(phi.max()) == float(phi.min()):
        vs, lam = [], -phi.to(torch.complex128)
        for a in range(d):  # axis a of the array: ws[d - 1 - a]
            am, a0, ap = _rows(ws[d - 1 - a])
            lv, v = np.linalg.eig(np.diag(a0) + np.diag(am[1:], -1) + np.diag(ap[:-1], 1))
            vs.append((torch.from_numpy(np.linalg.inv(v)).cuda(), torch.from_numpy(v).cuda()))
            lam = lam + torch.from_numpy(lv).cuda().reshape([-1 if k == a else 1 for k in range(d)])

        def inverse(r):
            for a in range(d):
                r = torch.tensordot(vs[a][0], r, dims=([1], [a])).movedim(0, a)
            r = r / lam
            for a in range(d):
                r = torch.tensordot(vs[a][1], r, dims=([1], [a])).movedim(0, a)
            return r
    else:
        am, _, ap = (torch.from_numpy(v).cuda() for v in _rows(ws[1]))
        xm, _, xp = (torch.from_numpy(v).cuda() for v in _rows(ws[0]))
        T = torch.diag(xm[1:], -1) + torch.diag(xp[:-1], 1)
        inv = []
        for j in range(phi.shape[0]):
            D = T + torch.diag(H.diag[j])
            if j:
                D = D - am[j] * ap[j - 1] * inv[-1]
            inv.append(torch.linalg.inv(D))

        def inverse(r):
            g = [inv[0] @ r[0]]
            for j in range(1, len(inv)):
                g.append(inv[j] @ (r[j] - am[j] * g[-1]))
            for j in range(len(inv) - 2, -1, -1):
                g[j] = g[j] - ap[j] * (inv[j] @ g[j + 1])
            return torch.stack(g)
    x = inverse(b)
    for _ in range(2):
        x = x + inverse(b - H.apply(x))
    return x


def exact(case, seed):
    c = case
    got = []
    for i, (p, bump) in enumerate(_instances(c)):
        ws, phi = _grid(p, bump)
        if c["do"] in ("solve", "batch"):
            got.append(_solved(ws, phi, _source(p, seed + 1000 * i).reshape(phi.shape)).reshape(-1))
        else:
            r = _vector(p, seed).reshape(phi.shape)
            got.append((_cycle(c, _levels(c, ws, phi), 0, r) if c["do"] == "vcycle" else _sw(ws, phi, 1.0).apply(r)).reshape(-1))
    return got if c["do"] == "batch" else got[0]
