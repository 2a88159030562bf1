"""Workloads that stand for what a program does with this library, each one call of a public entry
point of ``paper_1012_4307_gb300.helm`` on data that is already on the GPU:

  apply         y = A x on a grid (the operator by itself: residuals, checks, other outer solvers)
  precondition  one multigrid cycle from zero on an outer vector (the solvers' preconditioner call,
                also what a user's own outer iteration calls), complex64 or complex128
  solve         A x = f to a relative residual, FGMRES or Bi-CGSTAB around that cycle
  backward      the reverse step of a solve: the adjoint solve and the gradients by k^2 and f
  batch         many independent problems of several sizes and energies in one call

Grids are [-1, 1]^dim with exterior-complex-scaled layers beyond 0.75 of every half width (the
shorter axes of an oblong grid are cut so that the spacing is the same everywhere).  The
wavenumber fields are the repository's own: a Gaussian well with growth toward the boundary up to
k h = 0.6 ("well", workloads.k2_well_growth) with an energy drawn from [0.5, 4], or a constant k
(the paper's first model problem and the parity configuration).
"""
import math

import torch

from paper_1012_4307_gb300 import helm, workloads

THETA = math.pi / 6  # angle of the absorbing layers
LAYER = 0.75         # where they start, as a part of the half width
KH = 0.6             # largest k h of a well field

_BASE = {"op": "precondition", "dim": 2, "nx": 129, "ny": 129, "nz": 1, "field": "well", "k": 0.0, "prec": "c64",
         "pc": "csg", "smoother": "jacobi", "nu": 2, "omega": 0.8, "gamma_c": 1, "coarsest_n": 17, "method": "none",
         "gs": "fp64", "restart": 0, "tol": 0.0, "count": 1, "tuned": False}


def _case(**kw):
    c = dict(_BASE)
    c.update(kw)
    return c


def listed():
    return [
        # The smallest call in use: one cycle on the smallest grid of the batch workload. A program
        # with its own outer iteration calls it once a step, so its latency is what counts.
        _case(name="cycle-2d-129-c64", nx=129, ny=129),
        # The same call on the benchmark's grid (levels that fit the L2 cache).
        _case(name="cycle-2d-1025-c64", nx=1025, ny=1025),
        # The cycle of the 3D workload, every fine vector larger than the L2 cache.
        _case(name="cycle-3d-257-c64", dim=3, nx=257, ny=257, nz=257, coarsest_n=9),
        # The paper's tables run F cycles in double precision: the grid of its second and third
        # model problems (640 cells a side) with one sweep each way and the shifted Laplacian.
        _case(name="cycle-2d-641-c128-f", nx=641, ny=641, prec="c128", pc="csl", nu=1, gamma_c=3),
        # A double-precision 3D cycle on an oblong grid with red-black smoothing, the plain method
        # that results are checked against.
        _case(name="cycle-3d-oblong-c128-rb", dim=3, nx=193, ny=129, nz=97, prec="c128", smoother="rb", nu=1,
              omega=1.0, coarsest_n=9),
        # The operator alone in double precision on a ragged 3D grid: a true residual.
        _case(name="apply-3d-ragged-c128", op="apply", dim=3, nx=225, ny=193, nz=161, prec="c128", coarsest_n=9),
        # The benchmark's solve as it runs it: autotuned complex64 cycle, float-pair Arnoldi process.
        _case(name="solve-2d-1025-mixed", op="solve", nx=1025, ny=1025, method="fgmres", gs="dcgs2", restart=30,
              tol=1e-10, tuned=True),
        # The solve that a user gets without choosing anything (complex64 cycle, double-precision
        # Arnoldi process), on the grid of the adjoint workload.
        _case(name="solve-2d-513-default", op="solve", nx=513, ny=513, method="fgmres", restart=30, tol=1e-10),
        # The 3D solve in mixed precision on a grid between the sizes of the tests and the benchmark.
        _case(name="solve-3d-161-mixed", op="solve", dim=3, nx=161, ny=161, nz=161, coarsest_n=9, method="fgmres",
              gs="dcgs2", restart=20, tol=1e-10),
        # The paper's own method on its first model problem's grid: Bi-CGSTAB with a
        # double-precision F cycle, constant k, a point source.
        _case(name="bicgstab-2d-385-c128", op="solve", nx=385, ny=385, field="constant", k=40.0, prec="c128", nu=1,
              gamma_c=3, method="bicgstab", tol=1e-11),
        # The backward direction: the adjoint solve and both gradients, at the size of a design loop
        # that steps through many of them.
        _case(name="backward-2d-257", op="backward", nx=257, ny=257, method="fgmres", restart=30, tol=1e-10),
        # A batch of energies on the four grids of the batch workload.
        _case(name="batch-12", op="batch", nx=1025, ny=1025, method="fgmres", gs="dcgs2", restart=30, tol=1e-10,
              count=12),
    ]


# Every grid the levels nest in: a coarsest grid of m cells a side doubled k times, so that sizes
# such as 161 = 10 * 2^4 + 1 or 193 = 12 * 2^4 + 1 come up beside 2^k + 1.
def _size(rng, lo, hi, m_lo, m_hi):
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    best = [m * 2 ** k + 1 for m in range(m_lo, m_hi + 1) for k in range(1, 12) if lo <= m * 2 ** k + 1 <= hi]
    near = sorted(best, key=lambda n: abs(math.log(n / want)))
    return near[rng.randrange(3)]


def _near(rng, n, m_lo, m_hi):
    """A second side for an oblong grid: half to all of n, as coarsenable as the levels need."""
    k = 0
    while (n - 1) % 2 ** (k + 1) == 0 and (n - 1) // 2 ** (k + 1) >= m_lo:
        k += 1
    m = (n - 1) // 2 ** k
    return max(m_lo, rng.randint((m + 1) // 2, m)) * 2 ** k + 1


def draw(rng):
    """One more case: the same operations over the same ranges of sizes, types and options."""
    op = rng.choice(["cycle2", "cycle2", "cycle3", "apply", "solve2", "solve2", "solve3", "bicgstab", "backward", "batch"])
    if op == "cycle2":
        n = _size(rng, 65, 1281, 8, 16)
        prec = rng.choice(["c64", "c64", "c128"])
        kw = dict(nx=n, ny=_near(rng, n, 8, 16), prec=prec, pc=rng.choice(["csg", "csg", "csl"]))
        if prec == "c128" or rng.random() < 0.3:
            kw.update(nu=1, gamma_c=rng.choice([1, 2, 3]), smoother=rng.choice(["jacobi", "jacobi", "rb"]))
        return _case(**kw)
    if op in ("cycle3", "apply"):
        prec = rng.choice(["c64", "c128"])
        n = _size(rng, 49, 257 if prec == "c64" or op == "apply" else 209, 4, 8)
        kw = dict(dim=3, nx=n, ny=_near(rng, n, 4, 8), nz=_near(rng, n, 4, 8), prec=prec, coarsest_n=9)
        if op == "apply":
            return _case(op="apply", **kw)
        return _case(smoother=rng.choice(["jacobi", "jacobi", "rb"]), nu=rng.choice([1, 2]), **kw)
    if op in ("solve2", "backward"):
        n = _size(rng, 97, 1025 if op == "solve2" else 513, 8, 16)
        gs = rng.choice(["dcgs2", "fp64", "df"])
        return _case(op=op.rstrip("2"), nx=n, ny=n, method="fgmres", gs=gs, restart=rng.choice([20, 30]), tol=1e-10,
                     prec=rng.choice(["c64", "c64", "c128"]) if n <= 513 else "c64",
                     tuned=gs == "dcgs2" and rng.random() < 0.5)
    if op == "solve3":
        n = _size(rng, 49, 161, 4, 8)
        return _case(op="solve", dim=3, nx=n, ny=n, nz=n, coarsest_n=9, method="fgmres",
                     gs=rng.choice(["dcgs2", "fp64"]) if n <= 129 else "dcgs2", restart=20, tol=1e-10)
    if op == "bicgstab":
        n = _size(rng, 129, 449, 8, 16)
        return _case(op="solve", nx=n, ny=n, field="constant", k=round(rng.uniform(10.0, 40.0), 2),
                     prec=rng.choice(["c128", "c128", "c64"]), nu=1, gamma_c=rng.choice([1, 2, 3]), method="bicgstab",
                     tol=1e-11)
    return _case(op="batch", nx=1025, ny=1025, method="fgmres", gs="dcgs2", restart=30, tol=1e-10,
                 count=rng.randint(5, 12))


# ---------------------------------------------------------------------------------- inputs
def _axes(c):
    """Half width and nodes of every axis, x first."""
    n = [c["nx"], c["ny"], c["nz"]][:c["dim"]]
    return [((m - 1) / (max(n) - 1), m) for m in n]


def _coords(axes):
    out = []
    for a, (w, m) in enumerate(axes):
        shape = [1] * len(axes)
        shape[len(axes) - 1 - a] = m
        out.append(torch.linspace(-w, w, m, dtype=torch.float64, device="cuda").reshape(shape))
    return out


def _k2(c, axes, energy):
    shape = [m for _, m in reversed(axes)]
    if c["field"] == "constant":
        return torch.full(shape, c["k"] ** 2, dtype=torch.float64, device="cuda")
    r2 = sum(x * x for x in _coords(axes))
    corner = sum(w * w for w, _ in axes)
    h = 2.0 / (max(m for _, m in axes) - 1)
    growth = ((KH / h) ** 2 / 2.0 - energy - 5.0 * math.exp(-corner / 0.04)) / corner ** 2
    return (2.0 * (energy + 5.0 * torch.exp(-r2 / 0.04) + growth * r2 * r2)).expand(shape).contiguous()


def _inside(shape):
    """0 on the boundary nodes, 1 elsewhere."""
    m = torch.zeros(shape, dtype=torch.float64, device="cuda")
    m[tuple(slice(1, -1) for _ in shape)] = 1.0
    return m


def _random(axes, gen):
    """A vector as the outer solvers hand it over: unit norm, values everywhere inside."""
    shape = [m for _, m in reversed(axes)]
    v = torch.complex(torch.randn(shape, generator=gen, dtype=torch.float64, device="cuda"),
                      torch.randn(shape, generator=gen, dtype=torch.float64, device="cuda")) * _inside(shape)
    return v / torch.linalg.vector_norm(v)


def _source(c, axes, gen):
    """A localised source: random values in the middle of the domain, or one node's (constant k)."""
    shape = [m for _, m in reversed(axes)]
    if c["field"] == "constant":
        f = torch.zeros(shape, dtype=torch.complex128, device="cuda")
        at = torch.randint(-(1 << 20), 1 << 20, (len(shape),), generator=gen, device="cuda").tolist()
        f[tuple(m // 2 + int(0.25 * m * a / (1 << 20)) for m, a in zip(shape, at))] = 1.0
        return f
    near = 1.0
    for x, (w, _) in zip(_coords(axes), axes):
        near = near * (x.abs() < 0.5 * w)
    return _random(axes, gen) * near


def _bump(axes, gen):
    """A Gaussian source (width 0.05) around a point in the middle of the domain."""
    shape = [m for _, m in reversed(axes)]
    at = (torch.rand(len(axes), generator=gen, dtype=torch.float64, device="cuda") - 0.5).tolist()
    r2 = sum((x - a * w) ** 2 for x, a, (w, _) in zip(_coords(axes), at, axes))
    return (torch.exp(-r2 / 0.005).expand(shape) * _inside(shape)).to(torch.complex128)


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _energy(gen):
    return 0.5 + 3.5 * float(torch.rand(1, generator=gen, dtype=torch.float64, device="cuda"))


def _params(c):
    return helm.MGParams(kind=c["pc"], theta_a=math.pi / 14 if c["field"] == "constant" else workloads.WELL_THETA_A,
                         nu1=c["nu"], nu2=c["nu"], omega=c["omega"], smoother=c["smoother"], gamma_f=1,
                         gamma_c=c["gamma_c"], coarsest_n=c["coarsest_n"], prec=c["prec"], gs=c["gs"])


def _dtype(c):
    return torch.complex64 if c["prec"] == "c64" else torch.complex128


def _inputs(c, seed):
    """Everything that comes from the seed: the fields and the vectors."""
    gen = _gen(seed)
    if c["op"] == "batch":
        sizes = [129, 257, 513, 1025]
        out = []
        for i in range(c["count"]):  # every size in turn, the largest first
            n = sizes[3 - i % 4]
            one = dict(c, nx=n, ny=n)
            axes = _axes(one)
            out.append((one, axes, _k2(one, axes, _energy(gen)), _bump(axes, gen)))
        return out
    axes = _axes(c)
    k2 = _k2(c, axes, _energy(gen))
    if c["op"] == "apply":
        return axes, k2, _random(axes, gen).to(_dtype(c))
    if c["op"] == "precondition":
        return axes, k2, _random(axes, gen)
    if c["op"] == "solve":
        return axes, k2, _source(c, axes, gen)
    # backward: the forward solution's place is taken by a field of unit size, the incoming gradient
    # is that of a loss seen through a Gaussian probe
    return axes, k2, _bump(axes, gen), _random(axes, gen) * math.sqrt(k2.numel())


def prepare(case, seed):
    c = dict(_BASE)
    c.update(case)
    if c["op"] == "batch":
        problems = _inputs(c, seed)
        batch = helm.helm_create_batch([dict(dim=2, n=one["nx"], k2=k2, theta=THETA) for one, _, k2, _ in problems],
                                       mg=_params(c))
        rhs = [f for _, _, _, f in problems]
        return {"case": c, "batch": batch, "rhs": rhs, "x": [torch.zeros_like(f) for f in rhs]}
    axes, k2, *vectors = _inputs(c, seed)
    widths = [w for w, _ in axes]
    h = helm.helm_create(c["dim"], [m for _, m in axes], k2, theta=THETA, lo=[-w for w in widths], hi=widths,
                         r0_lo=[-LAYER * w for w in widths], r0_hi=[LAYER * w for w in widths], mg=_params(c))
    if c["tuned"]:
        helm.helm_autotune(h, c["prec"])
    s = {"case": c, "handle": h, "vectors": vectors}
    if c["op"] == "apply":
        s["y"] = torch.zeros_like(vectors[0])
    elif c["op"] == "solve":
        s["x"] = torch.zeros_like(vectors[0])
    elif c["op"] == "backward":
        s["grad_k2"] = torch.zeros_like(k2)
        s["grad_f"] = torch.zeros_like(vectors[0])
    return s


def run(state):
    c = state["case"]
    if c["op"] == "batch":
        for x in state["x"]:
            x.zero_()
        helm.helm_solve_batch(state["batch"], state["rhs"], state["x"], tol=c["tol"], restart=c["restart"], maxit=2000)
        return state["x"]
    h = state["handle"]
    v = state["vectors"]
    if c["op"] == "apply":
        return helm.helm_apply(h, v[0], state["y"])
    if c["op"] == "precondition":
        return helm.mg_precondition(h, v[0], _dtype(c))
    if c["op"] == "solve":
        state["x"].zero_()
        x, _ = helm.krylov_solve(h, v[0], state["x"], tol=c["tol"], restart=c["restart"] or 30, maxit=2000,
                                 method=c["method"])
        return x
    helm.helm_backward(h, v[0], v[1], state["grad_k2"], state["grad_f"], tol=c["tol"], restart=c["restart"], maxit=2000)
    return {"grad_k2": state["grad_k2"], "grad_f": state["grad_f"]}


# ---------------------------------------------------------------------------------- work
def _visits(c):
    """Fine-grid equivalents of one cycle: level l has 2^-dim l of the nodes and is visited
    once (V) or, with gamma_c > 1, as often as the F cycle's recursion does."""
    total, l = 0.0, 0
    n = max(c["nx"], c["ny"], c["nz"])
    while n > c["coarsest_n"]:
        total += (1 + (c["gamma_c"] - 1) * l) / 2.0 ** (c["dim"] * l)
        n = (n + 1) // 2
        l += 1
    return total


def _one(c):
    nodes = c["nx"] * c["ny"] * c["nz"]
    stencil = 8.0 * (2 * c["dim"] + 1) + 2.0       # flops of one operator application at a node
    real = 4 if c["prec"] == "c64" else 8
    if c["op"] == "apply":
        return nodes * (5.0 * real), nodes * stencil
    cycle = (2 * c["nu"] * (stencil + 10.0) + stencil) * _visits(c)
    if c["op"] == "precondition":
        return nodes * (16.0 + 2 * real + real), nodes * cycle
    # A solve reads f and k^2 and writes x; its flops are those of the iterations that such a
    # problem takes (about 20 in 3D and 75 on a well grid of 1025 nodes a side, two cycles each in
    # Bi-CGSTAB), each a cycle, an application of A and a Gram-Schmidt step against half a basis.
    cells = max(c["nx"], c["ny"])
    its = 30.0 if c["dim"] == 3 else 30.0 + 60.0 * cells / 1025.0
    if c["method"] == "bicgstab":
        step = 2 * (cycle + stencil) + 80.0
    else:
        step = cycle + stencil + 16.0 * c["restart"] / 2
    extra = 56.0 if c["op"] == "backward" else 40.0  # bytes a node: in and out
    return nodes * extra, nodes * its * step


def work(case):
    c = dict(_BASE)
    c.update(case)
    if c["op"] == "batch":
        sides = [[1025, 513, 257, 129][i % 4] for i in range(c["count"])]
        parts = [_one(dict(c, op="solve", nx=n, ny=n)) for n in sides]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    b, f = _one(c)
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------------- exact
# The same results from plain torch in 64 bits: the finite differences of the stretched grid, the
# cycle's components as whole-array expressions, and for solves a flexible GMRES run far below the
# cases' tolerances.
class _Exact:
    def __init__(self, c, axes, k2):
        self.c, self.dim = c, c["dim"]
        self.axes = axes
        z = []
        for w, m in axes:
            x = torch.linspace(-w, w, m, dtype=torch.float64, device="cuda")
            rot = complex(math.cos(THETA), math.sin(THETA))
            r0 = LAYER * w
            z.append(torch.where(x.abs() > r0, torch.sign(x) * r0 + (x - torch.sign(x) * r0) * rot, x.to(torch.complex128)))
        self.z = z
        self.A = self._operator(z, k2, 0.0, -1.0)
        theta_a = math.pi / 14 if c["field"] == "constant" else workloads.WELL_THETA_A
        shift, bk = (theta_a, -1.0) if c["pc"] == "csg" else (0.0, complex(-1.0, -0.5))
        self.levels = []
        while True:
            self.levels.append(self._operator(z, k2, shift, bk))
            n = [len(a) for a in z]
            if max(n) <= c["coarsest_n"] or any((m - 1) % 2 or (m + 1) // 2 < 3 for m in n):
                break
            z = [a[::2].clone() for a in z]
            k2 = k2[tuple(slice(None, None, 2) for _ in n)].contiguous()
        top = self.levels[-1]
        shape = [m - 2 for m in top["shape"]]
        nu = math.prod(shape)
        cols = []
        for i in range(nu):
            e = torch.zeros(nu, dtype=torch.complex128, device="cuda")
            e[i] = 1.0
            cols.append(self._inner(self.apply(top, self._pad(e.reshape(shape)))).reshape(-1))
        self.dense = torch.linalg.inv(torch.stack(cols, 1))

    def _operator(self, z, k2, shift, bk):
        rot = complex(math.cos(shift), math.sin(shift))
        tri = []
        for a, pos in enumerate(z):
            hm, hp = (pos[1:-1] - pos[:-2]) * rot, (pos[2:] - pos[1:-1]) * rot
            west, east = -2.0 / ((hm + hp) * hm), -2.0 / ((hm + hp) * hp)
            shape = [1] * self.dim
            shape[self.dim - 1 - a] = len(hm)
            tri.append((west.reshape(shape), east.reshape(shape)))
        diag = bk * self._inner(k2).to(torch.complex128)
        for west, east in tri:
            diag = diag - (west + east)
        return {"tri": tri, "diag": diag, "shape": list(k2.shape)}

    def _inner(self, x):
        return x[tuple(slice(1, -1) for _ in range(self.dim))]

    def _pad(self, x):
        return torch.nn.functional.pad(torch.view_as_real(x), [0, 0] + [1, 1] * self.dim).view(
            [m + 2 for m in x.shape] + [2]).contiguous().view(torch.complex128).reshape([m + 2 for m in x.shape])

    def _off(self, op, u):
        out = 0.0
        for a, (west, east) in enumerate(op["tri"]):
            lo = [slice(1, -1)] * self.dim
            hi = [slice(1, -1)] * self.dim
            lo[self.dim - 1 - a], hi[self.dim - 1 - a] = slice(0, -2), slice(2, None)
            out = out + west * u[tuple(lo)] + east * u[tuple(hi)]
        return out

    def apply(self, op, u):
        return self._pad(self._off(op, u) + op["diag"] * self._inner(u))

    def _smooth(self, op, b, u):
        for _ in range(self.c["nu"]):
            if self.c["smoother"] == "jacobi":
                r = self._inner(b) - self._off(op, u) - op["diag"] * self._inner(u)
                u = self._pad(self._inner(u) + self.c["omega"] * r / op["diag"])
                continue
            parity = sum(torch.arange(m, device="cuda").reshape([m if d == e else 1 for e in range(self.dim)])
                         for d, m in enumerate(op["shape"])) % 2
            for colour in (0, 1):
                r = self._inner(b) - self._off(op, u) - op["diag"] * self._inner(u)
                new = self._inner(u) + self.c["omega"] * r / op["diag"]
                u = self._pad(torch.where(self._inner(parity) == colour, new, self._inner(u)))
        return u

    def _down(self, r):
        for d in range(self.dim):
            n = r.shape[d]
            mid = r.narrow(d, 1, n - 2)
            full = 0.25 * r.narrow(d, 0, n - 2) + 0.5 * mid + 0.25 * r.narrow(d, 2, n - 2)
            keep = full.index_select(d, torch.arange(1, n - 2, 2, device="cuda"))
            pad = torch.zeros_like(keep.narrow(d, 0, 1))
            r = torch.cat([pad, keep, pad], d)
        return r

    def _up(self, e, shape):
        for d in range(self.dim):
            n = e.shape[d]
            out = torch.zeros([2 * n - 1 if i == d else m for i, m in enumerate(e.shape)], dtype=e.dtype, device="cuda")
            out.index_copy_(d, torch.arange(0, 2 * n - 1, 2, device="cuda"), e)
            out.index_copy_(d, torch.arange(1, 2 * n - 1, 2, device="cuda"), 0.5 * (e.narrow(d, 0, n - 1) + e.narrow(d, 1, n - 1)))
            e = out
        return self._pad(self._inner(e))

    def cycle(self, b, u=None, l=0, gf=1, gc=None):
        gc = self.c["gamma_c"] if gc is None else gc
        op = self.levels[l]
        if l == len(self.levels) - 1:
            inner = self._inner(b)
            return self._pad((self.dense @ inner.reshape(-1)).reshape(inner.shape))
        u = self._smooth(op, b, torch.zeros_like(b) if u is None else u)
        rc = self._down(self._pad(self._inner(b - self.apply(op, u))))
        if l + 1 == len(self.levels) - 1:
            e = self.cycle(rc, None, l + 1)
        else:
            e = self.cycle(rc, None, l + 1, gf, gc)
            for _ in range(gc - 1):
                e = self.cycle(rc, e, l + 1, gc, gf)
        return self._smooth(op, b, u + self._up(e, op["shape"]))

    def solve(self, f, tol=1e-13, restart=40, cycles=12):
        x = torch.zeros_like(f)
        norm = float(torch.linalg.vector_norm(f))
        best, best_rel = x, 1.0
        for _ in range(cycles):
            r = f - self.apply(self.A, x)
            beta = float(torch.linalg.vector_norm(r))
            if beta >= 0.5 * best_rel * norm and best_rel < 1e-11:
                break
            if beta / norm < best_rel:
                best, best_rel = x.clone(), beta / norm
            if beta <= tol * norm:
                break
            V = torch.zeros([restart + 1, f.numel()], dtype=f.dtype, device="cuda")
            Z = torch.zeros([restart, f.numel()], dtype=f.dtype, device="cuda")
            H = torch.zeros([restart + 1, restart], dtype=f.dtype, device="cuda")
            V[0] = r.reshape(-1) / beta
            for j in range(restart):
                Z[j] = self.cycle(V[j].reshape(f.shape)).reshape(-1)
                w = self.apply(self.A, Z[j].reshape(f.shape)).reshape(-1)
                for _ in range(2):
                    h = V[: j + 1].conj() @ w
                    w = w - h @ V[: j + 1]
                    H[: j + 1, j] += h
                H[j + 1, j] = torch.linalg.vector_norm(w)
                V[j + 1] = w / H[j + 1, j]
            e1 = torch.zeros([restart + 1, 1], dtype=f.dtype, device="cuda")
            e1[0] = beta
            y = torch.linalg.lstsq(H.cpu(), e1.cpu()).solution.to("cuda").reshape(-1)
            x = x + (y @ Z).reshape(f.shape)
            del V, Z
        return best

    def weights(self):
        """Dual volumes: the operator is complex symmetric once its rows are weighted by them."""
        out = 1.0
        for a, pos in enumerate(self.z):
            w = torch.ones_like(pos)
            w[1:-1] = 0.5 * (pos[2:] - pos[:-2])
            shape = [1] * self.dim
            shape[self.dim - 1 - a] = len(w)
            out = out * w.reshape(shape)
        return out


def exact(case, seed):
    c = dict(_BASE)
    c.update(case)
    if c["op"] == "batch":
        return [_Exact(one, axes, k2).solve(f) if one["nx"] <= 257 else None for one, axes, k2, f in _inputs(c, seed)]
    axes, k2, *v = _inputs(c, seed)
    E = _Exact(c, axes, k2)
    if c["op"] == "apply":
        return E.apply(E.A, v[0].to(torch.complex128))
    if c["op"] == "precondition":
        return E.cycle(v[0])
    if c["op"] == "solve":
        return E.solve(v[0])
    w = E.weights()
    inner = _inside(list(k2.shape))
    lam = w * E.solve(v[0].conj() / w * inner)
    return {"grad_k2": (lam * v[1]).real * inner, "grad_f": lam.conj().resolve_conj()}
