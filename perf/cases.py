"""The work that a user of this library has it do, through its public calls, as cases to time.

Four kinds of call, each over the range of sizes the repository's own configurations, tests
and benchmark use (2D grids of 32^2 to 1024^2 cells, 3D grids of 32^3 to 256^3):

  apply   the operator on a vector (residual checks, a caller's own Krylov method)
  post    the gradient and the unprescribed boundary quantity of a solution
  setup   the set-up re-run in place, the control points read back, new data, one operator
          application (a step of a time loop with a moving body or a new level set)
  solve   new data and the solve, from device buffers ("solve"), from host buffers ("host"),
          with the set-up re-run first ("step"), or for many problems at once ("batch")

The data come from polynomials of the scheme's degree, different ones on the two sides of an
interface.  The discretisation reproduces them exactly, so that the operator, the gradient,
the boundary quantity and the solution are known in closed form (``exact``).
"""
import math

import numpy as np
import torch

import paper_2503_22455_gb300 as iim

MG = {"fp32": iim.MG_FP32, "fp64": iim.MG_FP64, "bf16r": iim.MG_FP32_BF16R}
CYCLE = {"v": iim.CYCLE_V, "w": iim.CYCLE_W}
KRYLOV = {"fgmres": iim.KRYLOV_FGMRES, "left": iim.KRYLOV_GMRES_LEFT}


def _case(name, call, dim, n, order, bc, geom, side, mg="fp32", cycle="v", krylov="fgmres", count=1):
    c = {"call": call, "dim": dim, "n": n, "order": order, "bc": bc, "geom": geom, "side": side, "mg": mg,
         "cycle": cycle, "krylov": krylov, "count": count}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest problem of the repository (Laplace in a circle): one operator call is launches
        _case("apply circle 64", "apply", 2, 64, 4, "dirichlet", "circle", "inside"),
        # the benchmark's two-phase star, sixth order: the 2D operator at full size
        _case("apply star 1024", "apply", 2, 1024, 6, "interface", "star", "outside"),
        # the largest 3D configuration: exterior of an ellipsoid with Neumann data
        _case("apply ellipsoid 256", "apply", 3, 256, 4, "neumann", "ellipsoid", "outside"),
        # what a user does with a solution (forces, fluxes): a size that is no power of two
        _case("post star 480", "post", 2, 480, 6, "neumann", "star", "outside"),
        # a moving body: every step re-runs the set-up (a ragged size of the serving mix)
        _case("setup star 736", "setup", 2, 736, 6, "neumann", "star", "outside"),
        # the largest 3D request of the serving mix: its set-up
        _case("setup ellipsoid 192", "setup", 3, 192, 4, "dirichlet", "ellipsoid", "inside"),
        # one small solve: latency
        _case("solve circle 64", "solve", 2, 64, 4, "dirichlet", "circle", "inside"),
        # the benchmark's headline: set-up, data and solve of one two-phase problem
        _case("step star 1024", "step", 2, 1024, 6, "interface", "star", "outside"),
        # an ordinary ragged size from host buffers with the options of the paper's preconditioner study
        _case("host ellipse 416 fp64 w", "host", 2, 416, 4, "neumann", "ellipse", "outside", "fp64", "w", "left"),
        # the paper's 3D verification body, pure Neumann (the augmented system)
        _case("solve perturbed sphere 96", "solve", 3, 96, 4, "neumann", "perturbed_sphere", "inside"),
        # the benchmark's 3D configuration, set-up included: the largest single problem
        _case("step ellipsoid 256", "step", 3, 256, 4, "neumann", "ellipsoid", "outside"),
        # the mixed 2D batch: ellipses and stars, 64^2 to 512^2, both orders, both conditions
        _case("batch mixed 24", "batch", 2, 512, 6, "mixed", "mixed", "mixed", count=24),
    ]


def _coarsest(n):
    """Cells per axis of the coarsest multigrid level of a 2D grid."""
    while n % 2 == 0 and n // 2 >= 8:
        n //= 2
    return n


def _size(rng, dim, lo, hi):
    """A size between lo and hi, even over its logarithm: multiples of 32 as the batch and the
    serving mix draw them, finer steps for small grids; sizes whose coarsest level would hold
    more unknowns than that of any listed case are left out."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    if dim == 2:
        step = 4 if v < 128 else (8 if v < 250 else 32)
        fit = [m for m in range(step, hi + 1, step) if m >= lo and _coarsest(m) <= 23]
    else:
        fit = [m for m in (32, 40, 48, 56, 64, 80, 96, 112, 128, 160, 192) if lo <= m <= hi]
    return min(fit, key=lambda m: abs(math.log(m / v)))


def draw(rng):
    call = rng.choice(["apply", "apply", "post", "setup", "setup", "solve", "solve", "step", "host", "batch"])
    if call == "batch":
        n = _size(rng, 2, 64, 512)
        return _case(None, call, 2, n, 6, "mixed", "mixed", "mixed", rng.choice(["fp32", "bf16r"]), count=rng.randint(2, 24))
    dim = 3 if rng.random() < 0.4 else 2
    order = 4 if dim == 3 else rng.choice([4, 6])
    bc = rng.choice(["dirichlet", "neumann", "interface"] if call != "post" else ["dirichlet", "neumann"])
    if bc == "interface":
        side = "outside"
    else:
        side = rng.choice(["inside", "outside"])
    if dim == 3:
        geom = rng.choice(["sphere", "ellipsoid", "levelset"] + (["perturbed_sphere"] if side == "inside" else []))
    else:
        geom = rng.choice(["circle", "ellipse", "star", "levelset"])
    lo = (64 if order == 6 else 40) if side == "outside" else (48 if order == 6 else 32)
    if bc == "interface" or geom in ("star", "perturbed_sphere"):
        lo = max(lo, 64 if dim == 2 else 48)
    n = _size(rng, dim, lo, 1024 if dim == 2 else (128 if bc == "interface" else 192))
    mg, cycle, krylov = "fp32", "v", "fgmres"
    if call in ("solve", "step", "host") and rng.random() < 0.4:
        mg = rng.choice(["fp64", "bf16r", "fp32"])
        cycle = rng.choice(["v", "w"])
        krylov = rng.choice(["fgmres", "left"])
    return _case(None, call, dim, n, order, bc, geom, side, mg, cycle, krylov)


# ----------------------------------------------------------------------------- problem statements
class _Statement:
    """Geometry, conditions and the piecewise polynomial solution of one problem."""

    def __init__(self, dim, n, order, bc, geom, side, shape_rng, data_rng):
        rng = shape_rng
        self.dim, self.n, self.order, self.bc, self.geom = dim, n, order, bc, geom
        self.inside = side == "inside"                       # Omega+ is the inside of the body
        self.box = not self.inside
        c = list(rng.uniform(-0.03, 0.03, size=dim))
        e = 0.1 if n < 64 else 0.2
        if geom == "circle":
            self.params = c + [0.42 + 0.08 * rng.random()]
        elif geom == "sphere":
            self.params = c + [0.42 + 0.08 * rng.random()]
        elif geom in ("ellipse", "levelset") and dim == 2:
            self.params = c + list(0.45 * rng.uniform(1 - e, 1 + e, size=2)) + [rng.uniform(0, math.pi)]
        elif geom == "star":
            m, r0 = int(rng.integers(5, 8)), 0.48
            amp = min(0.1, 0.6 * r0 * r0 * (0.1 * n - 1 / r0) / (m * m))
            self.params = c + [r0, amp, float(m), rng.uniform(0, 2 * math.pi)]
        elif geom == "perturbed_sphere":
            self.params = c + [0.7, 0.1 if n >= 64 else 0.03]
        elif n >= 128:
            self.params = c + [0.6, 0.45, 0.35]
        else:
            self.params = c + list(0.45 * rng.uniform(1 - e, 1 + e, size=3))
        self.plus = self._polynomial(data_rng)
        self.minus = self._polynomial(data_rng) if bc == "interface" else None

    def _polynomial(self, rng):
        """Coefficients of a random polynomial of total degree <= order."""
        q = self.order
        c = rng.standard_normal((q + 1,) * self.dim)
        deg = sum(np.meshgrid(*[np.arange(q + 1)] * self.dim, indexing="ij"))
        return np.where(deg <= q, c, 0.0)

    def phi(self, x):
        """The level set (positive in Omega+) at the points with the coordinates x."""
        p = self.params
        d = [x[k] - p[k] for k in range(self.dim)]
        if self.geom in ("circle", "sphere"):
            g = torch.sqrt(sum(v * v for v in d)) - p[self.dim]
        elif self.geom == "star":
            r, th = torch.hypot(d[0], d[1]), torch.atan2(d[1], d[0])
            g = r - (p[2] + p[3] * torch.sin(p[4] * th + p[5]))
        elif self.geom == "perturbed_sphere":
            r = torch.sqrt(sum(v * v for v in d))
            g = r - p[3] - p[4] * (1.5 * math.sqrt(3.0)) * ((d[0] * d[0] - d[1] * d[1]) * d[2]) / r ** 3
        elif self.dim == 2:
            cs, sn = math.cos(p[4]), math.sin(p[4])
            g = ((cs * d[0] + sn * d[1]) / p[2]) ** 2 + ((cs * d[1] - sn * d[0]) / p[3]) ** 2 - 1.0
        else:
            g = sum((d[k] / p[3 + k]) ** 2 for k in range(3)) - 1.0
        return -g if self.inside else g

    def nodes(self, device):
        return -1.0 + (torch.arange(self.n, dtype=torch.float64, device=device) + 0.5) * (2.0 / self.n)

    def grid(self, device):
        """The nodes' coordinates, one tensor per axis over (n,) * dim with axis 0 fastest."""
        g = torch.meshgrid(*[self.nodes(device)] * self.dim, indexing="ij")
        return [v for v in reversed(g)]

    def phase(self, device):
        return self.phi(self.grid(device)) >= 0

    def on_grid(self, coef, device):
        """The polynomial at every node, flat with axis 0 fastest."""
        x = self.nodes(device)
        t = torch.as_tensor(coef, dtype=torch.float64, device=device)
        for _ in range(self.dim):                              # the first axis left is contracted
            v = torch.stack([x ** a for a in range(t.shape[0])], dim=0)
            t = torch.tensordot(t, v, dims=([0], [0]))         # its nodes become the last axis
        return t.permute(*reversed(range(self.dim))).reshape(-1)

    def at(self, coef, pts):
        """The polynomial at points of shape (K, dim)."""
        t = torch.as_tensor(coef, dtype=torch.float64, device=pts.device)
        out = torch.zeros(pts.shape[0], dtype=torch.float64, device=pts.device)
        for e in np.argwhere(coef != 0):
            v = t[tuple(e)]
            for k in range(self.dim):
                v = v * pts[:, k] ** int(e[k])
            out = out + v
        return out

    @staticmethod
    def derivative(coef, axis):
        c = np.moveaxis(coef, axis, 0)
        d = np.zeros_like(c)
        for a in range(1, c.shape[0]):
            d[a - 1] = a * c[a]
        return np.moveaxis(d, 0, axis)

    def laplacian(self, coef):
        return sum(self.derivative(self.derivative(coef, k), k) for k in range(self.dim))

    def piecewise(self, plus, minus, phase, device):
        v = self.on_grid(plus, device)
        other = torch.zeros_like(v) if minus is None else self.on_grid(minus, device)
        return torch.where(phase.reshape(-1), v, other)

    def solution(self, phase, device):
        return self.piecewise(self.plus, self.minus, phase, device)

    def source(self, phase, device):
        lm = None if self.minus is None else self.laplacian(self.minus)
        return self.piecewise(self.laplacian(self.plus), lm, phase, device)

    def boundary(self, xc, nc):
        """(g, j0, j1) at the control points xc with the normals nc."""
        flux = [sum(self.at(self.derivative(c, k), xc) * nc[:, k] for k in range(self.dim)).contiguous()
                for c in (self.plus, self.minus) if c is not None]
        if self.bc == "dirichlet":
            return self.at(self.plus, xc), None, None
        if self.bc == "neumann":
            return flux[0], None, None
        return None, (self.at(self.plus, xc) - self.at(self.minus, xc)).contiguous(), (flux[0] - flux[1]).contiguous()

    def crossings(self, device):
        """Control points and normals (out of Omega+) of the cut grid edges, axis by axis, in the
        order of the edges' lower nodes: bisection of the level set, its gradient."""
        x, phase, h = self.nodes(device), self.phase(device), 2.0 / self.n
        found = []
        for ax in range(self.dim):
            a = self.dim - 1 - ax                               # axis 0 is the last of the tensor
            m = self.n - 1
            cut = (phase.narrow(a, 0, m) != phase.narrow(a, 1, m)).nonzero()
            lo = torch.stack([x[cut[:, self.dim - 1 - k]] for k in range(self.dim)], dim=1)
            left, right = torch.zeros(len(lo), dtype=torch.float64, device=device), torch.ones(len(lo), dtype=torch.float64, device=device)

            def point(t):
                p = lo.clone()
                p[:, ax] += t * h
                return p

            s0 = self.phi(list(point(left).T)) >= 0
            for _ in range(56):
                mid = 0.5 * (left + right)
                same = (self.phi(list(point(mid).T)) >= 0) == s0
                left, right = torch.where(same, mid, left), torch.where(same, right, mid)
            found.append(point(0.5 * (left + right)))
        xc = torch.cat(found).requires_grad_(True)
        g = torch.autograd.grad(self.phi([xc[:, k] for k in range(self.dim)]).sum(), xc)[0]
        return xc.detach(), -g / g.norm(dim=1, keepdim=True)

    def problem(self, opts):
        kind, phi, plus_inside = iim.GEOM.get(self.geom), None, self.inside
        params = self.params
        if self.geom == "levelset":
            kind, params, plus_inside = iim.GEOM["levelset_grid"], [], False
            phi = self.phi(self.grid("cuda")).reshape(-1).contiguous()
        d = iim.make_desc(self.dim, self.n, kind, params, plus_inside, iim.BC[self.bc], int(self.box),
                          order=self.order, phi=phi)
        return iim.Problem(d, iim.default_options(**opts))

    def data(self, P):
        """The problem's data on the device: f, g, j0, j1, box values."""
        xc, nc = P.control_points()
        g, j0, j1 = self.boundary(xc, nc)
        f = self.source(P.phase().bool(), "cuda")
        box = self.at(self.plus, P.box_points()) if self.box else None
        return f, g, j0, j1, box


def _statements(case, seed):
    """The bodies follow from the case alone (their control points size the outputs), the data from the seed."""
    mix = np.random.default_rng([case["n"], case["dim"], case["order"], case["count"]])
    rng = np.random.default_rng([int(seed), case["n"], case["dim"], case["order"]])
    if case["call"] != "batch":
        return [_Statement(case["dim"], case["n"], case["order"], case["bc"], case["geom"], case["side"], mix, rng)]
    sizes = np.arange(64, max(64, case["n"]) + 1, 32)
    out = []
    for _ in range(case["count"]):
        n, order, inside = int(mix.choice(sizes)), int(mix.choice([4, 6])), mix.random() < 0.5
        geom = "ellipse" if mix.random() < 0.5 else "star"
        out.append(_Statement(2, n, order, "dirichlet" if inside else "neumann", geom, "inside" if inside else "outside", mix, rng))
    return out


# ----------------------------------------------------------------------------- the cases' passes
def prepare(case, seed):
    opts = {"mg_precision": MG[case["mg"]], "cycle": CYCLE[case["cycle"]], "krylov": KRYLOV[case["krylov"]]}
    problems, data, u = [], [], []
    for s in _statements(case, seed):
        P = s.problem(opts)
        d = s.data(P)
        if case["call"] in ("apply", "post", "setup"):
            P.set_data(*d)
            u.append(s.solution(P.phase().bool(), "cuda"))
        if case["call"] == "host":
            d = tuple(None if v is None else v.cpu().pin_memory() for v in d)
        problems.append(P)
        data.append(d)
    x = torch.empty(problems[0].N, dtype=torch.float64).pin_memory() if case["call"] == "host" else None
    return {"call": case["call"], "problems": problems, "data": data, "u": u, "x": x}


def run(state):
    call, P, data = state["call"], state["problems"][0], state["data"][0]
    if call == "apply":
        return P.apply(state["u"][0], include_data=True)
    if call == "post":
        return {"gradient": P.gradient(state["u"][0]), "boundary": P.boundary_values(state["u"][0])}
    if call == "setup":
        P.setup()
        xc, nc = P.control_points()
        P.set_data(*data)
        return {"points": xc, "normals": nc, "w": P.apply(state["u"][0], include_data=True)}
    if call == "host":
        return P.solve_host(*data, x=state["x"])[0]
    if call == "batch":
        for Q, d in zip(state["problems"], state["data"]):
            Q.set_data(*d)
        xs = [torch.zeros(Q.N, dtype=torch.float64, device="cuda") for Q in state["problems"]]
        iim.batch_solve(state["problems"], xs)
        return xs
    if call == "step":
        P.setup()
    P.set_data(*data)
    return P.solve()[0]


# typical FGMRES iterations to 1e-10 by condition (the work of a solve is counted with them)
ITERATIONS = {"dirichlet": 20, "neumann": 28, "interface": 34}


def work(case):
    nbytes = flops = 0.0
    for s in _statements(case, 0):
        N, w = float(s.n) ** s.dim, s.order // 2
        unknowns = N if s.bc == "interface" else N * (0.25 if s.inside and s.dim == 2 else 0.12 if s.inside else 0.8)
        # cut edges of a body of radius about 0.45, fits of the scheme's degree
        K = 4.0 * s.n * 0.45 * 1.0 if s.dim == 2 else 6.0 * math.pi * (0.225 * s.n) ** 2
        fits = K * (2 if s.bc == "interface" else 1)
        M = math.comb(s.order + s.dim, s.dim)
        R = 1.5 * M if s.dim == 2 else 2.5 * M
        app_b = 17.0 * N + fits * (w + 1) * R * 8
        app_f = (2.0 * s.dim * w + 2.0 * w + 2) * unknowns + 2.0 * fits * (w + 1) * R
        set_b = 17.0 * N + fits * (w + 1) * R * 8
        set_f = fits * 2.0 * R * M * M
        if case["call"] == "apply":
            nbytes, flops = nbytes + app_b, flops + app_f
        elif case["call"] == "post":
            nbytes, flops = nbytes + app_b + 8.0 * (s.dim - 1) * N, flops + app_f
        elif case["call"] == "setup":
            nbytes, flops = nbytes + app_b + set_b, flops + app_f + set_f
        else:
            it = ITERATIONS[s.bc]
            cyc = 1.0 / (1.0 - 0.5 ** s.dim)
            gs = 5.5                                           # basis vectors in use on average
            it_b = app_b + 36.0 * cyc * N + 2 * (gs + 1) * 8.0 * N
            it_f = app_f + 60.0 * cyc * unknowns + 4.0 * (gs + 1) * unknowns
            nbytes, flops = nbytes + it * it_b + 17.0 * N, flops + it * it_f
            if case["call"] == "step":
                nbytes, flops = nbytes + set_b, flops + set_f
    return {"bytes": nbytes, "flops": flops}


def exact(case, seed):
    out = []
    for s in _statements(case, seed):
        phase = s.phase("cuda")
        if case["call"] == "apply":
            return s.source(phase, "cuda")
        if case["call"] == "post":
            xc, nc = s.crossings("cuda")
            grad = torch.stack([s.piecewise(s.derivative(s.plus, k), None, phase, "cuda") for k in range(s.dim)])
            if s.bc == "neumann":
                return {"gradient": grad, "boundary": s.at(s.plus, xc)}
            return {"gradient": grad, "boundary": sum(s.at(s.derivative(s.plus, k), xc) * nc[:, k] for k in range(s.dim))}
        if case["call"] == "setup":
            xc, nc = s.crossings("cuda")
            return {"points": xc, "normals": nc, "w": s.source(phase, "cuda")}
        u = s.solution(phase, "cuda")
        if s.bc == "neumann" and not s.box:                    # pure Neumann: the mean-free solution
            u = torch.where(phase.reshape(-1), u - u.sum() / phase.sum(), torch.zeros_like(u))
        out.append(u)
    return out if case["call"] == "batch" else out[0]
