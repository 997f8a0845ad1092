"""Timed workloads of the MIUGKS solver: what a user's program has it do.

A pass of a flow case is the program's whole call: the initial fields go in from
host arrays, the solver iterates, and the macroscopic fields (and the wall
quantities of the flows that are run for them) come back to the host.  The
adjoint cases call the differentiation form through its host-array entry points.
The flows are the configurations of the paper's Sec. 4 as `workloads` builds
them, from a few hundred cells to the full square cylinder, in both precisions,
on the legacy default stream and on streams of their own, with odd and ragged
meshes and velocity grids.

`exact` gives the same results in 64 bits with plain torch operations, from the
equations the header of the library cites.
"""
import math

import numpy as np
import torch

from paper_1704_03151_gb300 import miugks, workloads

WALL, SYMMETRY, FARFIELD, OUTFLOW = 0, 1, 2, 3


# ---------------------------------------------------------------- cases
def _flow(name, flow, nx, ny, nu, nv, levels, precision, iters, kn, stream=True, **more):
    c = {"name": name, "call": "flow", "flow": flow, "nx": nx, "ny": ny, "nu": nu, "nv": nv, "levels": levels,
         "precision": precision, "iters": iters, "kn": kn, "stream": stream, "cycle": "V", "count": 1}
    c.update(more)
    return c


def listed():
    return [
        # the smallest calls: a coarse cavity of a parameter study on the default stream, where launches count
        _flow("cavity16_v12_mixed", "cavity", 16, 16, 12, 12, 1, "mixed", 4, 0.5, stream=False),
        # the paper's single-grid cavity (Sec. 4.1), from rest to a residual of 1e-6 or 300 iterations
        _flow("cavity24_v20_fp64_run", "cavity", 24, 24, 20, 20, 1, "fp64", 300, 1.0, stream=False, call="run"),
        # Couette / Fourier channel with symmetry sides: a ragged mesh, odd unequal velocity grids, F cycle
        _flow("channel28x44_v25x21_mixed", "channel", 28, 44, 25, 21, 3, "mixed", 4, 0.3, cycle="F"),
        # the cavity of the multigrid study (Sec. 4.1, 3 levels), both forms; the mixed one is the ordinary call
        _flow("cavity64_v32_mixed", "cavity", 64, 64, 32, 32, 3, "mixed", 5, 1.0),
        _flow("cavity64_v32_fp64", "cavity", 64, 64, 32, 32, 3, "fp64", 2, 0.075),
        # a parameter sweep: independent cavities at different Kn, each on its own stream, side by side
        _flow("sweep8_cavity96_v40_mixed", "cavity", 96, 96, 40, 40, 4, "mixed", 3, 1.0, count=8),
        # low-speed plate on a stretched mesh (Sec. 4.2): the bulk of a solve in the mixed form, its finish in FP64
        _flow("plate128x96_v48_mixed", "plate", 128, 96, 48, 48, 4, "mixed", 3, 0.1),
        _flow("plate128x96_v48_fp64", "plate", 128, 96, 48, 48, 4, "fp64", 1, 0.1),
        # Ma 5 square cylinder (Sec. 4.3): the full mesh, and the half-size one in FP64; 89 is odd, so rows are unaligned
        _flow("square160x120_v89_mixed", "square", 160, 120, 89, 89, 4, "mixed", 3, 0.1),
        _flow("square80x60_v89_fp64", "square", 80, 60, 89, 89, 3, "fp64", 2, 0.1),
        # backward: one product with the transposed Jacobian, as an outer optimiser's own Krylov solver calls it
        _flow("adjoint_product48_v32", "cavity", 48, 48, 32, 32, 1, "fp64", 1, 1.0, call="product"),
        # backward: the whole gradient d(lid shear) / d(lid speed) at a converged state
        _flow("adjoint_solve32_v20", "cavity", 32, 32, 20, 20, 3, "fp64", 1, 1.0, call="adjoint"),
    ]


def draw(rng):
    while True:
        c = _draw(rng)
        cells = c["count"] * c["iters"] * c["nx"] * c["ny"] * c["nu"] * c["nv"]
        if cells * (1 if c["precision"] == "mixed" else 7) < 4e8:     # no more than the largest listed case
            return c


def _draw(rng):
    def log(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["cavity", "cavity", "cavity", "channel", "plate", "square", "product", "sweep"])
    more = {"precision": rng.choice(["mixed", "fp64"]), "iters": rng.choice([1, 2, 3, 4]), "stream": rng.random() < 0.7,
            "kn": round(10.0 ** rng.uniform(-1.2, 1.0), 4)}
    levels = rng.choice([1, 2, 3, 4])
    if kind in ("plate", "square"):
        levels = min(levels, 3)
    m = 2 ** (levels - 1)
    if kind == "plate":
        q, v = m * max(1, log(2, 32) // m), log(16, 49)
        more["kn"] = round(rng.uniform(0.1, 0.4), 4)
        return _case("plate", 4 * q, m * max(1, log(8, 96) // m), v, v, levels, more)
    if kind == "square":
        h, v = rng.choice([4, 8, 12, 16]), 2 * log(16, 44) + 1        # h: cells along the square's side, a fifth of the mesh's
        more["kn"] = 0.1
        return _case("square", 5 * max(4, h * 4 // 3 // 4 * 4), 5 * h, v, v, levels, more)
    nx, ny = m * max(2, log(8, 128) // m), m * max(2, log(8, 128) // m)
    nu, nv = log(12, 49), log(12, 49)
    if kind == "channel":
        more["cycle"] = rng.choice("VWF")
        return _case("channel", nx, ny, nu, nv, levels, more)
    if kind == "product":
        more.update(precision="fp64", iters=1, call="product")
        return _case("cavity", log(8, 56), log(8, 56), log(12, 33), log(12, 33), 1, more)
    if kind == "sweep":
        more.update(precision="mixed", stream=True, count=rng.choice([2, 3, 4, 6]))
    else:
        more["cycle"] = rng.choice("VVVW")
    return _case("cavity", nx, ny, nu, nv, levels, more)


def _case(flow, nx, ny, nu, nv, levels, more):
    more = dict(more)
    c = _flow("", flow, nx, ny, nu, nv, levels, more.pop("precision"), more.pop("iters"), more.pop("kn"), **more)
    del c["name"]
    return c


# ---------------------------------------------------------------- what a program has in hand
def _unit(seed, q):
    """A number in [0, 1) of the seed."""
    return float(np.random.default_rng([int(seed), q]).random())


def _problems(case, seed):
    """The problem set-ups of a case: `count` dicts as the solver takes them."""
    out = []
    for q in range(case["count"]):
        kn = case["kn"] * (10.0 ** (2.0 * _unit(seed, 10 + q) - 1.0) if case["count"] > 1 else 1.0)
        if case["flow"] == "cavity":
            p = workloads.cavity(nx=case["nx"], ny=case["ny"], nvel=case["nu"], kn=kn, lid=0.1 + 0.2 * _unit(seed, 50 + q),
                                 levels=case["levels"])
        elif case["flow"] == "channel":
            p = workloads.couette(n=case["ny"], nx=case["nx"], nvel=case["nu"], kn=kn, t_bottom=1.0,
                                  t_top=1.2 + 0.3 * _unit(seed, 50), u_top=0.2, levels=case["levels"])
        elif case["flow"] == "plate":
            e = case["nx"] // 4
            p = workloads.flat_plate(kn=kn, ma=0.15 + 0.1 * _unit(seed, 50), nvel=case["nu"], levels=case["levels"],
                                     n_up=e, n_plate=2 * e, n_down=e, ny=case["ny"])
        else:
            sx, sy = case["nx"] // 5, case["ny"] // 5
            p = workloads.square_cylinder(kn=kn, nvel=case["nu"], levels=case["levels"], nx_side=2 * sx, nx_sq=sx,
                                          ny_side=2 * sy, ny_sq=sy)
        p["vgrid"] = dict(p["vgrid"], nu=case["nu"], nv=case["nv"])
        out.append(p)
    return out


def _fields(case, p, seed, q):
    """Initial rho, u, v, T per cell: the flow's start, smoothly perturbed by the seed."""
    if case["call"] == "run":
        return [np.full(p["nx"] * p["ny"], float(p["init"][k])) for k in ("rho", "u", "v", "t")]
    f = workloads.initial_fields(p)
    if case["flow"] == "square":
        r = workloads.random_fields(dict(p, init={"rho": 1.0, "u": 0.0, "v": 0.0, "t": 1.0}), seed + q, amp=0.02)
        return [f[0] * r[0], f[1], f[2], f[3] * r[3]]
    return workloads.random_fields(p, seed + 1000 * q, amp=0.05)


class _State:
    pass


def prepare(case, seed):
    st = _State()
    st.case = case
    st.problems = _problems(case, seed)
    st.fields = [_fields(case, p, seed, q) for q, p in enumerate(st.problems)]
    st.solvers = []
    for p in st.problems:
        stream = torch.cuda.Stream() if case["stream"] else None
        s = miugks.Solver(p, precision=case["precision"], stream=stream)
        if case["cycle"] != "V":
            s.set_cycle(case["cycle"])
        st.solvers.append(s)
    s, p = st.solvers[0], st.problems[0]
    if case["call"] == "product":
        # a state away from equilibrium, and a dual vector as a Krylov solver hands it over
        s.init_fields(*st.fields[0])
        s.set_f(_noisy(s, case, seed))
        st.mu = np.random.default_rng([int(seed), 7]).standard_normal((2, s.nc, s.nv))
    elif case["call"] == "adjoint":
        s.init_uniform(1.0, 0.0, 0.0, 1.0)
        s.run(1e-11, 200)
    return st


def _noise(case, seed, n, nv):
    return 1.0 + 0.02 * np.random.default_rng([int(seed), 8]).standard_normal((2, n, nv))


def _noisy(s, case, seed):
    return s.get_f() * _noise(case, seed, s.nc, s.nv)


# ---------------------------------------------------------------- one pass
def _result(case, m, wall):
    """The fields and wall quantities as a program keeps them: in FP32 from the mixed form, whose distribution
    function, and so every moment of it, is an FP32 quantity; in FP64 from the FP64 form."""
    t = np.float32 if case["precision"] == "mixed" else np.float64
    out = {"fields": np.stack([m[k] for k in ("rho", "u", "v", "t", "qx", "qy")]).astype(t)}
    if wall is not None:
        out["wall"] = np.stack(wall).astype(t)
    return out


def run(state):
    case, solvers = state.case, state.solvers
    s = solvers[0]
    if case["call"] == "product":
        return s.adjoint_residual(state.mu)
    if case["call"] == "adjoint":
        g, info = s.adjoint(0, 2, 1, tol=1e-12, max_iter=400)
        return np.array([g, info["J"]])
    if case["call"] == "run":
        p = state.problems[0]["init"]
        s.init_uniform(p["rho"], p["u"], p["v"], p["t"])
        s.run(1e-6, case["iters"])
        return _result(case, s.macro(), s.wall(2))
    for s, f in zip(solvers, state.fields):
        s.init_fields(*f)
    if len(solvers) == 1:
        s.step(case["iters"])
    else:
        for s in solvers:
            s.step_async(case["iters"])
        for s in solvers:
            s.wait()
    return [_result(case, s.macro(), s.wall(0) if case["flow"] in ("plate", "square") else None) for s in solvers]


def work(case):
    """Per iteration, f read and written once; the operations of the scheme per cell and velocity: the flux of two faces,
    the residual, the moments, and per smoothing two sweeps and one renewal of both components, over the levels."""
    size = 4 if case["precision"] == "mixed" else 8
    cv = case["count"] * case["nx"] * case["ny"] * case["nu"] * case["nv"]
    if case["call"] == "product":
        return {"bytes": 3 * 2 * cv * size, "flops": 500 * cv}
    if case["call"] == "adjoint":
        return {"bytes": 60 * 2 * 2 * cv * size, "flops": 60 * 900 * cv}
    smooth = sum((3.0 if l + 1 < case["levels"] else 4.0 if l else 1.0) / 4 ** l for l in range(case["levels"]))
    it = 40 if case["call"] == "run" else case["iters"]
    return {"bytes": it * 2 * 2 * cv * size, "flops": it * cv * (260 + 52 * smooth)}


# ================================================================ the same results in 64 bits, in plain torch
KI = 1.0   # internal degrees of freedom


def exact(case, seed):
    if case["call"] == "adjoint":
        return None
    # an estimate of the time: diagonals swept one by one, and the per-velocity arithmetic
    cv = case["nx"] * case["ny"] * case["nu"] * case["nv"]
    if case["count"] * case["iters"] * cv > 1.2e8 and case["call"] == "flow":
        return None
    out = []
    for q, p in enumerate(_problems(case, seed)):
        x = _Exact(p, case["cycle"], torch.device("cuda" if torch.cuda.is_available() else "cpu"))
        x.start(_fields(case, p, seed, q))
        if case["call"] == "product":
            x.f = x.f * x.tensor(_noise(case, seed, x.lev[0].nc, x.nv))
            mu = x.tensor(np.random.default_rng([int(seed), 7]).standard_normal((2, x.lev[0].nc, x.nv)))
            return x.product(mu).cpu().numpy()
        for _ in range(case["iters"]):
            res = x.iterate()
            if case["call"] == "run" and max(res) < 1e-6:
                break
        wall = x.wall(2) if case["call"] == "run" else x.wall(0) if case["flow"] in ("plate", "square") else None
        r = {"fields": x.fields().cpu().numpy()}
        if wall is not None:
            r["wall"] = wall.cpu().numpy()
        out.append(r)
    return out[0] if case["call"] == "run" else out


class _Level:
    pass


def _prim(W):
    rho = W[..., 0]
    U, V = W[..., 1] / rho, W[..., 2] / rho
    lam = (KI + 2) * rho / (4 * (W[..., 3] - 0.5 * (W[..., 1] * U + W[..., 2] * V)))
    return rho, U, V, lam


def _limited(a, b):
    on = a * b > 0
    one = torch.ones_like(a)
    a, b = torch.where(on, a, one), torch.where(on, b, one)
    return torch.where(on, 2 * a * b / (a + b), torch.zeros_like(a))


def _slope(d, U, V, lam):
    """Coefficients of the equilibrium's slope from the slopes of rho, m, E over rho."""
    c = U * U + V * V + (KI + 2) / (2 * lam)
    R4 = 2 * d[3] - c * d[0]
    R3 = d[2] - V * d[0]
    R2 = d[1] - U * d[0]
    a3 = 4 * lam * lam / (KI + 2) * (R4 - 2 * U * R2 - 2 * V * R3)
    a2 = 2 * lam * R3 - V * a3
    a1 = 2 * lam * R2 - U * a3
    return d[0] - U * a1 - V * a2 - 0.5 * a3 * c, a1, a2, a3


def _time_integrals(dt, tau):
    x = dt / tau
    s = torch.clamp(x, max=1.0)
    S = [torch.zeros_like(x) for _ in range(5)]
    for n in range(27, -1, -1):
        sg = -1.0 if n % 2 else 1.0
        f1, f2 = math.factorial(n + 1), math.factorial(n + 2)
        for m, c in enumerate((-sg / f1 if n else 0.0, sg * n / f2, -sg / f2 if n else 0.0, sg / f1, -sg * (n + 1) / f2)):
            S[m] = S[m] * s + c
    e, E1 = torch.exp(-x), -torch.expm1(-x)
    closed = [dt - tau * E1, -tau * dt * (1 + e) + 2 * tau * tau * E1, 0.5 * dt * dt - tau * dt + tau * tau * E1, tau * E1,
              tau * dt * e - tau * tau * E1]
    scale = [dt, dt * dt, dt * dt, dt, dt * dt]
    return [torch.where(x < 1, S[m] * scale[m], closed[m]) for m in range(5)]


def _euler(W, axis):
    U, V = W[..., 1] / W[..., 0], W[..., 2] / W[..., 0]
    p = 2 / (KI + 2) * (W[..., 3] - 0.5 * (W[..., 1] * U + W[..., 2] * V))
    Ua = V if axis else U
    T = [W[..., 1 + axis], W[..., 1] * Ua, W[..., 2] * Ua, (W[..., 3] + p) * Ua]
    T[1 + axis] = T[1 + axis] + p
    return torch.stack(T, -1)


class _Exact:
    """The outer iteration of the multigrid implicit scheme on one problem."""

    def __init__(self, p, cycle, dev):
        self.p, self.dev, self.cycle = p, dev, cycle
        T = self.tensor
        vg, g = p["vgrid"], p["gas"]
        ax = []
        for n, a, b in ((vg["nu"], vg["umin"], vg["umax"]), (vg["nv"], vg["vmin"], vg["vmax"])):
            h = (b - a) / (n - 1)
            x, w = 0.5 * (a + b) + (np.arange(n) - 0.5 * (n - 1)) * h, np.full(n, h)
            w[0] = w[-1] = 0.5 * h
            ax.append((x, w))
        self.nu, self.nvv, self.nv = vg["nu"], vg["nv"], vg["nu"] * vg["nv"]
        self.u, self.v = T(np.repeat(ax[0][0], self.nvv)), T(np.tile(ax[1][0], self.nu))
        self.w = T(np.outer(ax[0][1], ax[1][1]).ravel())
        self.e = 0.5 * (self.u ** 2 + self.v ** 2)
        k = np.arange(self.nv)
        self.mirror = [torch.as_tensor((self.nu - 1 - k // self.nvv) * self.nvv + k % self.nvv, device=dev),
                       torch.as_tensor(k // self.nvv * self.nvv + self.nvv - 1 - k % self.nvv, device=dev)]
        self.mu = 15 * math.sqrt(math.pi) * g["kn"] / (2 * (5 - 2 * g["omega"]) * (7 - 2 * g["omega"]))
        self.omega, self.pr = g["omega"], g["pr"]
        self.bcs, self.mg = p["bcs"], p["mg"]
        self.C = [(1 / b["t"]) / math.pi * torch.exp(-((self.u - b["u"]) ** 2 + (self.v - b["v"]) ** 2) / b["t"])
                  for b in self.bcs]
        self.lev = [self._level(p["nx"], p["ny"], np.asarray(p["x_nodes"], float), np.asarray(p["y_nodes"], float),
                                np.asarray(p["face_bc_x"]).reshape(p["ny"], p["nx"] + 1),
                                np.asarray(p["face_bc_y"]).reshape(p["ny"] + 1, p["nx"]),
                                np.asarray(p["solid"]).reshape(p["ny"], p["nx"]) > 0 if p.get("solid") is not None
                                else np.zeros((p["ny"], p["nx"]), bool))]
        for _ in range(1, self.mg["levels"]):
            F = self.lev[-1]
            self.lev.append(self._level(F.nx // 2, F.ny // 2, F.xn[::2], F.yn[::2], F.bx[::2, ::2], F.by[::2, ::2],
                                        F.sol[::2, ::2]))
            self._transfer(F, self.lev[-1])
        self.umax = max(abs(vg["umin"]), abs(vg["umax"]))
        self.vmax = max(abs(vg["vmin"]), abs(vg["vmax"]))
        L = self.lev[0]
        self.dtp = self.mg["cfl"] * min(np.minimum(d[1:], d[:-1]).min() / m for d, m in
                                        ((L.hx, self.umax), (L.hy, self.vmax)) if len(d) > 1)
        self.it = 0

    def tensor(self, a):
        return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=self.dev)

    # ------------------------------------------------------------ meshes
    def _level(self, nx, ny, xn, yn, bx, by, sol):
        L = _Level()
        L.nx, L.ny, L.nc, L.xn, L.yn, L.bx, L.by, L.sol = nx, ny, nx * ny, xn, yn, bx, by, sol
        L.hx, L.hy, L.xc, L.yc = np.diff(xn), np.diff(yn), 0.5 * (xn[1:] + xn[:-1]), 0.5 * (yn[1:] + yn[:-1])
        j, i = np.divmod(np.arange(nx * ny), nx)
        T = self.tensor
        L.dx, L.dy, L.vol = T(L.hx[i]), T(L.hy[j]), T(L.hx[i] * L.hy[j])
        L.solid = torch.as_tensor(sol.ravel(), device=self.dev)
        # faces of a cell: 0 west, 1 east, 2 south, 3 north
        L.bc = np.stack([bx[:, :-1], bx[:, 1:], by[:-1], by[1:]]).reshape(4, -1).copy()
        L.nb = np.stack([np.arange(nx * ny) + o for o in (-1, 1, -nx, nx)])
        ok = np.stack([i > 0, i < nx - 1, j > 0, j < ny - 1]) & (L.bc < 0)
        for f in range(4):
            ok[f][ok[f]] &= ~sol.ravel()[L.nb[f][ok[f]]]
        L.inner = ok & ~sol.ravel()[None]
        L.nb = np.where(L.inner, L.nb, np.arange(nx * ny)[None])
        L.bc = np.where(sol.ravel()[None], -1, L.bc)
        L.nbt = torch.as_tensor(L.nb, device=self.dev)
        L.int_ = torch.as_tensor(L.inner, device=self.dev).double()
        L.S = torch.stack([L.dy, L.dy, L.dx, L.dx])
        dist = []
        for f in range(4):
            c = (L.xc[i], L.xc[i], L.yc[j], L.yc[j])[f]
            n = L.nb[f]
            d = np.abs((L.xc[n % nx] if f < 2 else L.yc[n // nx]) - c)
            dist.append(np.where(L.inner[f], d, (L.hx[i] if f < 2 else L.hy[j])))
        L.dist = T(np.stack(dist))
        L.bcells = []          # boundary cells by face and id
        for f in range(4):
            for b in sorted(set(L.bc[f][L.bc[f] >= 0])):
                L.bcells.append((f, int(b), torch.as_tensor(np.nonzero(L.bc[f] == b)[0], device=self.dev)))
        d = i + j
        L.diag = [torch.as_tensor(np.nonzero((d == q) & ~sol.ravel())[0], device=self.dev) for q in range(nx + ny - 1)]
        L.side = []            # per pass and diagonal: (position on the diagonal, cell, its sweep-side boundary faces)
        for ps in range(2):
            per = []
            for q in range(nx + ny - 1):
                cells = np.nonzero((d == q) & ~sol.ravel())[0]
                per.append([(k, int(c), [(f, int(L.bc[f, c])) for f in (ps, 2 + ps) if L.bc[f, c] >= 0])
                            for k, c in enumerate(cells) if L.bc[ps, c] >= 0 or L.bc[2 + ps, c] >= 0])
            L.side.append(per)
        return L

    def _transfer(self, F, C):
        """Bilinear prolongation stencils on the fine cells (one-sided at edges and beside bodies), and restriction."""
        idx, wgt = np.zeros((F.nc, 4), np.int64), np.zeros((F.nc, 4))

        def fluid(a, b):
            return 0 <= a < C.nx and 0 <= b < C.ny and not C.sol[b, a]

        for j in range(F.ny):
            for i in range(F.nx):
                I, J = i // 2, j // 2
                own = J * C.nx + I
                c = j * F.nx + i
                idx[c] = own
                if F.sol[j, i]:
                    continue
                sx, sy = (-1 if F.xc[i] < C.xc[I] else 1), (-1 if F.yc[j] < C.yc[J] else 1)
                ox = [a for a in (I + sx, I - sx) if fluid(a, J)]
                oy = [b for b in (J + sy, J - sy) if fluid(I, b)]
                n, m = (ox[0] if ox else I), (oy[0] if oy else J)
                if ox and oy and not fluid(n, m):
                    n, m = next(((a, b) for a in ox for b in oy if fluid(a, b)), (n, J))
                bx = (F.xc[i] - C.xc[I]) / (C.xc[n] - C.xc[I]) if n != I else 0.0
                by = (F.yc[j] - C.yc[J]) / (C.yc[m] - C.yc[J]) if m != J else 0.0
                idx[c] = own, J * C.nx + n, m * C.nx + I, m * C.nx + n
                wgt[c] = (1 - bx) * (1 - by), bx * (1 - by), (1 - bx) * by, bx * by
        F.pidx, F.pw = torch.as_tensor(idx, device=self.dev), self.tensor(wgt)
        F.child = torch.as_tensor(np.stack([((2 * (np.arange(C.nc) // C.nx) + b) * F.nx + 2 * (np.arange(C.nc) % C.nx) + a)
                                            for b in (0, 1) for a in (0, 1)]), device=self.dev)

    def restrict(self, l, a):
        """Volume-weighted mean of the four children; the cell axis is the last but one."""
        F = self.lev[l]
        V = F.vol[F.child]
        return sum(a.index_select(-2, F.child[q]) * V[q][:, None] for q in range(4)) / V.sum(0)[:, None]

    def prolong(self, l, a):
        F = self.lev[l]
        return sum(a.index_select(-2, F.pidx[:, q]) * F.pw[:, q][:, None] for q in range(4))

    # ------------------------------------------------------------ gas
    def moments(self, f):
        w = self.w
        W = torch.stack([f[0] @ w, f[0] @ (w * self.u), f[0] @ (w * self.v), f[0] @ (w * self.e) + f[1] @ w], -1)
        U, V = (W[:, 1] / W[:, 0])[:, None], (W[:, 2] / W[:, 0])[:, None]
        cx, cy = self.u - U, self.v - V
        e = (0.5 * (cx * cx + cy * cy) * f[0] + f[1]) * w
        return W, torch.stack([(cx * e).sum(-1), (cy * e).sum(-1)], -1)

    def tau(self, rho, lam):
        return self.mu * lam ** (-self.omega) / (0.5 * rho / lam)

    def maxwell(self, rho, U, V, lam):
        return (rho * lam / math.pi)[:, None] * torch.exp(-lam[:, None] * ((self.u - U[:, None]) ** 2 +
                                                                          (self.v - V[:, None]) ** 2))

    def start(self, fields):
        rho, U, V, T = (self.tensor(a) for a in fields)
        g = self.maxwell(rho, U, V, 1 / T)
        self.f = torch.stack([g, g * (KI / 4 * T)[:, None]])
        self.W, self.q = self.moments(self.f)
        self.it = 0

    def fields(self):
        rho, U, V, lam = _prim(self.W)
        return torch.stack([rho, U, V, 1 / lam, self.q[:, 0], self.q[:, 1]])

    # ------------------------------------------------------------ Step 1: interface fluxes
    def flux(self, f, W):
        """Divergence of the time-averaged fluxes of f and of W over every cell."""
        L = self.lev[0]
        div, R = torch.zeros_like(f), torch.zeros_like(W)
        div, R = [div], [R]
        for axis in (0, 1):
            fc = 1 + 2 * axis                     # the upper face of a cell along this axis
            lo = np.nonzero(L.inner[fc])[0]
            step = max(1, int(2.5e7 // self.nv))
            for a in range(0, len(lo), step):
                c = torch.as_tensor(lo[a:a + step], device=self.dev)
                ph, F = self.inner_face(f, W, axis, c)
                n = L.nbt[fc][c]
                for cell, sg in ((c, -1.0), (n, 1.0)):
                    s = (sg * L.S[fc] / L.vol)[cell]
                    div[0] = div[0].index_add(1, cell, ph * s[:, None])
                    R[0] = R[0].index_add(0, cell, F * s[:, None])
        for fc, b, c in L.bcells:
            ph, F = self.edge_face(f, fc, b, c)
            s = (L.S[fc] / L.vol)[c] * (-1.0 if fc & 1 else 1.0)
            div[0] = div[0].index_add(1, c, ph * s[:, None])
            R[0] = R[0].index_add(0, c, F * s[:, None])
        return div[0], R[0]

    def flux_moments(self, ph):
        w = self.w
        return torch.stack([ph[0] @ w, ph[0] @ (w * self.u), ph[0] @ (w * self.v), ph[0] @ (w * self.e) + ph[1] @ w], -1)

    def inner_face(self, f, W, axis, c):
        L = self.lev[0]
        n, p, nn = L.nbt[1 + 2 * axis][c], L.nbt[2 * axis][c], None
        nn = L.nbt[1 + 2 * axis][n]
        ctr = self.tensor(np.tile(L.xc, L.ny) if axis == 0 else np.repeat(L.yc, L.nx))
        edge = self.tensor(np.tile(L.xn[1:], L.ny) if axis == 0 else np.repeat(L.yn[1:], L.nx))[c]
        h = (L.dx if axis == 0 else L.dy)
        un = self.v if axis else self.u
        hasL, hasR = (p != c), (nn != n)
        one = torch.ones_like(edge)
        r1 = 1 / torch.where(hasL, ctr[c] - ctr[p], one)
        r2 = 1 / (ctr[n] - ctr[c])
        r3 = 1 / torch.where(hasR, ctr[nn] - ctr[n], one)
        hL, hR = edge - ctr[c], ctr[n] - edge
        fL, fR = f[:, c], f[:, n]
        d2 = (fR - fL) * r2[:, None]
        sL = _limited((fL - f[:, p]) * r1[:, None], d2) * hasL[:, None]
        sR = _limited(d2, (f[:, nn] - fR) * r3[:, None]) * hasR[:, None]
        up = torch.where(un > 0, 1.0, torch.where(un < 0, 0.0, 0.5))
        f0 = up * (fL + sL * hL[:, None]) + (1 - up) * (fR - sR * hR[:, None])
        sg = up * sL + (1 - up) * sR
        W0 = self.flux_moments(f0)
        rho, U, V, lam = _prim(W0)
        dt = self.mg["cfl"] * torch.minimum(h[c], h[n]) / (self.vmax if axis else self.umax)
        tau = self.tau(rho, lam)
        aL = _slope([(W0[:, m] - W[c, m]) / (rho * hL) for m in range(4)], U, V, lam)
        aR = _slope([(W[n, m] - W0[:, m]) / (rho * hR) for m in range(4)], U, V, lam)
        gM = self.maxwell(rho, U, V, lam)
        hM = gM * (KI / (4 * lam))[:, None]
        x4 = (KI * (KI + 2) / (16 * lam * lam))[:, None]

        def psi(a):
            b = a[0][:, None] + a[1][:, None] * self.u + a[2][:, None] * self.v + a[3][:, None] * self.e
            return torch.stack([b * gM + a[3][:, None] * hM, b * hM + a[3][:, None] * x4 * gM])

        ma = torch.where(un > 0, psi(aL), psi(aR))
        s = self.flux_moments(ma * un)
        A = psi(_slope([-s[:, m] / rho for m in range(4)], U, V, lam))
        cx, cy = self.u - U[:, None], self.v - V[:, None]
        c2 = cx * cx + cy * cy
        e = self.w * (0.5 * c2 * f0[0] + f0[1])
        qx, qy = (cx * e).sum(-1), (cy * e).sum(-1)
        Fq = ((1 - self.pr) * 4 * lam * lam / (5 * rho))[:, None] * (cx * qx[:, None] + cy * qy[:, None])
        g = torch.stack([gM * (1 + Fq * (2 * lam[:, None] * c2 - 4)), hM * (1 + Fq * (2 * lam[:, None] * c2 - 2))])
        q1, q2, q3, q4, q5 = ((t / dt)[:, None] for t in _time_integrals(dt, tau))
        ph = un * (q1 * g + q2 * un * ma + q3 * A + q4 * f0 + q5 * un * sg)
        return ph, self.flux_moments(ph)

    def edge_face(self, f, fc, b, c):
        """Free transport of the face distribution at boundary faces of id b on side fc of the cells c."""
        B, axis, out = self.bcs[b], fc >> 1, 1.0 if fc & 1 else -1.0
        un = self.v if axis else self.u
        uo = out * un
        fb = f[:, c]
        H = KI * B["t"] / 4
        if B["type"] == WALL:
            z = (self.w * uo * self.C[b])[uo < 0].sum()
            rho = -(fb[0] * (self.w * uo * (uo > 0))).sum(-1) / z
            g = rho[:, None] * self.C[b]
            ghost = torch.stack([g, g * H])
        elif B["type"] == SYMMETRY:
            ghost = fb[:, :, self.mirror[axis]]
        elif B["type"] == FARFIELD:
            g = (B["rho"] * self.C[b]).expand(len(c), -1)
            ghost = torch.stack([g, g * H])
        else:
            ghost = fb
        ph = un * torch.where(uo >= 0, fb, ghost)
        return ph, self.flux_moments(ph)

    # ------------------------------------------------------------ Step 2: prediction (FAS)
    def ghost(self, b, axis, W):
        """Ghost state of a boundary face and its Jacobian dB/dW."""
        B = self.bcs[b]
        n = len(W)
        M = torch.zeros(n, 4, 4, dtype=W.dtype, device=self.dev)
        if B["type"] == WALL:
            rho, U, V, lam = _prim(W)
            lw = 1 / B["t"]
            lg, Ug, Vg = 2 * lw - lam, 2 * B["u"] - U, 2 * B["v"] - V
            G = torch.stack([rho, rho * Ug, rho * Vg, 0.5 * rho * (Ug * Ug + Vg * Vg) + (KI + 2) * rho / (4 * lg)], -1)
            Y, K = lam / (lam - 2 * lw), KI + 2
            M[:, 0, 0] = 1
            M[:, 1, 0], M[:, 1, 1] = 2 * B["u"], -1
            M[:, 2, 0], M[:, 2, 2] = 2 * B["v"], -1
            M[:, 3, 0] = 2 * (B["u"] ** 2 + B["v"] ** 2) - 0.5 * (U * U + V * V) * (1 + Y * Y) + K / (4 * lam) * (Y * Y - Y)
            M[:, 3, 1], M[:, 3, 2], M[:, 3, 3] = U - 2 * B["u"] + U * Y * Y, V - 2 * B["v"] + V * Y * Y, -Y * Y
        elif B["type"] == FARFIELD:
            r, u, v = B["rho"], B["u"], B["v"]
            G = self.tensor([r, r * u, r * v, 0.5 * r * (u * u + v * v) + (KI + 2) * r * B["t"] / 4]).expand(n, 4)
        else:
            M += torch.eye(4, dtype=W.dtype, device=self.dev)
            G = W.clone()
            if B["type"] == SYMMETRY:
                G[:, 1 + axis] = -G[:, 1 + axis]
                M[:, 1 + axis, 1 + axis] = -1
        return G, M

    def outer(self, L, W):
        """The states across the four faces of every cell."""
        out = [W[L.nbt[f]] for f in range(4)]
        for f, b, c in L.bcells:
            out[f] = out[f].index_copy(0, c, self.ghost(b, f >> 1, W[c])[0])
        return out

    def gamma(self, L, W):
        gam = (KI + 4) / (KI + 2)
        G = []
        for f, o in enumerate(self.outer(L, W)):
            rho, U, V, lam = _prim(0.5 * (W + o))
            g = (V if f >> 1 else U).abs() + torch.sqrt(gam / (2 * lam)) + 2 * self.mu * lam ** (-self.omega) / rho / L.dist[f]
            G.append(g)
        L.G = G
        L.idiag = 1 / (sum(L.S[f] * G[f] for f in range(4)) / (2 * L.vol) + self.dti)
        L.idiag = torch.where(L.solid, torch.zeros_like(L.idiag), L.idiag)

    def split(self, L, W):
        acc = 0
        for f, o in enumerate(self.outer(L, W)):
            sg = 1.0 if f & 1 else -1.0
            T = sg * (_euler(W, f >> 1) + _euler(o, f >> 1)) + L.G[f][:, None] * (W - o)
            acc = acc + 0.5 * L.S[f][:, None] * T
        return torch.where(L.solid[:, None], torch.zeros_like(W), -acc / L.vol[:, None])

    def sgs_macro(self, L, W, R):
        hv = 0.5 / L.vol * L.idiag
        own = R * L.idiag[:, None]
        T0 = [_euler(W, 0), _euler(W, 1)]
        for ps in (0, 1):
            dW = torch.zeros_like(W)
            if ps:
                g = torch.zeros_like(W)
                for f, b, c in L.bcells:
                    if f & 1:
                        G, M = self.ghost(b, f >> 1, W[c])
                        dG = torch.einsum("nij,nj->ni", M, own[c])
                        t = _euler(G + dG, f >> 1) - _euler(G, f >> 1) - L.G[f][c][:, None] * dG
                        g = g.index_add(0, c, L.S[f][c][:, None] * t)
                own = own - g * hv[:, None]
            sg = 1.0 if ps else -1.0
            for d in (reversed(range(len(L.diag))) if ps else range(len(L.diag))):
                c = L.diag[d]
                if not len(c):
                    continue
                acc = 0
                for axis in (0, 1):
                    f = 2 * axis + ps
                    n = L.nbt[f][c]
                    on = (L.int_[f][c] * L.S[f][c])[:, None]
                    acc = acc + on * (sg * (_euler(W[n] + dW[n], axis) - T0[axis][n]) - L.G[f][c][:, None] * dW[n])
                dW[c] = own[c] - acc * hv[c][:, None]
            own = dW
        return dW

    def positive(self, W):
        return ((W[:, 0] > 0) & (W[:, 3] * W[:, 0] - 0.5 * (W[:, 1] ** 2 + W[:, 2] ** 2) > 0))[:, None]

    def fas(self, l, cyc):
        L = self.lev[l]
        self.gamma(L, L.Wn)
        L.P = L.Rc - self.split(L, L.Wn)
        L.Wc = L.Wn.clone()
        self.visit(l, cyc, True)

    def visit(self, l, cyc, first):
        L = self.lev[l]
        L.R = L.Rc if first else L.P + self.split(L, L.Wc)
        last = l == len(self.lev) - 1
        n = (1 if len(self.lev) == 1 else self.mg["nuc"]) if last else self.mg["nu1"]
        for m in range(n):
            L.Wc = L.Wc + self.sgs_macro(L, L.Wc, L.R)
            if last and m == n - 1:
                return
            L.R = L.P + self.split(L, L.Wc)
        C = self.lev[l + 1]
        C.Wn, C.Rc = self.restrict(l, L.Wc), self.restrict(l, L.R)
        self.fas(l + 1, cyc)
        if cyc in "WF":
            self.visit(l + 1, "W" if cyc == "W" else "V", False)
        t = L.Wc + self.prolong(l, C.Wc - C.Wn)
        L.Wc = torch.where(self.positive(t), t, L.Wc)
        for _ in range(self.mg["nu2"]):
            L.R = L.P + self.split(L, L.Wc)
            L.Wc = L.Wc + self.sgs_macro(L, L.Wc, L.R)

    # ------------------------------------------------------------ Steps 3-5: evolution (CS)
    def coef(self, f, L, c):
        """Coefficient of the neighbour across face f of the cells c (zero unless the velocity enters)."""
        un = (self.v if f >> 1 else self.u) * (1.0 if f & 1 else -1.0)
        return torch.clamp(un, max=0.0) * (1 / (L.dy if f >> 1 else L.dx)[c])[:, None]

    def diagonal(self, L):
        return L.it[:, None] + self.u.abs() / L.dx[:, None] + self.v.abs() / L.dy[:, None]

    def wall_rho(self, f, b, x):
        uo = (self.v if f >> 1 else self.u) * (1.0 if f & 1 else -1.0)
        z = (self.w * uo * self.C[b])[uo < 0].sum()
        return -(x[0] * (self.w * uo * (uo > 0))).sum(-1) / z

    def apply(self, L, x):
        y = self.diagonal(L) * x
        every = torch.arange(L.nc, device=self.dev)
        for f in range(4):
            y = y + self.coef(f, L, every) * L.int_[f][:, None] * x[:, L.nbt[f]]
        for f, b, c in L.bcells:
            t, H = self.bcs[b]["type"], KI * self.bcs[b]["t"] / 4
            xb = x[:, c]
            if t == WALL:
                g = self.wall_rho(f, b, xb)[:, None] * self.C[b]
                ghost = torch.stack([g, g * H])
            elif t == SYMMETRY:
                ghost = xb[:, :, self.mirror[f >> 1]]
            elif t == OUTFLOW:
                ghost = xb
            else:
                continue
            y = y.index_add(1, c, self.coef(f, L, c) * ghost)
        return y * ~L.solid[:, None]

    def sgs_micro(self, L, r):
        D = self.diagonal(L)
        b = r
        for ps in (0, 1):
            x = torch.zeros_like(r)
            order = range(len(L.diag))
            for d in (reversed(order) if ps else order):
                c = L.diag[d]
                if not len(c):
                    continue
                base = b[:, c]
                for f in (ps, 2 + ps):
                    base = base - self.coef(f, L, c) * L.int_[f][c][:, None] * x[:, L.nbt[f][c]]
                den = D[c]
                new = base / den
                for k, cell, faces in L.side[ps][d]:
                    new[:, k] = self.edge_cell(L, c[k:k + 1], faces, base[:, k], den[k])
                x[:, c] = new
            b = D * x
        return x

    def edge_cell(self, L, c, faces, base, den):
        """A cell with boundary faces on the sweep side: its value together with those faces' ghosts."""
        Db = [self.coef(f, L, c)[0] for f, _ in faces]
        typ = [self.bcs[b]["type"] for _, b in faces]
        for t, D in zip(typ, Db):
            if t == OUTFLOW:
                den = den + D
        x = base / den
        H = [KI * self.bcs[b]["t"] / 4 for _, b in faces]
        if typ == [WALL, WALL]:
            k = [self.wall_rho(f, b, x) for f, b in faces]
            m = [-self.wall_rho(f, b, [Db[1 - q] * self.C[faces[1 - q][1]] / den]) for q, (f, b) in enumerate(faces)]
            # rho_0 = k_0 + m_0 rho_1, rho_1 = k_1 + m_1 rho_0
            r0 = (k[0] + m[0] * k[1]) / (1 - m[0] * m[1])
            rho = [r0, k[1] + m[1] * r0]
            a = base.clone()
            for q, (f, b) in enumerate(faces):
                g = Db[q] * self.C[b] * rho[q]
                a = a - torch.stack([g, g * H[q]])
            return a / den
        for _ in range(3 if SYMMETRY in typ else 1):
            a = base
            for q, (f, b) in enumerate(faces):
                if typ[q] == WALL:
                    g = self.C[b] * self.wall_rho(f, b, x)
                    a = a - Db[q] * torch.stack([g, g * H[q]])
                elif typ[q] == SYMMETRY:
                    a = a - Db[q] * x[:, self.mirror[f >> 1]]
            x = a / den
        return x

    def cs(self, l, r, cyc):
        L = self.lev[l]
        df = torch.zeros_like(r)
        last = l == len(self.lev) - 1
        n = (1 if len(self.lev) == 1 else self.mg["nuc"]) if last else self.mg["nu1"]
        for m in range(n):
            x = self.sgs_micro(L, r)
            df = df + x
            if last and m == n - 1:
                return df
            r = r - self.apply(L, x)
        rc = self.restrict(l, r)
        dc = self.cs(l + 1, rc, cyc)
        if cyc in "WF":
            dc = dc + self.cs(l + 1, rc - self.apply(self.lev[l + 1], dc), "W" if cyc == "W" else "V")
        x = self.prolong(l, dc)
        df = df + x
        for _ in range(self.mg["nu2"]):
            r = r - self.apply(L, x)
            x = self.sgs_micro(L, r)
            df = df + x
        return df

    def equilibrium(self, W, q):
        rho, U, V, lam = _prim(W)
        g = self.maxwell(rho, U, V, lam)
        cx, cy = self.u - U[:, None], self.v - V[:, None]
        l2c2 = 2 * lam[:, None] * (cx * cx + cy * cy)
        Fq = ((1 - self.pr) * 4 * lam * lam / (5 * rho))[:, None] * (cx * q[:, :1] + cy * q[:, 1:])
        return torch.stack([g * (1 + Fq * (l2c2 - 4)), g * (KI / (4 * lam))[:, None] * (1 + Fq * (l2c2 - 2))]), \
            1 / self.tau(rho, lam)

    def iterate(self):
        L = self.lev[0]
        a = self.mg["dtn_growth"]
        self.dti = 1 / (a ** self.it * self.dtp) if a > 0 else 0.0
        div, R = self.flux(self.f, self.W)
        fluid = ~L.solid
        L.Wn, L.Rc = self.W, R
        self.fas(0, self.cycle)
        Wt = torch.where(self.positive(L.Wc), L.Wc, L.Wn)
        g, it = self.equilibrium(Wt, self.q)
        r = ((g - self.f) * it[:, None] + div) * fluid[:, None]
        del g, div
        for l, V in enumerate(self.lev):
            if l:
                Wt = self.restrict(l - 1, Wt)
            rho, _, _, lam = _prim(Wt)
            V.it = 1 / self.tau(rho, lam) + self.dti
        df = self.cs(0, r, self.cycle)
        W, _ = self.moments(self.f + df)
        self.f = torch.where(self.positive(W), self.f + df, self.f)
        self.W, self.q = self.moments(self.f)
        self.it += 1
        return [float(t) for t in torch.sqrt((R * R).sum(0) / int(fluid.sum()))]

    def wall(self, b):
        """Pressure, shear and heat flux on the faces of wall b, x-faces first, in face order."""
        L, B = self.lev[0], self.bcs[b]
        rows = []
        for f, bb, cells in L.bcells:
            if bb != b:
                continue
            axis, uo = f >> 1, (self.v if f >> 1 else self.u) * (1.0 if f & 1 else -1.0)
            fb = self.f[:, cells]
            g = self.wall_rho(f, b, fb)[:, None] * self.C[b]
            g = torch.where(uo >= 0, fb, torch.stack([g, g * (KI * B["t"] / 4)]))
            ut = self.u - B["u"] if axis else self.v - B["v"]
            e = 0.5 * ((self.u - B["u"]) ** 2 + (self.v - B["v"]) ** 2)
            q = torch.stack([g[0] @ (self.w * uo * uo), g[0] @ (self.w * uo * ut),
                             g[0] @ (self.w * uo * e) + g[1] @ (self.w * uo)])
            i, j = cells % L.nx, cells // L.nx
            key = (j * (L.nx + 1) + i + (f & 1)) if axis == 0 else ((1 << 30) + (j + (f & 1)) * L.nx + i)
            rows.append((key, q))
        key, q = torch.cat([k for k, _ in rows]), torch.cat([v for _, v in rows], -1)
        return q[:, torch.argsort(key)]

    # ------------------------------------------------------------ transposed Jacobian of the steady equations
    def product(self, mu):
        f = self.f.clone().requires_grad_(True)
        W, q = self.moments(f)
        g, it = self.equilibrium(W, q)
        N = (g - f) * it[:, None] + self.flux(f, W)[0]
        return torch.autograd.grad((N * mu).sum(), f)[0]
