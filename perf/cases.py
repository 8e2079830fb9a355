"""Performance cases of the matrix-free FMG Stokes library, through the public
binding (paper_2010_13513_gb300.hhg).

Every case is one call (or one pair of transfer calls) that a user's solver
makes, on a problem set up and autotuned as the benchmark does.  Sizes are
those of the repository's own workloads: the P1-P1 level-4 problem in FP64,
the P2-P1 level-6 and level-7 problems on the 6-tetrahedron cube, the
variable-viscosity P1-P1 problem on the 48-tetrahedron cube, and a batch of
uneven problems.

`exact` restates the same steps in 64 bits with plain torch on the canonical
nodal lattices (element matrices by quadrature, gathered and scattered element
by element; the Gauss-Seidel phases from the stencils summed from them).
"""
import itertools
import math

import numpy as np
import torch

from paper_2010_13513_gb300 import hhg

# groups of P2 velocity DoFs by parity offset (x, y, z), in array order
GROUP_OFF = ((0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, 0, 1), (0, 1, 1), (1, 1, 1))
# the smoothing tuples of the benchmark: the level-7 headline, the
# variable-viscosity problem, V(3,3), and the batch (by discretisation)
TUPLES = {
    "headline": dict(nu_pre=1, nu_post=3, nu_inc=1, kappa=1, ahat="f", xi=3),
    "visc": dict(nu_pre=2, nu_post=3, nu_inc=2, kappa=1, ahat="s", xi=1),
    "v33": dict(nu_pre=3, nu_post=3, nu_inc=0, kappa=1, ahat="s", xi=1),
    "batch_p1": dict(nu_pre=2, nu_post=2, nu_inc=2, kappa=2, ahat="s", xi=1),
    "batch_p2": dict(nu_pre=1, nu_post=2, nu_inc=1, kappa=2, ahat="f", xi=3),
}
OMEGA_INV = {"P1P1": 0.6, "P2P1": 0.32}


def listed():
    """The cases, smallest first."""

    def c(name, kind, disc, prec, L, box=(1, 1, 1), nu_a=0.0, tuple_="headline", count=1):
        return dict(name=name, kind=kind, disc=disc, prec=prec, L=L, mx=box[0], my=box[1], mz=box[2], nu_a=nu_a,
                    tuple=tuple_, count=count)

    return [
        # the convergence check after a cycle of the smallest workload: residual and its norms, read by the host
        c("residual_norms_p1_l4_fp64", "residual", "P1P1", "fp64", 4),
        # the smallest whole solve: plain FP64 P1-P1 at level 4 with V(3,3), replayed as a graph (launch-bound)
        c("fmg_p1_l4_fp64", "fmg", "P1P1", "fp64", 4, tuple_="v33"),
        # one smoothing step of the FP64-only P2-P1 solve on a middle level
        c("smooth_p2_l5_fp64", "smooth", "P2P1", "fp64", 5),
        # both transfers between two levels of a V-cycle, on a box that is no cube
        c("transfer_p2_l6_fp32", "transfer", "P2P1", "fp32", 6, box=(2, 1, 1)),
        # symmetric smoothing of the variable-viscosity problem on the 48-tetrahedron cube, one level below the finest
        c("smooth_p1_visc_l6_fp32", "smooth", "P1P1", "fp32", 6, box=(2, 2, 2), nu_a=2.5478, tuple_="visc"),
        # one FP32 V-cycle of the level-6 P2-P1 problem: every level's smoother, residual and transfers
        c("vcycle_p2_l6_fp32", "vcycle", "P2P1", "fp32", 6),
        # the operator apply that the roofline is quoted on
        c("apply_p2_l7_fp32", "apply", "P2P1", "fp32", 7),
        # the same for the variable-viscosity P1-P1 problem at its full size
        c("apply_p1_visc_l7_fp32", "apply", "P1P1", "fp32", 7, box=(2, 2, 2), nu_a=2.5478, tuple_="visc"),
        # the defect of one iterative-refinement step at the largest size
        c("defect_p2_l7", "defect", "P2P1", "mixed", 7),
        # one smoothing step on the finest level: most of a solve's time
        c("smooth_p2_l7_fp32", "smooth", "P2P1", "fp32", 7),
        # the headline: a whole mixed-precision FMG solve at level 7
        c("fmg_p2_l7_mixed", "fmg", "P2P1", "mixed", 7),
        # many independent problems of uneven size and both discretisations, one graph
        c("batch_12_uneven_fp64", "batch", "P1P1", "fp64", 5, tuple_="batch_p1", count=12),
    ]


def draw(rng):
    """One more case of the same ranges: any step, discretisation, precision and
    level, boxes of 1 to 3 cubes a side, at most the listed sizes."""
    kind = rng.choice(["residual", "apply", "smooth", "smooth", "transfer", "vcycle", "defect", "fmg", "batch"])
    disc = rng.choice(["P1P1", "P2P1"])
    p2 = disc == "P2P1"
    prec = {"defect": "mixed", "batch": "fp64", "fmg": rng.choice(["fp64", "mixed"]) if p2 else "fp64"}.get(
        kind, rng.choice(["fp32", "fp32", "fp64"]))
    mixed_fmg = kind == "fmg" and prec == "mixed"            # large problems: their FP64 solutions are its use
    # cells of the finest level, at most those of the listed case of the kind
    most = 2 ** (21 if p2 else 24)
    if prec == "fp64" or kind in ("fmg", "batch", "vcycle"):
        most = 2 ** (18 if p2 else 21) * (2 if mixed_fmg else 1)
    while True:
        L = 6 if mixed_fmg else rng.randint(3, 7)
        box = [rng.randint(1, 3) for _ in range(3)]
        if box[0] * box[1] * box[2] <= 9 and box[0] * box[1] * box[2] * 8 ** L <= most:
            break
    nu_a = rng.choice([0.0, 0.0, round(rng.uniform(0.5, 4.0), 4)])
    if kind == "batch":
        L, box, nu_a = rng.randint(3, 5), [1, 1, 1], 0.0
    tuple_ = rng.choice(["headline"] + ["v33"] * (not mixed_fmg)) if p2 else rng.choice(["visc", "v33"])
    if kind == "batch":
        disc, tuple_ = "P1P1", "batch_p1"
    return dict(kind=kind, disc=disc, prec=prec, L=L, mx=box[0], my=box[1], mz=box[2], nu_a=nu_a, tuple=tuple_,
                count=rng.randint(3, 12) if kind == "batch" else 1)


# ------------------------------------------------------------------ geometry
class Grid:
    """One level: cells, mesh width, nodal lattices and the device layout."""

    def __init__(self, disc, box, level):
        self.q = 2 if disc == "P2P1" else 1                  # velocity lattice: q nodes per cell and direction
        self.G = 8 if disc == "P2P1" else 1
        self.n = tuple(b * 2 ** level for b in box)          # cells (x, y, z)
        self.h = 1.0 / max(box) / 2 ** level
        self.vshape = (3,) + tuple(self.q * c + 1 for c in self.n[::-1])
        self.pshape = tuple(c + 1 for c in self.n[::-1])
        self.sites = self.pshape[0] * self.pshape[1] * self.pshape[2]
        sx = self.n[0] + 3
        self.sx = (sx + 3) // 4 * 4 if self.n[0] >= 64 else sx
        self.arr = (self.sx * (self.n[1] + 3) * (self.n[2] + 3) + 63) // 64 * 64
        self.dofs = 3 * math.prod(self.vshape[1:]) + self.sites

    def pack(self, u, p, dtype=torch.float64):
        """Canonical velocity and pressure lattices -> the library's vector."""
        nx, ny, nz = self.n
        out = torch.zeros(3 * self.G + 1, self.arr, dtype=dtype, device=u.device)
        v = out[:, :self.sx * (ny + 3) * (nz + 3)].unflatten(1, (nz + 3, ny + 3, self.sx))
        for c in range(3):
            for g in range(self.G):
                ox, oy, oz = GROUP_OFF[g]
                s = u[c, oz::self.q, oy::self.q, ox::self.q]
                v[c * self.G + g, 1:1 + s.shape[0], 1:1 + s.shape[1], 1:1 + s.shape[2]] = s
        v[3 * self.G, 1:nz + 2, 1:ny + 2, 1:nx + 2] = p
        return out.flatten()

    def coords(self, q, device):
        ax = [torch.arange(q * c + 1, dtype=torch.float64, device=device) * (self.h / q) for c in self.n]
        return ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]


def _box(case):
    return case["mx"], case["my"], case["mz"]


def _specs(case):
    """The problems of a case: (discretisation, box, level, tuple) each."""
    if case["kind"] != "batch":
        return [(case["disc"], _box(case), case["L"], case["tuple"])]
    rng = np.random.default_rng([case["count"], case["L"]])
    out = []
    for i in range(case["count"]):
        box = tuple(int(v) for v in rng.integers(1, 3, size=3))
        disc = "P1P1" if i % 2 == 0 else "P2P1"
        out.append((disc, box, int(rng.integers(3, case["L"] + 1)), "batch_p1" if disc == "P1P1" else "batch_p2"))
    return out


def _coarse(disc):
    return 0 if disc == "P1P1" else 1


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


# -------------------------------------------------------------------- inputs
def _modes(rng, X, kmax=4, n=8):
    """A sum of n sine modes with random wave vectors, phases and N(0, 1) amplitudes."""
    x, y, z = X
    out = 0.0
    for _ in range(n):
        k = rng.integers(1, kmax + 1, size=3)
        # sin(a + b + c) of a separable sum, as the imaginary part of a product
        e = [torch.exp(1j * math.pi * float(kk) * t) for kk, t in zip(k, (x, y, z))]
        e[0] = e[0] * (float(rng.standard_normal()) * np.exp(1j * rng.uniform(0, 2 * math.pi)))
        out = out + (e[2] * (e[1] * e[0])).imag
    return out


def _interior(grid, device):
    m = torch.zeros(grid.vshape[1:], dtype=torch.float64, device=device)
    m[1:-1, 1:-1, 1:-1] = 1.0
    return m


def _noise(shape, seed, device):
    gen = torch.Generator(device=device)
    gen.manual_seed(seed)
    return torch.randn(shape, generator=gen, dtype=torch.float64, device=device)


def _vector(grid, seed, which, scale=1.0):
    """A lifting-form vector (zero Dirichlet velocities): smooth modes plus a tenth of noise."""
    dev = _device()
    rng = np.random.default_rng([seed, which])
    Xu, Xp = grid.coords(grid.q, dev), grid.coords(1, dev)
    u = torch.empty(grid.vshape, dtype=torch.float64, device=dev)
    for c in range(3):
        u[c] = _modes(rng, Xu)
    p = _modes(rng, Xp)
    s = int(rng.integers(1 << 30))
    u += 0.1 * _noise(grid.vshape, s, dev)
    p = p + 0.1 * _noise(grid.pshape, s + 1, dev)
    u *= _interior(grid, dev)
    return scale * u, scale * p


def _nodal(grid, seed, which):
    """Forcing and Dirichlet data at the velocity nodes of an analytic solution of the benchmark's kind (a shear
    velocity per component and a product-of-sines pressure) with random amplitudes, wave numbers and phases."""
    dev = _device()
    rng = np.random.default_rng([seed, which])
    X = grid.coords(grid.q, dev)
    f = torch.empty(grid.vshape, dtype=torch.float64, device=dev)
    w = torch.empty_like(f)
    k = [float(v) for v in rng.uniform(2, 6, size=3)]
    arg = [k[d] * X[d] + float(rng.uniform(0, 6)) for d in range(3)]
    s, ds = [torch.sin(a) for a in arg], [kk * torch.cos(a) for kk, a in zip(k, arg)]
    for c, along in enumerate((2, 0, 1)):
        m = float(rng.uniform(2, 8))
        u = float(rng.uniform(1, 8)) * torch.cos(m * X[along] + float(rng.uniform(0, 6)))
        w[c] = u
        f[c] = m * m * u + math.prod(ds[d] if d == c else s[d] for d in range(3))
    return f, w


_STREAM = []


def _stream():
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())      # a created stream: whole solves replay as graphs
    return _STREAM[0]


def _params(disc, tuple_):
    return hhg.Params.make(**TUPLES[tuple_], omega_inv=OMEGA_INV[disc])


def _inputs(case, seed):
    """The vectors of a single-step case in 64 bits, canonical (u, p) each, by name."""
    g = Grid(case["disc"], _box(case), case["L"])
    kind = case["kind"]
    h3 = g.h ** 3
    if kind == "apply":
        return {"x": _vector(g, seed, 0)}
    if kind in ("residual", "defect"):
        return {"x": _vector(g, seed, 0), "b": _vector(g, seed, 1, h3)}
    if kind in ("smooth", "vcycle"):
        # the correction of a V-cycle: a small iterate and a defect of the load's size
        return {"x": _vector(g, seed, 0, 0.01), "b": _vector(g, seed, 1, h3)}
    gc = Grid(case["disc"], _box(case), case["L"] - 1)
    return {"rf": _vector(g, seed, 0, h3), "xc": _vector(gc, seed, 1, 0.01), "xf": _vector(g, seed, 2, 0.01)}


def prepare(case, seed):
    stream = _stream()
    state = {"case": case, "stream": stream}
    pbs = []
    with torch.cuda.stream(stream):
        for i, (disc, box, L, tuple_) in enumerate(_specs(case)):
            solve = "fp64" if case["prec"] == "fp64" else "mixed"
            pb = hhg.Problem(hhg.Mesh.box(*box, 1.0 / max(box)), disc=disc, L=L, coarse_level=_coarse(disc),
                             solve=solve, nu_a=case["nu_a"], stream=stream)
            pb.autotune(reps=3)
            if case["kind"] in ("fmg", "batch"):
                fs, ws = [], []
                for l in range(pb.lc, L + 1):
                    f, w = _nodal(Grid(disc, box, l), seed, i)
                    fs.append(f.flatten().cpu())
                    ws.append(w.flatten().cpu())
                pb.set_rhs_levels(pb.lc, fs, ws)
            pbs.append(pb)
        state["prm"] = [_params(s[0], s[3]) for s in _specs(case)]
        state["pb"] = pbs[0]
        if case["kind"] == "batch":
            state["batch"] = hhg.Batch(pbs)
            state["xs"] = [pb.level_vector(pb.L, "x") for pb in pbs]
        elif case["kind"] == "fmg":
            state["x"] = pbs[0].new_vector(case["L"])
        else:
            dtype = torch.float32 if case["prec"] == "fp32" else torch.float64
            for name, (u, p) in _inputs(case, seed).items():
                g = Grid(case["disc"], _box(case), case["L"] - (name == "xc"))
                state[name] = g.pack(u, p, dtype)
            prec = hhg.FP32 if case["prec"] != "fp64" else hhg.FP64
            state["y"] = pbs[0].new_vector(case["L"], prec)
            if case["kind"] == "transfer":
                state["rc"] = pbs[0].new_vector(case["L"] - 1, prec)
    stream.synchronize()
    return state


def run(state):
    case, pb, prm = state["case"], state["pb"], state["prm"][0]
    kind, L = case["kind"], case["L"]
    if kind == "apply":
        pb.apply(L, "FULL", state["x"], state["y"])
        return state["y"]
    if kind == "residual":
        norms = pb.residual(L, state["x"], state["b"], state["y"], norms=True)
        return [state["y"], norms[0], norms[1]]
    if kind == "defect":
        pb.refinement_residual(L, state["x"], state["b"], state["y"])
        return state["y"]
    if kind == "smooth":
        pb.smooth(L, prm, 1, state["x"], state["b"])
        return state["x"]
    if kind == "vcycle":
        pb.vcycle(L, prm, state["x"], state["b"])
        return state["x"]
    if kind == "transfer":
        pb.restrict(L, state["rf"], state["rc"])
        pb.prolongate_add(L, state["xc"], state["xf"])
        return [state["rc"], state["xf"]]
    if kind == "fmg":
        pb.fmg_solve(prm, state["x"], stats=False)
        return state["x"]
    state["batch"].fmg_solve(state["prm"], stream=state["stream"])
    return state["xs"]


# ---------------------------------------------------------------------- work
# multiply-adds per lattice site of the operator blocks (three components, constant viscosity, zero weights left out)
TERMS = {"P1P1": {"FULL": 112, "A": 21, "BT": 42, "BC": 49}, "P2P1": {"FULL": 870, "A": 558, "BT": 156, "BC": 156}}


def work(case):
    nbytes = flops = 0.0
    for disc, box, L, tuple_ in _specs(case):
        g, t, s = Grid(disc, box, L), TERMS[disc], TUPLES[tuple_]
        es = 8 if case["prec"] == "fp64" else 4
        sweep = t["BT"] + t["BC"] + t["A"] * s["xi"] * (2 if s["ahat"] == "s" else 1)
        cyc = (s["nu_pre"] + s["nu_post"]) * sweep + t["FULL"]
        kind = case["kind"]
        if kind == "apply":
            b, f = 2 * es * g.dofs, t["FULL"]
        elif kind == "residual":
            b, f = 3 * es * g.dofs, t["FULL"]
        elif kind == "defect":                         # x and b in FP64, the defect in FP32
            b, f = 20 * g.dofs, t["FULL"]
        elif kind == "smooth":                         # x read and written, b read
            b, f = 3 * es * g.dofs, sweep
        elif kind == "vcycle":
            b, f = 3 * es * g.dofs, cyc * 8 / 7
        elif kind == "transfer":                       # fine defect read, coarse written; coarse read, fine updated
            b, f = es * g.dofs * (3 + 2 / 8), 2 * (3 * 8 * 10 if disc == "P2P1" else 3 * 2)
        else:                                          # right-hand sides read, the solution written
            b, f = 8 * g.dofs * (1 + 8 / 7), cyc * s["kappa"] * 64 / 49
        nbytes += b
        flops += 2.0 * f * g.sites
    return {"bytes": nbytes, "flops": flops}


# --------------------------------------------------------------------- exact
PERMS = list(itertools.permutations(range(3)))
EDGES = ((0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3))


def _tets(order):
    """The six tetrahedra of a cube: local node positions (in 1 / order cells), vertices, place of the z step."""
    out = []
    for perm in PERMS:
        v = [np.zeros(3, dtype=int)]
        for d in perm:
            v.append(v[-1] + np.eye(3, dtype=int)[d])
        pos = [order * a for a in v] + ([v[i] + v[j] for i, j in EDGES] if order == 2 else [])
        out.append((np.array(pos), np.array(v), perm.index(2)))
    return out


def _element(v, order, h):
    """Element matrices of one tetrahedron by a quadrature rule exact for them."""
    X = h * v.astype(float)
    J = (X[1:] - X[0]).T
    vol, Ji = abs(np.linalg.det(J)) / 6, np.linalg.inv(J)
    gl = np.vstack([-Ji.sum(0), Ji])                         # gradients of the barycentric coordinates
    t, w = np.polynomial.legendre.leggauss(5)
    t, w = (t + 1) / 2, w / 2
    n = 4 if order == 1 else 10
    K, M, D, W = np.zeros((n, n)), np.zeros((n, n)), np.zeros((3, 4, n)), np.zeros(n)
    for (a, wa), (b, wb), (c, wc) in itertools.product(zip(t, w), repeat=3):
        l = np.array([0, a, (1 - a) * b, (1 - a) * (1 - b) * c])
        l[0] = 1 - l.sum()
        wq = 6 * vol * wa * wb * wc * (1 - a) ** 2 * (1 - b)
        if order == 1:
            phi, dphi = l, gl
        else:
            phi = np.array([x * (2 * x - 1) for x in l] + [4 * l[i] * l[j] for i, j in EDGES])
            dphi = np.vstack([(4 * l[i] - 1) * gl[i] for i in range(4)] +
                             [4 * (l[i] * gl[j] + l[j] * gl[i]) for i, j in EDGES])
        K += wq * dphi @ dphi.T
        M += wq * np.outer(phi, phi)
        W += wq * phi
        for d in range(3):
            D[d] -= wq * np.outer(l, dphi[:, d])
    stab = vol ** (2 / 3) / 12                               # PSPG: h_T^2 / 12
    return {"K": K, "M": M, "D": D, "C": stab * vol * gl @ gl.T, "load": -stab * np.einsum("kd,j->dkj", gl, W),
            "lump": vol / 4}


class Exact:
    """One level of the discrete problem in 64 bits on the canonical lattices."""

    def __init__(self, disc, box, level, nu_a, dev):
        self.g = g = Grid(disc, box, level)
        self.dev, self.disc, self.nu_a = dev, disc, nu_a
        self.tets = [(pos, 1 * v, zp, _element(v, g.q, g.h)) for pos, v, zp in _tets(g.q)]
        k = torch.arange(g.n[2], dtype=torch.float64, device=dev)
        self.nu = [torch.exp(nu_a * g.h * (k + (3 - zp) / 4))[:, None, None] for _, _, zp, _ in self.tets]
        self.mask = _interior(g, dev)
        one = torch.ones(g.pshape, dtype=torch.float64, device=dev)
        self.ml, self.mlhat = torch.zeros_like(one), torch.zeros_like(one)
        for (_, v, _, e), nu in zip(self.tets, self.nu):
            for a in v:
                self.at(self.ml, a, 1).add_(e["lump"])
                self.at(self.mlhat, a, 1).add_(e["lump"] / nu)
        self.rows = self._stencils()

    def at(self, x, pos, q):
        """The values at one local node of every cell."""
        n = self.g.n[::-1]
        s = tuple(slice(int(o), int(o) + q * (c - 1) + 1, q) for o, c in zip(pos[::-1], n))
        return x[(Ellipsis,) + s]

    def form(self, name, x, out, scale=0):
        """out += the form's element matrices applied to x; scale: power of the viscosity."""
        q = self.g.q
        for (pos, v, _, e), nu in zip(self.tets, self.nu):
            f = nu ** scale if scale else 1.0
            if name in ("K", "M"):
                src, dst, qs, qd, m = pos, pos, q, q, e[name]
            elif name == "C":
                src, dst, qs, qd, m = v, v, 1, 1, e["C"]
            elif name == "DT":
                src, dst, qs, qd, m = v, pos, 1, q, e["D"].transpose(0, 2, 1)
            else:
                src, dst, qs, qd, m = pos, v, q, 1, e[name]
            for a, pa in enumerate(dst):
                if name == "DT":
                    for d in range(3):
                        t = sum(float(m[d, a, b]) * self.at(x, pb, qs) for b, pb in enumerate(src) if m[d, a, b])
                        if not isinstance(t, int):
                            self.at(out[d], pa, qd).add_(t * f)
                elif name in ("D", "load"):
                    t = sum(float(m[d, a, b]) * self.at(x[d], pb, qs) for d in range(3) for b, pb in enumerate(src)
                            if m[d, a, b])
                    self.at(out, pa, qd).add_(t * f)
                else:
                    t = sum(float(m[a, b]) * self.at(x, pb, qs) for b, pb in enumerate(src) if m[a, b])
                    self.at(out, pa, qd).add_(t * f)
        return out

    def gradient(self, p):
        return self.form("DT", p, torch.zeros(self.g.vshape, dtype=torch.float64, device=self.dev)) * self.mask

    def continuity(self, u, p):
        out = self.form("D", u, torch.zeros_like(p))
        return out - self.form("C", p, torch.zeros_like(p), -1) if self.disc == "P1P1" else out

    def apply(self, u, p):
        return (self.form("K", u, torch.zeros_like(u), 1) * self.mask + self.gradient(p), self.continuity(u, p))

    def residual(self, x, b):
        y = self.apply(*x)
        return b[0] - y[0], b[1] - y[1]

    def rhs(self, f, w):
        wb = w * (1 - self.mask)
        r = (self.form("M", f, torch.zeros_like(f)) - self.form("K", wb, torch.zeros_like(f), 1)) * self.mask
        z = torch.zeros(self.g.pshape, dtype=torch.float64, device=self.dev)
        s = -self.form("D", wb, z.clone())
        if self.disc == "P1P1":
            s = s + self.form("load", f, z, -1)
        return r, s - s.mean()

    def _stencils(self):
        """Per parity offset the terms {offset: weight} of an interior velocity row, relative to exp(nu_a h k)."""
        q, rows = self.g.q, {}
        for o in GROUP_OFF[:self.g.G]:
            r = {}
            for pos, _, zp, e in self.tets:
                for a, pa in enumerate(pos):
                    if any((o[d] - pa[d]) % q for d in range(3)):
                        continue
                    cz = (o[2] - pa[2]) // q
                    f = math.exp(self.nu_a * self.g.h * (cz + (3 - zp) / 4))
                    for b, pb in enumerate(pos):
                        d = tuple(int(t) for t in pb - pa)
                        r[d] = r.get(d, 0.0) + f * e["K"][a, b]
            top = r[(0, 0, 0)]
            rows[o] = {d: w for d, w in r.items() if abs(w) > 1e-14 * top}
        return rows

    def phase(self, u, rhs, group, colour):
        """One Gauss-Seidel phase: an edge group, or one colour of the vertex group."""
        o, q, n = GROUP_OFF[group], self.g.q, self.g.n
        first = [x if x else q for x in o]
        last = [q * c - (x if x else q) for x, c in zip(o, n)]

        def cut(x, d):
            return x[(slice(None),) + tuple(slice(first[e] + d[e], last[e] + d[e] + 1, q) for e in (2, 1, 0))]

        if any(l < f for f, l in zip(first, last)):
            return
        k = torch.arange(first[2] // q, last[2] // q + 1, dtype=torch.float64, device=self.dev)[:, None, None]
        a = cut(rhs, (0, 0, 0)) * torch.exp(-self.nu_a * self.g.h * k)
        for d, w in self.rows[o].items():
            if d != (0, 0, 0):
                a = a - w * cut(u, d)
        a /= self.rows[o][(0, 0, 0)]
        if colour is not None:
            ix = [torch.arange(f // q, l // q + 1, device=self.dev) for f, l in zip(first, last)]
            m = (ix[2][:, None, None] + ix[1][:, None] + ix[0]) % 4 == colour
            a = torch.where(m, a, cut(u, (0, 0, 0)))
        cut(u, (0, 0, 0)).copy_(a)

    def smooth(self, x, b, s, omega_inv, sweeps):
        u, p = x
        phases = [(0, c) for c in range(4)] + [(e, None) for e in range(1, self.g.G)]
        for _ in range(sweeps):
            r = b[0] - self.gradient(p)
            for _ in range(s["xi"]):
                for ph in phases + (phases[::-1] if s["ahat"] == "s" else []):
                    self.phase(u, r, *ph)
            p = p - (b[1] - self.continuity(u, p)) / self.mlhat / omega_inv
        return u, p


def _interpolate(xc, q):
    """The pairs (fine slice, coarse slice, weight) of the P1 (q = 1) or P2 (q = 2) interpolation of a lattice."""
    m = 2 * q
    n = [(s - 1) // q for s in xc.shape[-3:]][::-1]
    for cls in itertools.product(range(m), repeat=3):        # position within the coarse cell, in fine lattice units
        order = sorted(range(3), key=lambda d: -cls[d])
        xi = [cls[d] / m for d in order]
        l = np.array([1 - xi[0], xi[0] - xi[1], xi[1] - xi[2], xi[2]])
        pos, v, _ = _tets(q)[PERMS.index(tuple(order))]
        phi = l if q == 1 else [x * (2 * x - 1) for x in l] + [4 * l[i] * l[j] for i, j in EDGES]
        cells = [c + 1 if cls[d] == 0 else c for d, c in enumerate(n)]
        fine = tuple(slice(cls[d], cls[d] + m * (cells[d] - 1) + 1, m) for d in (2, 1, 0))
        for w, o in zip(phi, pos):
            if w:
                yield fine, tuple(slice(int(o[d]), int(o[d]) + q * (cells[d] - 1) + 1, q) for d in (2, 1, 0)), float(w)


def _prolong(xc, q, shape):
    out = torch.zeros(shape, dtype=xc.dtype, device=xc.device)
    for f, c, w in _interpolate(xc, q):
        out[(Ellipsis,) + f] += w * xc[(Ellipsis,) + c]
    return out


def _restrict(xf, q, shape):
    out = torch.zeros(shape, dtype=xf.dtype, device=xf.device)
    for f, c, w in _interpolate(out, q):
        out[(Ellipsis,) + c] += w * xf[(Ellipsis,) + f]
    return out


class Hierarchy:
    def __init__(self, disc, box, L, nu_a, tuple_):
        self.lc, self.L, self.s, self.om = _coarse(disc), L, TUPLES[tuple_], OMEGA_INV[disc]
        self.lv = {l: Exact(disc, box, l, nu_a, _device()) for l in range(self.lc, L + 1)}

    def down(self, l, r):
        f, c = self.lv[l], self.lv[l - 1]
        return _restrict(r[0], f.g.q, c.g.vshape) * c.mask, _restrict(r[1], 1, c.g.pshape)

    def up(self, l, x):
        f = self.lv[l]
        return _prolong(x[0], f.g.q, f.g.vshape) * f.mask, _prolong(x[1], 1, f.g.pshape)

    def coarse(self, b):
        """Solution of the coarse system bordered by the mean-pressure constraint."""
        e = self.lv[self.lc]
        inner = (e.mask > 0).expand(e.g.vshape).flatten().nonzero().flatten()
        nu, np_ = len(inner), e.g.sites
        if not hasattr(self, "K"):
            K = torch.zeros(nu + np_ + 1, nu + np_ + 1, dtype=torch.float64)
            for j in range(nu + np_):
                u = torch.zeros(e.g.vshape, dtype=torch.float64, device=e.dev)
                p = torch.zeros(e.g.pshape, dtype=torch.float64, device=e.dev)
                (u.view(-1)[inner[j]] if j < nu else p.view(-1)[j - nu]).fill_(1.0)
                y = e.apply(u, p)
                K[:-1, j] = torch.cat([y[0].flatten()[inner], y[1].flatten()]).cpu()
            K[nu:-1, -1] = K[-1, nu:-1] = e.ml.flatten().cpu()
            self.K = torch.linalg.lu_factor(K)
        r = torch.cat([b[0].flatten()[inner].cpu(), b[1].flatten().cpu(), torch.zeros(1, dtype=torch.float64)])
        x = torch.linalg.lu_solve(*self.K, r[:, None])[:-1, 0].to(e.dev)
        u = torch.zeros(e.g.vshape, dtype=torch.float64, device=e.dev)
        u.view(-1)[inner] = x[:nu]
        return u, x[nu:].view(e.g.pshape)

    def vcycle(self, top, l, x, b):
        if l == self.lc:
            return self.coarse(b)
        e, s = self.lv[l], self.s
        extra = (top - l) * s["nu_inc"]
        x = e.smooth(x, b, s, self.om, s["nu_pre"] + extra)
        bc = self.down(l, e.residual(x, b))
        xc = self.vcycle(top, l - 1, tuple(torch.zeros_like(t) for t in bc), bc)
        d = self.up(l, xc)
        return e.smooth((x[0] + d[0], x[1] + d[1]), b, s, self.om, s["nu_post"] + extra)

    def centred(self, l, x):
        ml = self.lv[l].ml
        return x[0], x[1] - (ml * x[1]).sum() / ml.sum()

    def fmg(self, seed, which):
        for l in range(self.lc, self.L + 1):
            e = self.lv[l]
            f, w = _nodal(e.g, seed, which)
            b = e.rhs(f, w)
            if l == self.lc:
                x = self.centred(l, self.coarse(b))
            else:
                x = self.up(l, (x[0] + lift, x[1]))
                for _ in range(self.s["kappa"]):
                    x = self.centred(l, self.vcycle(l, l, x, b))
            lift = w * (1 - e.mask)
        return e.g.pack(*x)


def exact(case, seed):
    kind, L = case["kind"], case["L"]
    if kind in ("fmg", "batch"):
        specs = _specs(case)
        if sum(s[1][0] * s[1][1] * s[1][2] * 8 ** s[2] for s in specs) > 2 ** 20:
            return None                                      # a whole level-7 solve in torch takes over 20 s
        xs = [Hierarchy(d, b, l, case["nu_a"], t).fmg(seed, i) for i, (d, b, l, t) in enumerate(specs)]
        return xs if kind == "batch" else xs[0]
    dtype = torch.float32 if case["prec"] == "fp32" else torch.float64
    x = {k: tuple(t.to(dtype).double() for t in v) for k, v in _inputs(case, seed).items()}
    if kind == "vcycle":
        h = Hierarchy(case["disc"], _box(case), L, case["nu_a"], case["tuple"])
        return h.lv[L].g.pack(*h.vcycle(L, L, x["x"], x["b"]))
    e = Exact(case["disc"], _box(case), L, case["nu_a"], _device())
    if kind == "apply":
        return e.g.pack(*e.apply(*x["x"]))
    if kind == "defect":
        return e.g.pack(*e.residual(x["x"], x["b"]))
    if kind == "residual":
        r = e.residual(x["x"], x["b"])
        return [e.g.pack(*r), float(r[0].norm()), float(r[1].norm())]
    if kind == "smooth":
        return e.g.pack(*e.smooth(x["x"], x["b"], TUPLES[case["tuple"]], OMEGA_INV[case["disc"]], 1))
    gc = Grid(case["disc"], _box(case), L - 1)
    q = e.g.q
    rc = (_restrict(x["rf"][0], q, gc.vshape) * _interior(gc, _device()), _restrict(x["rf"][1], 1, gc.pshape))
    xf = (x["xf"][0] + _prolong(x["xc"][0], q, e.g.vshape) * e.mask, x["xf"][1] + _prolong(x["xc"][1], 1, e.g.pshape))
    return [gc.pack(*rc), e.g.pack(*xf)]
