"""Performance cases of the PDEP library: what its users call, over the range they call it in.

A case is one public call (or the short sequence a program makes) on one of
the model systems the library is configured, tested and benchmarked with:
periodic Gaussian wells on the cubic grids 24^3 .. 64^3 and on the 64 x 64 x
192 slab.  `kind` names the entry point:

  hpsi    Context.apply_hamiltonian    H x for n vectors, FP64 / FP32 / double-float
  chi0    Context.chi0_apply           chi0bar phi and the density response
  stern   Context.sternheimer_solve    first-order states for given potentials
  pdep    Context.pdep_solve, then W^p of the eigenpairs by screening_apply
  screen  Context.screening_apply      chibar, eps^-1 or W^p from given eigenpairs
  imag    Context.chi0_imag            B(i nu) and Lambda(i nu) from Lanczos chains

A program sets one system up and then calls the library many times on it, so
the context of the system in hand is kept between preparations (one at a
time); the vectors, potentials and start blocks come from the seed.
"""
import functools
import math

import numpy as np
import torch

import paper_1501_03141_gb300 as pg

DEVICE = "cuda"
PRECISIONS = {"fp64": pg.PDEP_FP64, "mixed": pg.PDEP_MIXED, "df64": pg.PDEP_APPLY_DF64}

#: name -> (grid, cell edges in bohr, occupied states, seed, well count).  The
#: 24^3 parity system, the 48^3 benchmark system, members of the uneven batch
#: (L = 10 N / 24, 8 wells per 1000 bohr^3) and the deep / shallow slab pair
#: with its 48 lowest states occupied.
SYSTEMS = {
    "cube24": ((24, 24, 24), (10.0,) * 3, 8, 1501031410, 8),
    "cube48": ((48, 48, 48), (20.0,) * 3, 64, 1501031411, 64),
    "slab": ((64, 64, 192), (20.0, 20.0, 60.0), 48, 1501031414, 0),
}
#: members of the uneven batch a drawn case may pick
MEMBERS = (0, 2, 3, 4, 5, 7, 8, 9, 13, 14, 18, 19, 23, 25, 28, 30)


class System:
    """One Kohn-Sham system: the fields pdep_setup reads."""

    def __init__(self, name, grid, cell, v_r, n_occ, n_pdep):
        self.name, self.grid, self.cell, self.v_r = name, grid, cell, v_r
        self.n_occ, self.n_pdep = n_occ, n_pdep


def _wells(rng, n, cell, depth, width, zrange=None):
    out = []
    for _ in range(n):
        r = rng.uniform(0.0, 1.0, size=3) * np.asarray(cell)
        if zrange is not None:
            r[2] = zrange[0] + (r[2] / cell[2]) * (zrange[1] - zrange[0])
        out.append((r, rng.uniform(*depth), rng.uniform(*width)))
    return out


def _gaussian_sum(grid, cell, wells, sign):
    """sign * sum_a D_a exp(-|r - R_a|^2 / 2 w_a^2), summed over the periodic images per axis."""
    out = np.zeros(grid)
    for r, d, w in wells:
        axes = []
        for n, l, c in zip(grid, cell, r):
            m = int(math.ceil((12.0 * w + l) / l)) + 1
            x = (np.arange(n) * (l / n) - c)[:, None] - l * np.arange(-m, m + 1)[None, :]
            axes.append(np.where(np.abs(x) < 12.0 * w, np.exp(-x * x / (2.0 * w * w)), 0.0).sum(axis=1))
        out += sign * d * (axes[0][:, None, None] * axes[1][None, :, None] * axes[2][None, None, :])
    return out


@functools.lru_cache(maxsize=4)
def _system(name):
    if name.startswith("member"):
        k = int(name[6:])
        rng = np.random.default_rng(1501031430 + k)
        n = int(rng.choice(np.asarray((24, 32, 40, 48, 64))))
        n_occ = int(rng.integers(8, 97))
        grid, cell = (n,) * 3, (n * 10.0 / 24.0,) * 3
        wells = _wells(rng, int(round(8.0 * (cell[0] / 10.0) ** 3)), cell, (1.0, 3.0), (0.8, 1.5))
    else:
        grid, cell, n_occ, seed, n_wells = SYSTEMS[name]
        rng = np.random.default_rng(seed)
        if name == "slab":
            wells = _wells(rng, 192, cell, (2.0, 4.0), (0.8, 1.5), (0.0, 30.0))
            wells += _wells(rng, 48, cell, (0.5, 1.5), (0.8, 1.5), (30.0, 60.0))
        else:
            wells = _wells(rng, n_wells, cell, (1.0, 3.0), (0.8, 1.5))
    return System(name, grid, cell, _gaussian_sum(grid, cell, wells, -1.0), n_occ, 2 * n_occ)


def listed():
    return [
        # a handful of vectors on the smallest grid: an outer solver that applies H
        # one small block at a time, where launches and latency are the cost
        {"name": "hpsi-24-fp64-x3", "kind": "hpsi", "system": "cube24", "n": 3, "precision": "fp64"},
        # a block of trial vectors of the benchmark system in FP32, an odd count
        {"name": "hpsi-48-mixed-x511", "kind": "hpsi", "system": "cube48", "n": 511, "precision": "mixed"},
        # H on the largest grid at full accuracy: residual checks of its states
        {"name": "hpsi-slab-fp64-x33", "kind": "hpsi", "system": "slab", "n": 33, "precision": "fp64"},
        # chi0 on one vector of the smallest system: a caller's own iteration
        # around chi0bar, one direction per step
        {"name": "chi0-24-mixed-x1", "kind": "chi0", "system": "cube24", "n": 1, "precision": "mixed"},
        # a block of directions on a middle-sized, many-state member of the batch
        {"name": "chi0-32-mixed-x16", "kind": "chi0", "system": "member5", "n": 16, "precision": "mixed"},
        # one Davidson block of the benchmark system: all 8192 right-hand sides
        {"name": "chi0-48-mixed-x128", "kind": "chi0", "system": "cube48", "n": 128, "precision": "mixed"},
        # the same operator at full precision on a few directions (reference checks)
        {"name": "chi0-48-fp64-x4", "kind": "chi0", "system": "cube48", "n": 4, "precision": "fp64"},
        # first-order states of a large cubic cell for a few applied potentials
        {"name": "stern-64-mixed-x3", "kind": "stern", "system": "member0", "n": 3, "precision": "mixed"},
        # the benchmark: 128 eigenpairs, 6 Davidson iterations, then W^p on probes
        {"name": "pdep-48-mixed", "kind": "pdep", "system": "cube48", "n": 64, "precision": "mixed",
         "n_pdep": 128, "iterations": 6},
        # the small parity system in FP64, Davidson to convergence
        {"name": "pdep-24-fp64", "kind": "pdep", "system": "cube24", "n": 5, "precision": "fp64",
         "n_pdep": 16, "iterations": 0},
        # W^p of the benchmark's eigenpairs on a few right-hand sides
        {"name": "screen-48-wp-x7", "kind": "screen", "system": "cube48", "n": 7, "precision": "fp64",
         "n_pdep": 128, "operator": "wp"},
        # imaginary-frequency response of a small basis (Lanczos chains)
        {"name": "imag-32-x12", "kind": "imag", "system": "member8", "n": 12, "precision": "fp64",
         "n_freq": 4, "steps": 40},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))


def draw(rng):
    kind = rng.choice(("hpsi", "hpsi", "chi0", "chi0", "chi0", "stern", "pdep", "screen", "imag"))
    members = ["member%d" % k for k in MEMBERS]
    if kind == "hpsi":
        case = {"kind": kind, "system": rng.choice(["cube24", "cube48", "slab"] + members),
                "n": _log_int(rng, 1, 400), "precision": rng.choice(("fp64", "mixed", "df64"))}
        if case["system"] == "slab":
            case["n"] = min(case["n"], 96)
    elif kind in ("chi0", "stern"):
        precision = rng.choice(("fp64", "mixed", "mixed"))
        name = rng.choice(["cube24", "cube48"] + members)
        # right-hand sides so that a call stays well below the benchmark's
        n_rhs = _log_int(rng, 1, 400 if precision == "fp64" else 3000)
        s = _system(name)
        most = rng.randint(8, 16) if kind == "stern" else rng.randint(48, 112)
        case = {"kind": kind, "system": name, "precision": precision,
                "n": max(1, min(most, n_rhs // s.n_occ))}
    elif kind == "pdep":
        name = rng.choice(("cube24", "member3", "member5", "member8", "member9", "member13", "member25"))
        case = {"kind": kind, "system": name, "n": _log_int(rng, 1, 64), "precision": "mixed",
                "n_pdep": _system(name).n_occ + rng.randint(0, 9), "iterations": rng.randint(2, 5)}
    elif kind == "screen":
        case = {"kind": kind, "system": rng.choice(["cube24", "cube48"] + members),
                "n": _log_int(rng, 1, 300), "precision": "fp64", "n_pdep": _log_int(rng, 8, 256),
                "operator": rng.choice(("wp", "chibar", "epsinv"))}
    else:
        case = {"kind": kind, "system": rng.choice(("cube24", "member2", "member8", "member9", "member13", "member14")),
                "n": rng.randint(2, 20), "precision": "fp64", "n_freq": rng.randint(1, 8),
                "steps": rng.randint(12, 48)}
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
_context = {"key": None, "ctx": None}


def _context_of(case):
    """The context of the case's system, kept while the same system is in use."""
    options = {}
    if case["kind"] == "pdep":
        options = {"dav_tol": 0.0 if case["iterations"] else 1e-8}
        if case["iterations"]:
            options["dav_max_iter"] = case["iterations"]
    precision = "mixed" if case["precision"] == "df64" else case["precision"]
    key = (case["system"], precision, case.get("n_pdep"), tuple(sorted(options.items())))
    if _context["key"] != key:
        _context.update(key=None, ctx=None)
        s = _system(case["system"])
        s = System(s.name, s.grid, s.cell, s.v_r, s.n_occ, case.get("n_pdep") or s.n_pdep)
        ctx = pg.Context(s, precision=PRECISIONS[precision], **options)
        _context.update(key=key, ctx=ctx)
    return _context["ctx"]


def _generator(seed):
    return torch.Generator(device=DEVICE).manual_seed(int(seed))


def _normal(gen, *shape):
    return torch.randn(*shape, dtype=torch.float64, device=DEVICE, generator=gen)


def _potentials(system, seed, n):
    """n smooth perturbing potentials (Ha): four signed periodic Gaussians each."""
    rng = np.random.default_rng(int(seed))
    dv = [_gaussian_sum(system.grid, system.cell, _wells(rng, 4, system.cell, (-1.0, 1.0), (1.0, 2.0)), 1.0).ravel()
          for _ in range(n)]
    return torch.tensor(np.stack(dv), device=DEVICE)


def _eigenpairs(gen, n_pdep, dim):
    """Orthonormal vectors and a decaying spectrum like that of chi0bar."""
    vec = torch.linalg.qr(_normal(gen, dim, n_pdep))[0].T.contiguous()
    u = torch.rand(n_pdep, dtype=torch.float64, device=DEVICE, generator=gen)
    val = -4.0 * torch.exp(-5.0 * torch.arange(n_pdep, dtype=torch.float64, device=DEVICE) / n_pdep) * (0.9 + 0.2 * u)
    return val, vec


def _phase(psi):
    """The sign of each state's largest coefficient (eigenvectors are defined up to it)."""
    return torch.sign(psi.gather(1, psi.abs().argmax(dim=1, keepdim=True)))[:, 0]


def _inputs(case, seed, n_pw, dim):
    """The seed's inputs, the same for run() and exact()."""
    gen, n = _generator(seed), case["n"]
    if case["kind"] == "hpsi":
        return {"x": _normal(gen, n, n_pw)}
    if case["kind"] == "chi0":
        return {"phi": _normal(gen, n, dim)}
    if case["kind"] == "stern":
        return {"dv": _potentials(_system(case["system"]), seed, n)}
    if case["kind"] == "pdep":
        return {"start": _normal(gen, case["n_pdep"], dim), "f": _normal(gen, n, dim)}
    if case["kind"] == "screen":
        val, vec = _eigenpairs(gen, min(case["n_pdep"], dim), dim)
        return {"val": val, "vec": vec, "f": _normal(gen, n, dim)}
    nu = torch.linspace(0.0, 2.0, case["n_freq"], dtype=torch.float64).numpy()
    return {"phi": torch.linalg.qr(_normal(gen, dim, n))[0].T.contiguous(), "nu": nu}


def prepare(case, seed):
    ctx = _context_of(case)
    size = ctx.sizes()
    state = {"case": case, "ctx": ctx, "size": size}
    state.update(_inputs(case, seed, size["n_pw"], size["n_pdep_dim"]))
    f64 = {"dtype": torch.float64, "device": DEVICE}
    if case["kind"] == "chi0":
        state["dn"] = torch.empty(case["n"], size["n_r"], **f64)
    elif case["kind"] == "stern":
        n_rhs = case["n"] * ctx.systems[0].n_occ
        state["dpsi"] = torch.empty(case["n"], ctx.systems[0].n_occ, size["n_pw"], **f64)
        state["iters"] = torch.empty(n_rhs, dtype=torch.int32, device=DEVICE)
        state["resid"] = torch.empty(n_rhs, **f64)
        psi = torch.tensor(ctx.occupied()[0], device=DEVICE)
        state["phase"] = _phase(psi)[:, None]
    elif case["kind"] == "pdep":
        state["val"] = torch.empty(case["n_pdep"], **f64)
        state["vec"] = torch.empty(case["n_pdep"], size["n_pdep_dim"], **f64)
    return state


def run(state):
    case, ctx = state["case"], state["ctx"]
    if case["kind"] == "hpsi":
        y = ctx.apply_hamiltonian(state["x"], precision=PRECISIONS[case["precision"]])
        # the FP32 transforms' result carries FP32 accuracy: kept as such
        return y.float() if case["precision"] == "mixed" else y
    if case["kind"] == "chi0":
        return {"chi0": ctx.chi0_apply(state["phi"], dn=state["dn"]), "dn": state["dn"]}
    if case["kind"] == "stern":
        # iteration counts and final residuals are diagnostics of the solver, not
        # results; the responses go with each state's largest coefficient positive
        ctx.sternheimer_solve(state["dv"], dpsi=state["dpsi"], iters=state["iters"], resid=state["resid"])
        return state["dpsi"].mul_(state["phase"])
    if case["kind"] == "pdep":
        # eigenvectors are defined up to their sign: what a program does with
        # them, the screened interaction on its probes, is what is returned
        ctx.pdep_solve(phi0=state["start"], eigvals=state["val"], eigvecs=state["vec"])
        wp = ctx.screening_apply("wp", state["val"], state["vec"], state["f"])
        # after a few mixed iterations the last kept eigenvectors carry the FP32
        # noise over the gap at the truncation (1e-9 between two runs): FP32 then
        return {"eigvals": state["val"], "wp": wp.float() if case["precision"] == "mixed" else wp}
    if case["kind"] == "screen":
        return ctx.screening_apply(case["operator"], state["val"], state["vec"], state["f"])
    b, lam = ctx.chi0_imag(state["phi"], state["nu"], n_steps=case["steps"])
    return {"b": b, "lambda": lam}


# ---------------------------------------------------------------------------
# the plane-wave sphere, the work of a pass, and the results in 64 bits
# ---------------------------------------------------------------------------
class Sphere:
    """Half-space sphere of the alias-free cut-off: members sorted by (n3, n2, n1)."""

    def __init__(self, grid, cell):
        self.grid, self.omega = grid, float(np.prod(cell))
        lim = [(n - 1) // 4 for n in grid]
        n1, n2, n3 = np.meshgrid(*[np.arange(-m, m + 1) for m in lim], indexing="ij")
        n = np.stack([n1.ravel(), n2.ravel(), n3.ravel()], axis=1)
        g = 2.0 * math.pi * n / np.asarray(cell)
        g2 = (g * g).sum(axis=1)
        gmax = min(2.0 * math.pi * ((m - 1) / 4.0) / l for m, l in zip(grid, cell))
        inside = 0.5 * g2 <= 0.5 * gmax * gmax
        self.n_col = len({(b, c) for _, b, c in n[inside]})
        self.n_planes = len({c for _, _, c in n[inside]})
        half = inside & ((n[:, 2] > 0) | ((n[:, 2] == 0) & ((n[:, 1] > 0) | ((n[:, 1] == 0) & (n[:, 0] > 0)))))
        order = np.lexsort((n[half, 0], n[half, 1], n[half, 2]))
        self.n, self.g2 = n[half][order], g2[half][order]
        self.n_pw = 2 * len(self.g2) + 1
        self.dim = self.n_pw - 1
        self.n_r = int(np.prod(grid))


@functools.lru_cache(maxsize=4)
def _sphere(name):
    s = _system(name)
    return Sphere(s.grid, s.cell)


#: H applications a Sternheimer solve to 1e-10 takes on these systems (CG
#: steps in FP64, or FP32 steps in the mixed mode plus the refinement)
STEPS = 35


def work(case):
    s, sp = _system(case["system"]), _sphere(case["system"])
    grid, n, nocc = s.grid, case["n"], s.n_occ

    def line(m):
        return 5.0 * m * math.log2(m)

    # sphere -> grid or back, of two real vectors packed in one complex field
    one_way = sp.n_col * line(grid[0]) + grid[0] * (sp.n_planes * line(grid[1]) + grid[1] * line(grid[2]))
    h = one_way + 2.0 * sp.n_r / 2  # H x of one vector: both ways for half a pair, and V
    n_pdep = case.get("n_pdep", 0)
    solve = STEPS * (h + 4.0 * nocc * sp.n_pw)  # CG steps of H and the projector
    chi0 = nocc * (solve + one_way + 4.0 * nocc * sp.n_pw)  # one perturbation
    if case["kind"] == "hpsi":
        return {"bytes": 16.0 * n * sp.n_pw + 8.0 * sp.n_r, "flops": n * h}
    fixed = 8.0 * (sp.n_r + nocc * sp.n_pw)  # the potential and the occupied states
    if case["kind"] == "chi0":
        return {"bytes": fixed + 8.0 * n * (2 * sp.dim + sp.n_r), "flops": n * chi0}
    if case["kind"] == "stern":
        return {"bytes": fixed + 8.0 * n * (sp.n_r + nocc * sp.n_pw), "flops": n * chi0}
    screen = 4.0 * n_pdep * sp.dim * n
    if case["kind"] == "pdep":
        blocks = case["iterations"] or 8
        return {"bytes": fixed + 8.0 * (2 * n_pdep + 2 * n) * sp.dim,
                "flops": blocks * n_pdep * chi0 + screen}
    if case["kind"] == "screen":
        return {"bytes": 8.0 * (n_pdep + 2 * n) * sp.dim, "flops": screen}
    steps = case["steps"]
    chains = n * nocc * (steps * (h + 4.0 * nocc * sp.n_pw) + 2.0 * n * steps * sp.n_pw)
    return {"bytes": fixed + 8.0 * (n * sp.dim + 2 * case["n_freq"] * n * n), "flops": chains}


class Exact:
    """Plain FFTs and dense algebra in 64 bits, the real-coefficient layout of the library."""

    def __init__(self, name):
        self.s, self.sp = _system(name), _sphere(name)
        self.n = torch.tensor(self.sp.n, device=DEVICE)
        self.g2 = torch.tensor(self.sp.g2, device=DEVICE)
        self.kin = torch.cat([(0.5 * self.g2).repeat_interleave(2), torch.zeros(1, dtype=torch.float64, device=DEVICE)])
        self.root = torch.sqrt(4.0 * math.pi / self.g2).repeat_interleave(2)  # v^{1/2}
        self.v = torch.tensor(self.s.v_r, device=DEVICE).reshape(1, -1)

    def chunks(self, n):
        step = max(1, (1 << 25) // self.sp.n_r)
        return [slice(i, min(n, i + step)) for i in range(0, n, step)]

    def to_grid(self, x):
        c = torch.complex(x[:, 0:-1:2], x[:, 1:-1:2]) / math.sqrt(2.0)
        f = torch.zeros((x.shape[0],) + tuple(self.sp.grid), dtype=torch.complex128, device=DEVICE)
        f[:, self.n[:, 0], self.n[:, 1], self.n[:, 2]] = c
        f[:, -self.n[:, 0], -self.n[:, 1], -self.n[:, 2]] = c.conj()
        f[:, 0, 0, 0] = x[:, -1].to(torch.complex128)
        return torch.fft.ifftn(f, dim=(1, 2, 3), norm="forward").real.reshape(x.shape[0], -1)

    def from_grid(self, u):
        f = torch.fft.fftn(u.reshape((-1,) + tuple(self.sp.grid)), dim=(1, 2, 3), norm="forward")
        c = f[:, self.n[:, 0], self.n[:, 1], self.n[:, 2]] * math.sqrt(2.0)
        x = torch.empty(u.shape[0], self.sp.n_pw, dtype=torch.float64, device=DEVICE)
        x[:, 0:-1:2], x[:, 1:-1:2], x[:, -1] = c.real, c.imag, f[:, 0, 0, 0].real
        return x

    def h(self, x):
        y = torch.empty_like(x)
        for c in self.chunks(x.shape[0]):
            y[c] = self.kin * x[c] + self.from_grid(self.v * self.to_grid(x[c]))
        return y

    def states(self):
        """All eigenpairs of H; the occupied states on the grid."""
        m = self.h(torch.eye(self.sp.n_pw, dtype=torch.float64, device=DEVICE))
        self.eps, self.c = torch.linalg.eigh(0.5 * (m + m.T))
        self.u = self.to_grid(self.c[:, :self.s.n_occ].T.contiguous())
        return self

    def dv(self, phi):
        zero = torch.zeros(phi.shape[0], 1, dtype=torch.float64, device=DEVICE)
        return self.to_grid(torch.cat([phi * self.root, zero], dim=1)) / math.sqrt(self.sp.omega)

    def overlaps(self, dv, v):
        """<c| dV |psi_v> over the empty states c, for every dV."""
        return self.from_grid(dv * self.u[v]) @ self.c[:, self.s.n_occ:]

    def dpsi(self, dv, v):
        return -(self.overlaps(dv, v) / (self.eps[self.s.n_occ:] - self.eps[v])) @ self.c[:, self.s.n_occ:].T

    def chi0(self, phi):
        out, dn = torch.empty_like(phi), torch.zeros(phi.shape[0], self.sp.n_r, dtype=torch.float64, device=DEVICE)
        for c in self.chunks(phi.shape[0]):
            dv = self.dv(phi[c])
            for v in range(self.s.n_occ):
                dn[c] += (4.0 / self.sp.omega) * self.u[v] * self.to_grid(self.dpsi(dv, v))
            out[c] = self.root * math.sqrt(self.sp.omega) * self.from_grid(dn[c])[:, :-1]
        return out, dn

    def screen(self, operator, val, vec, f):
        w = val / (1.0 - val)
        if operator == "wp":
            return self.root * (((f * self.root) @ vec.T * w) @ vec)
        out = (f @ vec.T * w) @ vec
        return out + f if operator == "epsinv" else out


def exact(case, seed):
    """The same results by plain FFTs, sums over all states and dense eigenpairs, in 64 bits."""
    sp = _sphere(case["system"])
    kind = case["kind"]
    if kind not in ("hpsi", "screen") and sp.n_pw > 2000:
        return None  # all states of these systems take too long
    if kind == "pdep" and (case["iterations"] or sp.n_pw > 1000):
        return None  # a fixed number of Davidson steps has no closed form
    e, i = Exact(case["system"]), _inputs(case, seed, sp.n_pw, sp.dim)
    if kind == "hpsi":
        return e.h(i["x"])
    if kind == "screen":
        return e.screen(case["operator"], i["val"], i["vec"], i["f"])
    e.states()
    if kind == "chi0":
        out, dn = e.chi0(i["phi"])
        return {"chi0": out, "dn": dn}
    if kind == "stern":
        phase = _phase(e.c[:, :e.s.n_occ].T)
        return torch.stack([phase[v] * e.dpsi(i["dv"], v) for v in range(e.s.n_occ)], dim=1)
    if kind == "pdep":
        m = e.chi0(torch.eye(sp.dim, dtype=torch.float64, device=DEVICE))[0]
        val, vec = torch.linalg.eigh(0.5 * (m + m.T))
        val, vec = val[:case["n_pdep"]], vec[:, :case["n_pdep"]].T
        return {"eigvals": val, "wp": e.screen("wp", val, vec, i["f"])}
    dv = e.dv(i["phi"])
    b = torch.zeros(case["n_freq"], case["n"], case["n"], dtype=torch.float64, device=DEVICE)
    for v in range(e.s.n_occ):
        q, d = e.overlaps(dv, v), e.eps[e.s.n_occ:] - e.eps[v]
        for f, nu in enumerate(i["nu"]):
            b[f] -= 4.0 * (q * (d / (d * d + float(nu) ** 2))) @ q.T
    one = torch.eye(case["n"], dtype=torch.float64, device=DEVICE)
    return {"b": b, "lambda": torch.linalg.solve(one - b, b)}
