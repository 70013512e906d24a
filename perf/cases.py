"""Performance cases of the multigrid library: what its users run, through the public entry points.

Every case is a dict of plain values.  `prepare` makes what a program holds before the call (a
solver handle, kept between calls as a time-stepping or parameter-sweep program keeps it, and the
right-hand side of this call), `run` is one call, `exact` the same result in plain float64 torch.
"""
import functools
import math

import numpy as np
import torch

from paper_1705_09282_gb300 import _lib, inputs, warmstart
from paper_1705_09282_gb300.solver import Solver, solve_batch

PRECISIONS = {"fp64": _lib.IGAMG_FP64, "fp32ir": _lib.IGAMG_FP32_IR, "fgmres": _lib.IGAMG_FGMRES_FP64}
SIGMAS = (1e-4, 1e-2, 1.0, 1e2, 1e4)          # the sigma / nu sweep of the square benchmark
BATCH_SIZES = ((64, 5), (96, 5), (128, 6))    # (elements, grids) of the independent-solves mix
RTOL = 1e-8


def _grid_case(kind, p, n, levels, sigma, nu=1.0, dim=2, beta=0.0, geometry="square", precision="fp64"):
    return {"kind": kind, "dim": dim, "p": p, "n": n, "levels": levels, "sigma": sigma, "nu": nu, "beta": beta,
            "geometry": geometry, "precision": precision}


def listed():
    return [
        # one V-cycle as a preconditioner on a small mesh: launches and latency
        dict(_grid_case("vcycle", 2, 16, 3, 1.0), name="vcycle-p2-16"),
        # the higher degree on a mesh that is not a power of two, reaction-dominated
        dict(_grid_case("vcycle", 3, 72, 4, 1e4), name="vcycle-p3-72"),
        # the headline solve: generalized Stokes on 256 x 256 elements, FP64, to 1e-8
        dict(_grid_case("solve", 2, 256, 7, 1.0), name="solve-p2-256"),
        # the same mesh at p = 3 in mixed precision (FP32 V-cycles in FP64 refinement)
        dict(_grid_case("solve", 3, 256, 7, 1e-2, precision="fp32ir"), name="solve-p3-256-mixed"),
        # the headline sweep: p = 2, 3 and five reaction / viscosity ratios, solved side by side
        {"kind": "sweep", "n": 256, "levels": 7, "name": "sweep-256"},
        # many independent solves of mixed sizes
        {"kind": "batch", "p": 2, "count": 48, "sizes": "mixed", "name": "batch-48"},
        # generalized Oseen on 512 x 512 elements: per-row operators streamed from memory
        dict(_grid_case("vcycle", 2, 512, 8, 1.0, nu=1e-2, beta=0.5), name="vcycle-oseen-512"),
        # mapped domain: quarter annulus, FGMRES around the V-cycle
        dict(_grid_case("solve", 2, 128, 6, 1.0, geometry="annulus", precision="fgmres"), name="annulus-128-fgmres"),
        # 3D generalized Stokes on 64^3 elements
        dict(_grid_case("vcycle", 2, 64, 5, 1.0, dim=3), name="cube-64"),
        # 3D generalized Oseen in mixed precision
        dict(_grid_case("solve", 2, 32, 4, 10.0, nu=1e-2, dim=3, beta=1.0, precision="fp32ir"), name="cube-oseen-32-mixed"),
        # the learned warm start: inference on the grids of sixteen 128 x 128 problems
        {"kind": "infer", "batch": 16, "size": 130, "name": "infer-16x130"},
        # and the loss and gradient of one training minibatch
        {"kind": "train", "batch": 8, "size": 66, "name": "train-8x66"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mesh(rng, lo, hi, coarsest=(4, 9)):
    """(n, levels) with lo <= n <= hi, n = m 2^(levels-1), m in the coarsest range."""
    while True:
        m, levels = rng.randint(*coarsest), rng.randint(2, 8)
        n = m << (levels - 1)
        if lo <= n <= hi and rng.random() < 0.5:
            return n, levels


def draw(rng):
    kind = rng.choice(["stokes", "stokes", "stokes", "solve", "mixed", "batch", "oseen", "annulus", "cube", "cube-oseen",
                       "infer", "train"])
    sigma = round(10 ** rng.uniform(-4, 4), 6)
    p = rng.choice([2, 3])
    if kind == "stokes":
        n, levels = _mesh(rng, 8, 448)
        return _grid_case("vcycle", p, n, levels, sigma)
    if kind in ("solve", "mixed"):
        n, levels = _mesh(rng, 16, 256)
        return _grid_case("solve", p, n, levels, sigma, precision="fp64" if kind == "solve" else "fp32ir")
    if kind == "batch":
        return {"kind": "batch", "p": p, "count": rng.randint(8, 36), "sizes": rng.choice(["mixed", "same"])}
    if kind == "oseen":
        n, levels = _mesh(rng, 16, 448)
        return _grid_case("vcycle", p, n, levels, 10.0, nu=1e-2, beta=round(rng.uniform(0.1, 0.5), 3))
    if kind == "annulus":
        n, levels = _mesh(rng, 16, 112)
        return _grid_case("solve", 2, n, levels, sigma, geometry="annulus", precision="fgmres")
    if kind == "cube":
        n, levels = _mesh(rng, 8, 48 if p == 2 else 12, (4, 5) if p == 2 else (4, 4))
        return _grid_case("vcycle", p, n, levels, sigma, dim=3)
    if kind == "cube-oseen":
        n, levels = _mesh(rng, 8, 24, (4, 5))
        return _grid_case("solve", 2, n, levels, round(rng.uniform(1.0, 20.0), 3), nu=0.1, dim=3, beta=1.0, precision="fp32ir")
    if kind == "infer":
        return {"kind": "infer", "batch": rng.randint(1, 24), "size": _log_int(rng, 18, 130)}
    return {"kind": "train", "batch": rng.randint(1, 12), "size": _log_int(rng, 18, 66)}


# ---- inputs ---------------------------------------------------------------------------------

def _field(gen, axes, features=64, length=0.1):
    """A smooth random field of unit variance and the given correlation length on the tensor
    product of `axes` (slowest first): random Fourier features, float64 on the host."""
    w = torch.randn(len(axes), features, generator=gen, dtype=torch.float64) / length
    phase = 2 * math.pi * torch.rand(features, generator=gen, dtype=torch.float64)
    out = torch.exp(1j * phase)
    for k, x in enumerate(axes):
        f = torch.exp(1j * w[k][:, None] * x[None, :])
        out = out.reshape(features, -1)[:, :, None] * f[:, None, :] if k + 1 < len(axes) else torch.einsum(
            "km,kx->mx", out.reshape(features, -1), f)
    return math.sqrt(2.0 / features) * out.real.reshape([len(x) for x in axes])


def _load(dim, p, n, seed):
    """A load vector (velocity blocks = a random field at the basis functions times their size,
    pressure and multiplier rows zero) in the library's layout, float64 on the host."""
    gen = torch.Generator().manual_seed(int(seed))
    ni, nq = n + p - 2, n + p - 1
    xi, xq = torch.linspace(0, 1, ni + 2, dtype=torch.float64)[1:-1], torch.linspace(0, 1, nq, dtype=torch.float64)
    blocks = []
    for c in range(dim):
        axes = [xi if a == c else xq for a in reversed(range(dim))]
        blocks.append(_field(gen, axes).reshape(-1) / float(n) ** dim)
    blocks.append(torch.zeros(nq ** dim + 1, dtype=torch.float64))
    return torch.cat(blocks)


def _weights(seed):
    """Network parameters as He initialisation gives them, with small biases (float32, flat)."""
    gen = torch.Generator().manual_seed(1000 + int(seed))
    parts = []
    for cout, cin in ((32, 3), (32, 32), (32, 32), (2, 32)):
        parts.append(torch.randn(cout * cin * 9, generator=gen) * math.sqrt(2.0 / (9 * cin)))
        parts.append(0.05 * torch.randn(cout, generator=gen))
    return torch.cat(parts)


def _images(case, seed, channels):
    """(batch, channels, size, size): smooth fields, the third channel log10(sigma / nu)."""
    gen = torch.Generator().manual_seed(int(seed))
    x = torch.linspace(0, 1, case["size"], dtype=torch.float64)
    out = torch.empty(case["batch"], channels, case["size"], case["size"])
    for b in range(case["batch"]):
        for c in range(channels):
            out[b, c] = _field(gen, [x, x]) if c < 2 else 6 * torch.rand((), generator=gen) - 2
    return out


# ---- handles --------------------------------------------------------------------------------

@functools.lru_cache(maxsize=24)
def _solver(slot, dim, p, n, levels, sigma, nu, beta, geometry, precision):
    """A handle and its pair of vectors, kept for all right-hand sides of one problem."""
    b = None
    if beta:
        b = inputs.oseen_advection(p, n, beta) if dim == 2 else inputs.oseen_advection_3d(p, n, beta)
    geo = _lib.IGAMG_GEOM_QUARTER_ANNULUS if geometry == "annulus" else _lib.IGAMG_GEOM_SQUARE
    s = Solver(p, n, levels, sigma, nu, precision=PRECISIONS[precision], beta=b, dim=dim, geometry=geo)
    return s, s.empty(), s.empty()


@functools.lru_cache(maxsize=4)
def _network(weights_seed):
    net = warmstart.Network()
    net.set_params(_weights(weights_seed).numpy())
    return net


@functools.lru_cache(maxsize=2)
def _group(case_items):
    """The handles of a group of independent solves, their vectors views of two buffers."""
    case = dict(case_items)
    if case["kind"] == "sweep":
        spec = [(p, case["n"], case["levels"], s) for p in (2, 3) for s in SIGMAS]
    else:
        rs = np.random.RandomState(7)
        spec = []
        for i in range(case["count"]):
            n, levels = BATCH_SIZES[i % 3 if case["sizes"] == "mixed" else 1]
            spec.append((case["p"], n, levels, float(10 ** rs.uniform(-2, 4))))
    solvers = [Solver(p, n, levels, s, 1.0) for p, n, levels, s in spec]
    sizes = [s.ndof() for s in solvers]
    u, f = (torch.zeros(sum(sizes), dtype=torch.float64, device="cuda") for _ in range(2))
    return spec, solvers, u, f, list(u.split(sizes)), list(f.split(sizes))


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("vcycle", "solve"):
        args = [case[k] for k in ("dim", "p", "n", "levels", "sigma", "nu", "beta", "geometry", "precision")]
        solver, u, f = _solver(0, *args)
        return {"kind": kind, "solver": solver, "U": u, "F": f, "load": _load(case["dim"], case["p"], case["n"], seed).cuda()}
    if kind in ("sweep", "batch"):
        spec, solvers, u, f, us, fs = _group(tuple(sorted((k, v) for k, v in case.items() if k != "name")))
        loads = torch.cat([_load(2, p, n, seed * 1000 + i) for i, (p, n, _, _) in enumerate(spec)]).cuda()
        return {"kind": kind, "solvers": solvers, "U": u, "F": f, "Us": us, "Fs": fs, "load": loads}
    net = _network(1)
    state = {"kind": kind, "net": net, "x": _images(case, seed, 3).cuda()}
    if kind == "train":
        state["target"] = _images(case, seed + 77, 2).cuda()
    return state


def run(state):
    kind = state["kind"]
    if kind == "vcycle":
        state["F"].copy_(state["load"])
        state["U"].zero_()
        return state["solver"].vcycle(state["U"], state["F"])
    if kind == "solve":
        state["F"].copy_(state["load"])
        state["U"].zero_()
        rep = state["solver"].solve(state["U"], state["F"], rtol=RTOL, max_cycles=100, history=False)
        return {"U": state["U"], "cycles": rep["cycles"], "converged": int(rep["converged"])}
    if kind in ("sweep", "batch"):
        state["F"].copy_(state["load"])
        state["U"].zero_()
        reps = solve_batch(state["solvers"], state["Us"], state["Fs"], rtol=RTOL, max_cycles=100)
        return {"U": state["U"], "cycles": [r["cycles"] for r in reps] if len(reps) <= 16 else sum(r["cycles"] for r in reps)}
    if kind == "infer":
        return state["net"].forward(state["x"])
    loss, grad = state["net"].loss_grad(state["x"], state["target"])
    return {"loss": loss, "grad": grad}


# ---- the work of one pass ---------------------------------------------------------------------

def _grid_work(dim, p, n, levels, records):
    """Bytes and flops of one V(2,2) cycle on a hierarchy: per level four sweeps and one residual
    (and one for the norm on the finest), vectors read and written once per level pass; per-row
    operators (records) read once per level."""
    q = p - 1
    row = (2 * p + 1) * (2 * q + 1) ** (dim - 1) + 2 * p * (2 * q + 1) ** (dim - 1) * (1 if dim == 2 else 1.25)
    byts = flops = 0.0
    for l in range(1, levels):
        m = n >> (levels - 1 - l)
        ni, nq = m + p - 2, m + p - 1
        rows = dim * ni * nq ** (dim - 1) + nq ** dim
        patches = ni ** 2 if dim == 2 else 3 * nq * ni ** 2
        flops += 4 * patches * (8 * 2 * row + 2 * 64) + 2 * rows * row
        byts += 8 * rows * (3 + (row + 8 if records else 0))
    return byts, flops


def _cycles(case):
    if case["kind"] == "vcycle":
        return 1
    if case["dim"] == 3:
        return 8
    return 6 if case["p"] == 3 else 16


def work(case):
    kind = case["kind"]
    if kind in ("vcycle", "solve"):
        b, f = _grid_work(case["dim"], case["p"], case["n"], case["levels"], case["beta"] > 0 or case["geometry"] != "square")
        return {"bytes": _cycles(case) * b, "flops": _cycles(case) * f}
    if kind in ("sweep", "batch"):
        if kind == "sweep":
            each = [(p, case["n"], case["levels"], 16 if p == 2 else 6) for p in (2, 3) for _ in SIGMAS]
        else:
            each = [(case["p"], *BATCH_SIZES[i % 3 if case["sizes"] == "mixed" else 1], 13 if case["p"] == 2 else 6)
                    for i in range(case["count"])]
        total = [(c * b, c * f) for p, n, levels, c in each for b, f in [_grid_work(2, p, n, levels, False)]]
        return {"bytes": sum(t[0] for t in total), "flops": sum(t[1] for t in total)}
    pix = case["batch"] * case["size"] ** 2
    macs = 9 * (3 * 32 + 2 * 32 * 32 + 32 * 2)
    if kind == "infer":
        return {"bytes": 4.0 * pix * 5, "flops": 2.0 * pix * macs}
    return {"bytes": 4.0 * pix * (5 + 3 * 32), "flops": 2.0 * pix * (3 * macs - 9 * 3 * 32)}


# ---- the same in plain float64 ----------------------------------------------------------------

def _basis(d, n, x, deriv=False):
    """Values (or derivatives) at x of the degree-d B-splines on n uniform elements, open knots."""
    t = np.concatenate([np.zeros(d), np.linspace(0, 1, n + 1), np.ones(d)])
    e = np.minimum((x * n).astype(int), n - 1)
    N = np.zeros((len(x), len(t) - 1))
    N[np.arange(len(x)), e + d] = 1.0
    for k in range(1, (d if not deriv else d - 1) + 1):
        a, b = t[k:-1] - t[:-k - 1], t[k + 1:] - t[1:-k]
        ia, ib = np.where(a > 0, 1 / np.where(a > 0, a, 1), 0), np.where(b > 0, 1 / np.where(b > 0, b, 1), 0)
        N = (x[:, None] - t[:-k - 1]) * ia * N[:, :-1] + (t[k + 1:] - x[:, None]) * ib * N[:, 1:]
    if not deriv:
        return N
    a, b = t[d:-1] - t[:-d - 1], t[d + 1:] - t[1:-d]
    ia, ib = np.where(a > 0, 1 / np.where(a > 0, a, 1), 0), np.where(b > 0, 1 / np.where(b > 0, b, 1), 0)
    return d * (ia * N[:, :-1] - ib * N[:, 1:])


def _refine(d, n):
    """Knot insertion: coefficients on 2n elements of the degree-d splines on n elements."""
    t = np.concatenate([np.zeros(d), np.linspace(0, 1, 2 * n + 1), np.ones(d)])
    g = np.array([t[i + 1:i + d + 1].mean() for i in range(2 * n + d)])
    T = np.linalg.solve(_basis(d, 2 * n, g), _basis(d, n, g))
    return np.where(np.abs(T) > 1e-12, T, 0.0)


class _Multigrid:
    """Algorithm 1 (V(2,2), multiplicative Schwarz over the supports of the potential's basis
    functions) for generalized Stokes on the unit square or cube, in float64 torch: operators as
    sums of Kronecker products of dense 1D matrices."""

    def __init__(self, dim, p, n, levels, sigma, nu):
        self.dim, self.p, self.dev = dim, p, "cuda" if torch.cuda.is_available() else "cpu"
        q = p - 1
        gx, gw = np.polynomial.legendre.leggauss(p + 2)
        x = (np.arange(n)[:, None] + 0.5 * (gx + 1)[None]).reshape(-1) / n
        w = np.tile(0.5 * gw / n, n)
        bp, dp, bq, dq = _basis(p, n, x), _basis(p, n, x, True), _basis(q, n, x), _basis(q, n, x, True)
        I = slice(1, n + p - 1)
        mp, sp = (bp.T * w @ bp)[I, I], (dp.T * w @ dp)[I, I]
        mq, sq = bq.T * w @ bq, dq.T * w @ dq
        wall = np.zeros_like(mq)
        ends = np.array([0.0, 1.0])
        v, dv = _basis(q, n, ends), _basis(q, n, ends, True)
        for k, s in enumerate((-1.0, 1.0)):
            wall += -s * (np.outer(v[k], dv[k]) + np.outer(dv[k], v[k])) + 4 * (p - 1) * n * np.outer(v[k], v[k])
        f = {"X1": sigma * mp + nu * sp, "X2": nu * mp, "Mq": mq, "Y2": sq + wall, "D": (dp.T * w @ bq)[I], "m": bq.T @ w}
        self.levels = [dict(f, n=n)]
        for _ in range(levels - 1):
            f = self.levels[0]
            m = f["n"] // 2
            Tp, Tq = _refine(p, m)[1:-1, 1:-1], _refine(q, m)
            f["Tp"], f["Tq"] = Tp, Tq
            self.levels.insert(0, {"n": m, "X1": Tp.T @ f["X1"] @ Tp, "X2": Tp.T @ f["X2"] @ Tp, "Mq": Tq.T @ f["Mq"] @ Tq,
                                   "Y2": Tq.T @ f["Y2"] @ Tq, "D": Tp.T @ f["D"] @ Tq, "m": Tq.T @ f["m"]})
        for l, f in enumerate(self.levels):
            if l:
                self._patches(f)
            for k, v in list(f.items()):
                if isinstance(v, np.ndarray):
                    f[k] = torch.tensor(v, device=self.dev)
        f = self.levels[0]
        N = sum(math.prod(s) for s in self._shapes(f["n"])) + 1
        eye = torch.eye(N, dtype=torch.float64, device=self.dev)
        self.K0 = torch.stack([self._apply(f, eye[i]) for i in range(N)], 1)

    def _shapes(self, n):
        ni, nq = n + self.p - 2, n + self.p - 1
        return [[ni if a == c else nq for a in reversed(range(self.dim))] for c in range(self.dim)] + [[nq] * self.dim]

    def _split(self, n, U):
        out, at = [], 0
        for s in self._shapes(n):
            k = math.prod(s)
            out.append(U[at:at + k].reshape(s))
            at += k
        return out, U[-1]

    def _along(self, M, T, a):
        k = self.dim - 1 - a
        return torch.movedim(torch.tensordot(M, T, ([1], [k])), 0, k)

    def _kron(self, T, mats):
        for a, M in enumerate(mats):
            T = self._along(M, T, a)
        return T

    def _apply(self, f, U):
        (*u, pr), lam = self._split(f["n"], U)
        d, out, div = self.dim, [], 0.0
        for c in range(d):
            mats = [f["X1"] if a == c else f["Mq"] for a in range(d)]
            r = self._kron(u[c], mats)
            for b in range(d):
                if b != c:
                    r = r + self._kron(u[c], [f["X2"] if a == c else f["Y2"] if a == b else f["Mq"] for a in range(d)])
            r = r - self._kron(pr, [f["D"] if a == c else f["Mq"] for a in range(d)])
            out.append(r.reshape(-1))
            div = div + self._kron(u[c], [f["D"].T if a == c else f["Mq"] for a in range(d)])
        m = f["m"]
        mean = m
        for _ in range(d - 1):
            mean = mean[..., None] * m
        out.append((div + lam * mean).reshape(-1))
        out.append((mean * pr).sum().reshape(1))
        return torch.cat(out)

    def _patches(self, f):
        """Per colour: degree-of-freedom lists (padded with the last, spare entry) and inverses."""
        d, p, n = self.dim, self.p, f["n"]
        q, ni, nq, T = p - 1, n + p - 2, n + p - 1, 2 * p + 1
        shapes = self._shapes(n)
        base = np.concatenate([[0], np.cumsum([math.prod(s) for s in shapes])])
        spare = int(base[-1]) + 1
        deg = lambda c, a: p if a == c else q                               # noqa: E731

        @functools.lru_cache(maxsize=None)
        def local(dpsi, i, dd):                                             # supports inside [i - dpsi, i]
            lo, hi = max(i - dpsi, 0), min(i, n - 1)
            r = range(1, ni + 1) if dd == p else range(nq)
            return np.array([j for j in r if max(j - dd, 0) >= lo and min(j, n - 1) <= hi], dtype=np.int64)

        families = [tuple([p] * d)] if d == 2 else [tuple(q if a == c else p for a in range(d)) for c in range(d)]
        colours, inverses = {}, {}
        for fam, dpsi in enumerate(families):
            stride = [p + 1 if dpsi[a] == p else p for a in range(d)]
            ranges = [range(1, ni + 1) if dpsi[a] == p else range(nq) for a in range(d)]
            cls = [[i if i < T else (ranges[a][-1] - i - T if ranges[a][-1] - i < T else T) for i in ranges[a]] for a in range(d)]
            groups = {}
            for a in range(d):
                byc = {}
                for i, c in zip(ranges[a], cls[a]):
                    byc.setdefault((c, i % stride[a]), []).append(i)
                groups[a] = byc
            combos = [()]
            for a in range(d):
                combos = [x + ((k, v),) for x in combos for k, v in groups[a].items()]
            for combo in combos:
                rep = [v[0] for _, v in combo]
                sets = [[local(dpsi[a], rep[a], deg(c, a)) for a in range(d)] for c in range(d + 1)]
                # the representative's degrees of freedom; the others' move with their patch
                idx, coords = [], []
                for c in range(d + 1):
                    grid = np.meshgrid(*[sets[c][a] for a in reversed(range(d))], indexing="ij")
                    coords.append([g.reshape(-1) for g in reversed(grid)])    # per axis a
                key = (fam,) + tuple(k[0] for k, _ in combo)
                if key not in inverses:
                    nv, npr = sum(len(coords[c][0]) for c in range(d)), len(coords[d][0])
                    K = np.zeros((nv + npr + 1, nv + npr + 1))
                    at = 0
                    sub = lambda M, i, j: M[np.ix_(i, j)]                     # noqa: E731
                    for c in range(d):
                        co = [x - 1 if a == c else x for a, x in enumerate(coords[c])]
                        k = len(co[0])
                        blk = np.ones((k, k))
                        for a in range(d):
                            blk = blk * sub(f["X1"] if a == c else f["Mq"], co[a], co[a])
                        for b in range(d):
                            if b != c:
                                t = np.ones((k, k))
                                for a in range(d):
                                    t = t * sub(f["X2"] if a == c else f["Y2"] if a == b else f["Mq"], co[a], co[a])
                                blk = blk + t
                        B = np.ones((k, npr))
                        for a in range(d):
                            B = B * sub(f["D"] if a == c else f["Mq"], co[a], coords[d][a])
                        K[at:at + k, at:at + k] = blk
                        K[at:at + k, nv:nv + npr] = -B
                        K[nv:nv + npr, at:at + k] = B.T
                        at += k
                    m = np.ones(npr)
                    for a in range(d):
                        m = m * f["m"][coords[d][a]]
                    K[nv:nv + npr, -1] = m
                    K[-1, nv:nv + npr] = m
                    inverses[key] = np.linalg.inv(K)[:-1, :-1]
                shift = np.meshgrid(*[np.array(combo[a][1]) - rep[a] for a in reversed(range(d))], indexing="ij")
                shift = [s.reshape(-1) for s in reversed(shift)]
                for c in range(d + 1):
                    s = shapes[c]
                    g = np.zeros((len(shift[0]), len(coords[c][0])), dtype=np.int64)
                    for a in reversed(range(d)):
                        pos = coords[c][a][None] + shift[a][:, None] - (1 if a == c else 0)
                        g = g * s[d - 1 - a] + pos
                    idx.append(g + base[c])
                idx = np.concatenate(idx, 1)
                col = 0
                for a in reversed(range(d)):
                    col = col * stride[a] + combo[a][0][1]
                colours.setdefault((fam, col), []).append((idx, key))
        f["colours"] = []
        for c in sorted(colours):
            steps = []
            for small in (True, False):
                part = [(i, k) for i, k in colours[c] if (i.shape[1] == 8) == small]
                if not part:
                    continue
                width = max(i.shape[1] for i, _ in part)
                table = np.zeros((len(part), width, width))
                rows, cls = [], []
                for j, (i, k) in enumerate(part):
                    m = i.shape[1]
                    table[j, :m, :m] = inverses[k]
                    rows.append(np.concatenate([i, np.full((len(i), width - m), spare)], 1))
                    cls.append(np.full(len(i), j))
                steps.append((torch.tensor(np.concatenate(rows), device=self.dev),
                              torch.tensor(np.concatenate(cls), device=self.dev), torch.tensor(table, device=self.dev)))
            f["colours"].append(steps)

    def _smooth(self, f, U, F, sweeps):
        zero = torch.zeros(1, dtype=torch.float64, device=self.dev)
        for _ in range(sweeps):
            for steps in f["colours"]:
                r = torch.cat([F - self._apply(f, U), zero])
                V = torch.cat([U, zero])
                for idx, cls, inv in steps:
                    V[idx] += torch.bmm(inv[cls], r[idx][..., None])[..., 0]
                U = V[:-1]
        return U

    def cycle(self, l, U, F):
        f = self.levels[l]
        if l == 0:
            return torch.linalg.solve(self.K0, F)
        U = self._smooth(f, U, F, 2)
        (*r, rp), lam = self._split(f["n"], F - self._apply(f, U))
        G = [self._kron(b, [(f["Tp"] if a == c else f["Tq"]).T.contiguous() for a in range(self.dim)]).reshape(-1)
             for c, b in enumerate(r + [rp])]
        E = self.cycle(l - 1, torch.zeros_like(torch.cat(G + [lam.reshape(1)])), torch.cat(G + [lam.reshape(1)]))
        (*e, ep), lam = self._split(self.levels[l - 1]["n"], E)
        U = U + torch.cat([self._kron(b, [f["Tp"] if a == c else f["Tq"] for a in range(self.dim)]).reshape(-1)
                           for c, b in enumerate(e + [ep])] + [lam.reshape(1)])
        return self._smooth(f, U, F, 2)

    def solve(self, F, rtol, cycles):
        U = torch.zeros_like(F)
        f, r0, k = self.levels[-1], float(F.norm()), 0
        while k < cycles:
            U = self.cycle(len(self.levels) - 1, U, F)
            k += 1
            if float((F - self._apply(f, U)).norm()) <= rtol * r0:
                break
        return U, k


def _network_exact(x, weights):
    """The network's output in float64 with its weights rounded to bfloat16 as it holds them."""
    at = 0
    for layer, (cout, cin, dil) in enumerate(((32, 3, 1), (32, 32, 2), (32, 32, 4), (2, 32, 8))):
        w = weights[at:at + cout * cin * 9].reshape(cout, cin, 3, 3)
        b = weights[at + w.numel():at + w.numel() + cout]
        at += w.numel() + cout
        w = w + (w.detach().float().bfloat16().double() - w.detach())
        y = b[None, :, None, None]
        for i in range(3):
            for j in range(3):
                s = torch.nn.functional.pad(x, (dil,) * 4)[:, :, i * dil:i * dil + x.shape[2], j * dil:j * dil + x.shape[3]]
                y = y + torch.einsum("oc,bchw->bohw", w[:, :, i, j], s)
        x = 0.5 * y * (1 + torch.erf(y / math.sqrt(2.0))) if layer < 3 else y
    return x


def exact(case, seed):
    kind, dev = case["kind"], "cuda" if torch.cuda.is_available() else "cpu"
    if kind in ("vcycle", "solve"):
        if case["beta"] or case["geometry"] != "square" or case["precision"] != "fp64" or (case["dim"] == 3 and case["n"] > 64):
            return None
        if kind == "solve" and case["p"] == 3 and case["n"] > 192:
            return None
        mg = _Multigrid(case["dim"], case["p"], case["n"], case["levels"], case["sigma"], case["nu"])
        F = _load(case["dim"], case["p"], case["n"], seed).to(mg.dev)
        if kind == "vcycle":
            return mg.cycle(case["levels"] - 1, torch.zeros_like(F), F)
        U, k = mg.solve(F, RTOL, 100)
        return {"U": U, "cycles": k, "converged": 1}
    if kind in ("sweep", "batch"):
        return None
    w = _weights(1).double().to(dev)
    x = _images(case, seed, 3).double().to(dev)
    if kind == "infer":
        return _network_exact(x, w)
    w.requires_grad_(True)
    d = _network_exact(x, w) - _images(case, seed + 77, 2).double().to(dev)
    loss = d[:, 0, 1:-1, 1:-1].square().mean() + d[:, 1, :-1, :-1].square().mean()
    loss.backward()
    return {"loss": loss.detach(), "grad": w.grad}
