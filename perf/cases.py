"""Cases for measuring the solver's speed: what its users call, over the sizes they call it with.

A program holds one solver per (model, frequency): it creates it, factors the layers once, and then
solves for shots that keep arriving.  So a case prepares a factored solver and the shots' volume
sources, and one pass is one call with them.  Media, PML thicknesses, layer counts and column
counts are those of this repository's workloads, or lie between them.
"""
import math

import numpy as np
import torch

from paper_1801_08655_gb300 import hz
from paper_1801_08655_gb300 import workloads as W

# Tolerances that callers use: the benchmark's (five digits), its stricter setting, and the close ones of a caller that
# wants all digits the volume residual can certify in mixed precision, or GMRES in FP64.
TOLERANCES = {"five_digits": dict(gmres_tol=1e-4, refine_tol=1e-5),
              "six_digits": dict(gmres_tol=1e-5, refine_tol=1e-6),
              "close": dict(gmres_tol=1e-7, refine_tol=1e-10, max_refine=5),
              "fp64": dict(gmres_tol=1e-10)}


def solve_case(name, nx, ny, nz, npml, layers, rhs, precision="mixed", tol="five_digits", medium="smooth",
               density=False, krylov=0, blocks=0, ppw=10.0, refactor=False):
    case = dict(name=name, kind="solve", nx=nx, ny=ny, nz=nz, npml=npml, layers=layers, rhs=rhs,
                precision=precision, tol=tol, medium=medium, density=density, krylov=krylov, blocks=blocks, ppw=ppw,
                refactor=refactor)
    if name is None:
        del case["name"]
    return case


def listed():
    return [
        # one point source on the smallest grid: launches and latency
        solve_case("point_24", 24, 24, 24, 5, 2, 1, tol="close", medium="bump", ppw=8.0),
        # the FP64 path, few shots
        solve_case("fp64_40", 40, 40, 40, 8, 4, 4, precision="fp64", tol="fp64"),
        # a few shots on a small grid
        solve_case("shots_48", 48, 48, 48, 8, 6, 4, tol="close"),
        # odd box, odd column count, variable density
        solve_case("ragged_density", 67, 51, 59, 8, 5, 13, tol="close", density=True),
        # the 64^3 workload: one gather of 16 shots
        solve_case("survey_64", 64, 64, 64, 8, 8, 16),
        # the same grid with all shots at once
        solve_case("wide_64", 64, 64, 64, 8, 8, 128),
        # the widest member of the batched workload
        solve_case("wide_80", 80, 80, 80, 8, 10, 64),
        # the 128^3 workload in the serving loop's batches of 32 columns
        solve_case("large_128", 128, 128, 128, 10, 16, 32, medium="layered", ppw=8.0),
        # explicit trace-to-trace blocks: small grid, few shots, many solves
        solve_case("blocks_48", 48, 48, 48, 8, 6, 8, tol="six_digits", blocks=32),
        # a new factorization, and the first shot with it
        solve_case("factor_64", 64, 64, 64, 8, 8, 1, tol="close", refactor=True),
        # the FP64 volume residual that certifies a solution, on the largest grid
        dict(name="residual_128", kind="residual", nx=128, ny=128, nz=128, npml=10, layers=16, rhs=16, ppw=8.0),
        # problems of different sizes solved at once
        dict(name="group_40_48_64", kind="group", members="40:4:1,48:6:4,64:8:16", npml=8, ppw=10.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: boxes of 22 to 96 cells a side, of unequal sides, 1 to 128 columns."""
    kind = rng.choice(["solve"] * 8 + ["factor", "residual"])
    if kind == "residual":
        n = _log_int(rng, 24, 128)
        return dict(kind=kind, nx=n + rng.randint(-2, 2), ny=n, nz=n + rng.randint(-2, 2), npml=rng.choice([5, 8]),
                    layers=2, rhs=min(_log_int(rng, 1, 128), max(1, (1 << 25) // n ** 3)), ppw=10.0)
    n = _log_int(rng, 24, 96)
    nx, ny, nz = (max(22, n + rng.randint(-n // 8, n // 8)) for _ in range(3))
    npml = 5 if n < 40 else 8
    layers = max(2, (nz - 2 * npml) // rng.choice([6, 7, 8]))
    if kind == "factor":
        return solve_case(None, nx, ny, nz, npml, layers, rng.randint(1, 4), tol="close", refactor=True)
    rhs = min(_log_int(rng, 1, 128), max(1, (1 << 25) // (nx * ny * nz)))
    option = rng.choice(["plain"] * 6 + ["density", "density", "bicgstab", "fp64", "blocks"])
    if option == "fp64" and nx * ny * nz * rhs <= 1 << 19:
        return solve_case(None, nx, ny, nz, npml, layers, rhs, precision="fp64", tol="fp64")
    blocks = 32 if option == "blocks" and nx * ny <= 3000 and rhs <= 32 else 0
    tol = rng.choice(["six_digits", "close"]) if n >= 40 and rhs >= 4 else "close"
    return solve_case(None, nx, ny, nz, npml, layers, rhs, tol=tol,
                      density=option == "density", krylov=int(option == "bicgstab"), blocks=blocks,
                      ppw=float(rng.choice([8, 9, 10, 11, 12])))


# ---------------------------------------------------------------------------------------------- inputs

def _model(case, seed):
    """m, b (or None), omega, C: host arrays and numbers, as a user reads a model from a file."""
    nx, ny, nz, npml = case["nx"], case["ny"], case["nz"], case["npml"]
    n = max(nx, ny, nz)
    b = None
    if case.get("medium", "smooth") == "bump":
        amp = 0.25 + 0.1 * np.random.default_rng(seed).random()
        return W.medium_gaussian_bump(n, amp=amp), None, W.omega_for_ppw(1.0, case["ppw"]), W.pml_constant(1.0)
    if case.get("medium") == "layered":
        c_block = 4.2 + 0.3 * np.random.default_rng(seed).random()
        m = W.medium_layered_block(n, npml, c_block=c_block)
    elif case["kind"] == "residual":
        c = 1.5 + 3.0 * np.random.default_rng(seed).random((nz, ny, nx))
        m = 1.0 / (c * c)
    else:
        m = np.ascontiguousarray(W.medium_smooth_random(n, seed=seed)[:nz, :ny, :nx])
    if case.get("density"):
        b = np.ascontiguousarray(W.density_smooth_random(n, seed=seed + 1)[:nz, :ny, :nx])
    return m, b, W.omega_for_ppw(1.5, case["ppw"]), W.pml_constant(4.5)


def _shots(case, seed):
    """Unit point sources, one per column, at distinct places of a plane near the surface."""
    nx, ny, nz, p, R = case["nx"], case["ny"], case["nz"], case["npml"], case["rhs"]
    rng = np.random.default_rng(seed + 7)
    px, py = nx - 2 * p, ny - 2 * p
    at = rng.choice(px * py, size=R, replace=px * py < R)
    z = nz // 2 if case["medium"] == "bump" else p + 2
    f = torch.zeros((R, nz, ny, nx), dtype=torch.complex128, device="cuda")
    f[torch.arange(R), z, torch.from_numpy(p + at // px), torch.from_numpy(p + at % px)] = 1.0
    return f


def _random(shape, seed):
    g = torch.Generator(device="cuda").manual_seed(seed + 13)
    return torch.randn(shape, dtype=torch.complex128, device="cuda", generator=g)


def _members(case):
    out = []
    for i, member in enumerate(case["members"].split(",")):
        n, layers, rhs = (int(v) for v in member.split(":"))
        out.append(solve_case("member%d" % i, n, n, n, case["npml"], layers, rhs, tol="close", ppw=case["ppw"]))
    return out


def _options(case):
    o = hz.default_opts(case["precision"])
    for k, v in TOLERANCES[case["tol"]].items():
        setattr(o, k, v)
    o.krylov = case["krylov"]
    return o


def _solver(case, seed, stream=None, factor=True):
    m, b, omega, C = _model(case, seed)
    s = hz.Solver(m, omega, case["npml"], C, case["layers"], precision=case.get("precision", "mixed"), b=b,
                  stream=stream)
    if factor:
        s.factor()
    if case.get("blocks"):
        s.trace_blocks(case["blocks"])
    return s


def prepare(case, seed):
    kind = case["kind"]
    if kind == "group":   # every member on a stream of its own, as hz_solve_group wants it
        parts = _members(case)
        solvers = [_solver(c, seed + 100 * i, stream=torch.cuda.Stream()) for i, c in enumerate(parts)]
        return dict(kind=kind, solvers=solvers, rhs=[_shots(c, seed + 100 * i) for i, c in enumerate(parts)],
                    opts=_options(parts[0]))
    if kind == "residual":
        shape = (case["rhs"], case["nz"], case["ny"], case["nx"])
        s = _solver(case, seed, factor=False)
        return dict(kind=kind, solver=s, rhs=_random(shape, seed), u=_random(shape, seed + 1))
    f = _shots(case, seed)
    return dict(kind=kind, solver=_solver(case, seed), rhs=f, opts=_options(case),
                u=torch.empty_like(f), single=case["tol"].endswith("digits"), refactor=case["refactor"])


def run(state):
    kind = state["kind"]
    if kind == "group":
        return hz.solve_group(state["solvers"], state["rhs"], state["opts"])[0]
    s = state["solver"]
    if kind == "residual":
        rel, r = s.volume_residual(state["rhs"], state["u"], want_r=True)
        return rel, r
    if state["refactor"]:
        s.factor()
    u, _, _ = s.solve(state["rhs"], state["opts"], u=state["u"])
    # wavefields solved to five or six digits are kept in single precision
    return u.to(torch.complex64) if state["single"] else u


# ---------------------------------------------------------------------------------------------- work

def _entries(nx, ny, nz):
    """Stored factor entries of one box: triangular L11 and rectangular L21 of every tree node."""
    s = hz.symbolic_shape(nx, ny, nz)
    o = s["nown"].astype(np.float64)
    u = np.diff(np.append(s["upd_off"], len(s["upd_idx"]))).astype(np.float64)
    return float((o * (o + 1) / 2 + o * u).sum()), float(8 * (o ** 3 / 3 + u * o * o / 2 + u * u * o / 2).sum())


def _layers(case):
    """(owned lo, hi, local zlo, zhi) of every layer."""
    nz, p, L = case["nz"], case["npml"], case["layers"]
    q, r = divmod(nz - 2 * p, L)
    out, start = [], p
    for ell in range(L):
        lo, hi = start, start + q + (ell < r) - 1
        start = hi + 1
        lo, hi = (0 if ell == 0 else lo), (nz - 1 if ell == L - 1 else hi)
        out.append((lo, hi, lo - p if ell else lo, hi + p if ell < L - 1 else hi))
    return out


def work(case):
    """Bytes: the inputs, the factors and the outputs once.  Flops of a solve: one product with every
    factor entry forward and one backward per local-solve column, for the right-hand side, the
    reconstruction and ITERATIONS applications of P M_pol (four source blocks, three sweeps), and the
    factorization where the pass has one."""
    ITERATIONS = 4
    if case["kind"] == "group":
        parts = [work(c) for c in _members(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    n3, R = case["nx"] * case["ny"] * case["nz"], case["rhs"]
    if case["kind"] == "residual":   # 7-point complex stencil: 7 products and 6 sums, the scaling, two norms
        return {"bytes": 48.0 * n3 * R, "flops": (7 * 6 + 6 * 2 + 6 + 2 + 8) * float(n3) * R}
    shapes = {}
    entries, factor_flops = 0.0, 0.0
    for lo, hi, zlo, zhi in _layers(case):
        k = zhi - zlo + 1
        if k not in shapes:
            shapes[k] = _entries(case["nx"], case["ny"], k)
        entries += shapes[k][0]
        factor_flops += shapes[k][1]
    cell = 16.0 if case.get("precision") == "fp64" else 8.0
    return {"bytes": 32.0 * n3 * R + cell * entries,
            "flops": 16.0 * entries * R * (2 + 7 * ITERATIONS) + (factor_flops if case["refactor"] else 0.0)}


# ---------------------------------------------------------------------------------------------- exact

def _sigma(z, n, p, C):
    d = np.maximum(np.maximum(p - z, z - (n - 1 - p)), 0.0)
    return (C / p) * (d / p) ** 2


def _profile(n, p, C, omega):
    x = np.arange(n, dtype=np.float64)
    return 1 + 1j * _sigma(x, n, p, C) / omega, 1 + 1j * _sigma(np.arange(n + 1) - 0.5, n, p, C) / omega


def _half(b, axis):
    ext = np.concatenate([np.take(b, [0], axis), b, np.take(b, [-1], axis)], axis)
    n = b.shape[axis]
    return 0.5 * (np.take(ext, np.arange(n + 1), axis) + np.take(ext, np.arange(1, n + 2), axis))


class _Operator:
    """The stretched 7-point operator of one box in 64 bits: `lo[a]`, `hi[a]` couple a cell with its
    neighbours along axis a (z, y, x), `diag` with itself."""

    def __init__(self, m, b, omega, profiles):
        (szn, szh), (syn, syh), (sxn, sxh) = profiles
        sz, sy, sx = szn[:, None, None], syn[None, :, None], sxn[None, None, :]
        halves = [sy * sx / szh[:, None, None], sz * sx / syh[None, :, None], sz * sy / sxh[None, None, :]]
        if b is not None:
            halves = [h * _half(b, a) for a, h in enumerate(halves)]
        lo = [np.take(h, np.arange(m.shape[a]), a) for a, h in enumerate(halves)]
        hi = [np.take(h, np.arange(1, m.shape[a] + 1), a) for a, h in enumerate(halves)]
        dev = lambda v: torch.from_numpy(np.array(np.broadcast_to(v, m.shape))).cuda()  # noqa: E731
        self.S = dev(sz * sy * sx)
        self.lo, self.hi = [dev(v) for v in lo], [dev(v) for v in hi]
        self.diag = dev(omega * omega * m) * self.S - sum(self.lo) - sum(self.hi)

    def __call__(self, u):
        out = self.diag * u
        for a in range(3):
            n = u.shape[a + 1]
            if n > 1:
                first, last = [slice(None)] * 4, [slice(None)] * 4
                first[a + 1], last[a + 1] = slice(0, n - 1), slice(1, n)
                first, last = tuple(first), tuple(last)
                out[last] += self.lo[a][last[1:]] * u[first]
                out[first] += self.hi[a][first[1:]] * u[last]
        return out

    def solve(self, g):
        """Block elimination plane by plane in single precision, refined with 64-bit residuals."""
        nz, ny, nx = self.diag.shape
        P = ny * nx
        cells = torch.arange(P, device="cuda").reshape(ny, nx)
        inv = []
        for k in range(nz):
            A = torch.zeros((P, P), dtype=torch.complex64, device="cuda")
            A[cells.ravel(), cells.ravel()] = self.diag[k].ravel().to(torch.complex64)
            for a, first, last in ((1, cells[:-1], cells[1:]), (2, cells[:, :-1], cells[:, 1:])):
                lo = self.lo[a][k][1:] if a == 1 else self.lo[a][k][:, 1:]
                hi = self.hi[a][k][:-1] if a == 1 else self.hi[a][k][:, :-1]
                A[last.ravel(), first.ravel()] = lo.ravel().to(torch.complex64)
                A[first.ravel(), last.ravel()] = hi.ravel().to(torch.complex64)
            if k:
                low, up = self.lo[0][k].ravel().to(torch.complex64), self.hi[0][k - 1].ravel().to(torch.complex64)
                A -= low[:, None] * inv[-1] * up[None, :]
            inv.append(torch.linalg.inv(A))

        def approximate(r):
            r = r.reshape(r.shape[0], nz, P)
            scale = r.abs().amax(dim=(1, 2)).clamp_min(1e-300)
            r = (r / scale[:, None, None]).to(torch.complex64)
            y = [r[:, 0]]
            for k in range(1, nz):
                y.append(r[:, k] - (y[-1] @ inv[k - 1].T) * self.lo[0][k].ravel().to(torch.complex64))
            x = [None] * nz
            x[-1] = y[-1] @ inv[-1].T
            for k in range(nz - 2, -1, -1):
                x[k] = (y[k] - x[k + 1] * self.hi[0][k].ravel().to(torch.complex64)) @ inv[k].T
            return torch.stack(x, 1).to(torch.complex128).reshape(-1, nz, ny, nx) * scale[:, None, None, None]

        u, norm = approximate(g), float(g.norm())
        for _ in range(20):
            r = g - self(u)
            if float(r.norm()) <= 1e-14 * norm:
                break
            u = u + approximate(r)
        return u


def exact(case, seed):
    """The global problem's direct solution (the layers are only a way to it), by block elimination."""
    if case["kind"] == "group":
        return [exact(c, seed + 100 * i) for i, c in enumerate(_members(case))]
    nx, ny, nz, p = case["nx"], case["ny"], case["nz"], case["npml"]
    m, b, omega, C = _model(case, seed)
    px, py, pz = (_profile(n, p, C, omega) for n in (nx, ny, nz))
    if case["kind"] == "residual":
        shape = (case["rhs"], nz, ny, nx)
        op = _Operator(m, b, omega, (pz, py, px))
        g = op.S * _random(shape, seed)
        r = g - op(_random(shape, seed + 1))
        rel = torch.linalg.vector_norm(r, dim=(1, 2, 3)) / torch.linalg.vector_norm(g, dim=(1, 2, 3))
        return [float(v) for v in rel], r
    if float(nx * ny) ** 3 * nz > 6e12:
        return None
    op = _Operator(m, b, omega, (pz, py, px))
    return op.solve(op.S * _shots(case, seed))
