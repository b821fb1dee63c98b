"""Performance cases of the GB300 three-grid IOFD Helmholtz library.

Each case is one call a program makes on a resident handle: a stencil
application, a Jacobi map, a residual, one preconditioner application
(Algorithm 1, forward or adjoint), a solve or a gradient.  The sizes are those
of ``hz_workloads.py``, ``bench.py`` and the tests, and cuboids in between.

A case is a dict:
  kind    apply | jacobi | resid | precond | solve | grad
  nx, ny, nz   intervals of the fine grid, PML included (nodes are one more, so
          every row is odd)
  pml     PML layers per side of the fine grid
  medium  homogeneous | lens | layers | random
  level   0, 1, 2: grid of spacing h, 2h, 4h (single-level kinds)
  op      A | B | Q | A_ADJ | B_ADJ (single-level kinds)
  prec    c64 | c128
  nrhs    right-hand sides in the call (sources for solve and grad)
"""
import math
import os

import numpy as np
import torch

import paper_2608_22946_gb300 as hz

GAMMA_MAX = 1.119058
PPW = 6.0
OMEGA_J = (0.8, 0.8, 0.2)     # Jacobi weights of the three levels
SIGMA = 0.9                   # complex shift of B
OPS = {"A": hz.HZ_OP_A, "B": hz.HZ_OP_B, "Q": hz.HZ_OP_Q, "A_ADJ": hz.HZ_OP_A_ADJ, "B_ADJ": hz.HZ_OP_B_ADJ}


def _case(name, kind, n, pml, medium, level=0, op="A", prec="c64", nrhs=1):
    c = {"kind": kind, "nx": int(n[0]), "ny": int(n[1]), "nz": int(n[2]), "pml": pml, "medium": medium, "level": level, "op": op,
         "prec": prec, "nrhs": nrhs}
    if name:
        c["name"] = name
    return c


def _n(case):
    return [case["nx"], case["ny"], case["nz"]]


def listed():
    lens = ([288] * 3, 16, "lens")
    return [
        # the outer Krylov step's A_h v on the benchmark grid, and the call the headline stencil rate is quoted on
        _case("apply_fine_289", "apply", *lens),
        # the fine smoother's two-sweep Jacobi map on the same grid
        _case("jacobi_fine_289", "jacobi", *lens),
        # the smoother of the shifted cycle: the most frequent large launch of a solve
        _case("jacobi_2h_145", "jacobi", *lens, level=1, op="B"),
        # the bottom solve's B_4h p: the smallest calls, where latency counts
        _case("apply_4h_73", "apply", *lens, level=2, op="B"),
        # many sources at once: 16 right-hand sides share the coefficients of the layered model
        _case("apply_225x16", "apply", [224] * 3, 16, "layers", nrhs=16),
        # the FP64 true residual and its norm, which decides convergence in the refinement loop
        _case("resid_c128_289", "resid", *lens, prec="c128"),
        # one application of Algorithm 1 on the benchmark grid: 97 % of a solve
        _case("precond_289", "precond", *lens),
        # the same for the eight sources of an inversion model
        _case("precond_153x8", "precond", [152] * 3, 12, "random", nrhs=8),
        # its adjoint: half of every gradient
        _case("precond_adj_153", "precond", [152] * 3, 12, "random", op="A_ADJ"),
        # a small model, all latency and launches
        _case("precond_49", "precond", [48] * 3, 8, "homogeneous"),
        # a whole solve in complex128 to 1e-6, as a small model is checked
        _case("solve_c128_49", "solve", [48] * 3, 8, "homogeneous", prec="c128"),
        # receiver misfit and its gradient in the squared slowness: forward and adjoint solve
        _case("grad_c128_49", "grad", [48] * 3, 4, "random", prec="c128"),
    ]


def _size(rng, lo, hi, cube):
    """Intervals per axis, multiples of 4 spread over the logarithm of the range; a cuboid unless cube."""
    one = lambda a, b: 4 * int(round(math.exp(rng.uniform(math.log(a), math.log(b))) / 4))
    n = one(lo, hi)
    return [n] * 3 if cube else [min(hi, max(lo, 4 * round(n * rng.uniform(0.7, 1.3) / 4))) for _ in range(3)]


def draw(rng):
    kind = rng.choice(["apply", "apply", "jacobi", "jacobi", "resid", "precond", "precond"])
    cube = rng.random() < 0.3
    if kind == "precond":
        n = _size(rng, 64, 224, cube)
        pml = rng.choice([8, 12, 16])
        nodes = (n[0] + 1) * (n[1] + 1) * (n[2] + 1)
        nrhs = min(rng.choice([1, 1, 2, 3, 4, 8]), max(1, int(2.8e7 / nodes)))
        op = rng.choice(["A", "A", "A_ADJ"]) if nodes * nrhs < 5e6 else "A"
        return _case(None, kind, n, pml, rng.choice(["layers", "random"]), op=op, nrhs=nrhs)
    n = _size(rng, 32, 288, cube)
    pml = rng.choice([p for p in (0, 4, 8, 12, 16, 24) if 2 * p < min(n) - 8])
    level = rng.choice([0, 0, 1, 1, 2])
    prec = rng.choice(["c64", "c64", "c64", "c128"])
    medium = rng.choice(["homogeneous", "lens", "layers", "random"])
    nodes = np.prod([v // 2 ** level + 1 for v in n])
    nrhs = min(rng.choice([1, 1, 1, 2, 3, 4, 8, 16]), max(1, int(1.0e8 / nodes)))
    if kind == "jacobi":
        op = "B" if level else "A"
    elif kind == "resid":
        op = rng.choice(["A", "B", "A_ADJ"])
        nrhs = min(nrhs, 2)
    else:
        op = rng.choice(["A", "A", "B", "A_ADJ", "B_ADJ"] + (["Q"] if level == 0 else []))
    return _case(None, kind, n, pml, medium, level, op, prec, nrhs)


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------
def _gen(seed, salt):
    return torch.Generator("cuda").manual_seed((int(seed) * 1000003 + salt) & 0x7FFFFFFF)


def _velocity(case, seed):
    """Wave speed on every fine node, [z, y, x], float64 on the GPU: the recipes of hz_workloads.py."""
    nx, ny, nz = _n(case)
    p = case["pml"]
    ax = [(torch.arange(n + 1, dtype=torch.float64, device="cuda") - p) / (n - 2 * p) for n in (nz, ny, nx)]
    Z, Y, X = ax[0][:, None, None], ax[1][None, :, None], ax[2][None, None, :]
    one = torch.ones((nz + 1, ny + 1, nx + 1), dtype=torch.float64, device="cuda")
    if case["medium"] == "homogeneous":
        return one
    if case["medium"] == "lens":
        return one + 0.5 * torch.exp(-((X - 0.5) ** 2 + (Y - 0.5) ** 2 + (Z - 0.5) ** 2) / (2 * 0.15 ** 2))
    if case["medium"] == "layers":
        u = torch.rand(13, dtype=torch.float64, device="cuda", generator=_gen(seed, 1)).tolist()
        depth, vel = sorted(0.1 + 0.8 * t for t in u[:4]), [1.5 + 3.0 * t for t in u[4:9]]
        c = one * vel[0]
        for d, v in zip(depth, vel[1:]):
            c = torch.where(Z > d, v, c)
        cen = [0.2 + 0.6 * t for t in u[9:12]]
        host = vel[sum(cen[2] > d for d in depth)]
        r2 = (X - cen[0]) ** 2 + (Y - cen[1]) ** 2 + (Z - cen[2]) ** 2
        return torch.where(r2 <= 0.08 ** 2, 10.0 * host, c).contiguous()
    g = torch.randn((nz + 1, ny + 1, nx + 1), dtype=torch.float64, device="cuda", generator=_gen(seed, 2))
    F = torch.fft.rfftn(g)
    k = [torch.fft.fftfreq(s, dtype=torch.float64, device="cuda") for s in g.shape[:2]]
    kx = torch.fft.rfftfreq(g.shape[2], dtype=torch.float64, device="cuda")
    F *= torch.exp(-2 * math.pi ** 2 * 100.0 * (k[0][:, None, None] ** 2 + k[1][None, :, None] ** 2 + kx ** 2))
    g = torch.fft.irfftn(F, s=g.shape)
    return (1.5 + 1.5 * (g - g.min()) / (g.max() - g.min())).contiguous()


def _spacing(case, c):
    """h and omega: unit physical box on the shortest axis, six points in the shortest wavelength."""
    h = 1.0 / (min(_n(case)) - 2 * case["pml"])
    return h, 2.0 * math.pi * float(c.min()) / (PPW * h)


def _shape(case):
    return tuple(v // 2 ** case["level"] + 1 for v in reversed(_n(case)))


def _field(case, seed, salt):
    """Complex Gaussian fields: the spectrum-filling vectors that residuals and Krylov bases are."""
    dt = torch.complex64 if case["prec"] == "c64" else torch.complex128
    return torch.randn((case["nrhs"],) + _shape(case), dtype=dt, device="cuda", generator=_gen(seed, salt))


def _points(case, seed, n, z):
    """n distinct nodes (ix, iy) of the physical box on plane z."""
    p, (nx, ny, _) = case["pml"], _n(case)
    rng = np.random.default_rng(seed)
    flat = rng.choice((nx - 2 * p - 3) * (ny - 2 * p - 3), size=n, replace=False)
    return [(p + 2 + int(f) % (nx - 2 * p - 3), p + 2 + int(f) // (nx - 2 * p - 3), z) for f in flat]


def prepare(case, seed):
    c = _velocity(case, seed)
    h, omega = _spacing(case, c)
    prec = hz.HZ_C64 if case["prec"] == "c64" else hz.HZ_C128
    whole = case["kind"] in ("precond", "solve", "grad")
    params = hz.default_params(tol=1e-6, precision=prec) if whole else hz.default_params()
    solver = hz.Solver(_n(case), case["pml"], h, omega, c, params=params, max_nrhs=case["nrhs"])
    st = {"case": case, "solver": solver}
    if case["kind"] == "solve":
        st["sources"] = [p + (1.0,) for p in _points(case, seed, case["nrhs"], case["nz"] // 2)]
    elif case["kind"] == "grad":
        st["sources"] = [p + (1.0,) for p in _points(case, seed, case["nrhs"], case["pml"] + 4)]
        st["rec"] = np.array(_points(case, seed + 1, 64, case["nz"] - case["pml"] - 4), dtype=np.int32)
        st["d_obs"] = np.zeros((case["nrhs"], 64), dtype=np.complex128)
    else:
        st["x"] = _field(case, seed, 3)
        st["out"] = torch.empty_like(st["x"])
        if case["kind"] == "resid":
            st["g"] = _field(case, seed, 4)
            st["norm2"] = torch.empty(case["nrhs"], dtype=torch.float64, device="cuda")
        if case["kind"] == "precond":
            # an application inside a Krylov loop runs on the loop's own stream
            st["stream"] = torch.cuda.Stream()
    return st


def run(state):
    case, s = state["case"], state["solver"]
    kind, level, op = case["kind"], case["level"], OPS[case["op"]]
    if kind == "apply":
        return s.iofd_apply(state["x"], op=op, level=level, out=state["out"])
    if kind == "jacobi":
        return s.iofd_jacobi(state["x"], level=level, out=state["out"])
    if kind == "resid":
        r, n2 = s.residual_static(state["g"], state["x"], op=op, level=level, out=state["out"],
                                  norm2_out=state["norm2"])
        # the norm of a complex64 residual carries single precision
        return r, (n2 if case["prec"] == "c128" else n2.float())
    if kind == "precond":
        own, cur = state["stream"], torch.cuda.current_stream()
        own.wait_stream(cur)
        with torch.cuda.stream(own):
            z = s.threegrid_precond(state["x"], adjoint=case["op"] == "A_ADJ", out=state["out"])
        cur.wait_stream(own)
        return z
    if kind == "solve":
        v, u, _ = s.helmholtz_solve(state["sources"])
        return v, u
    J, g, _ = s.helmholtz_adjoint_grad(state["sources"], state["rec"], state["d_obs"])
    return J, g


def work(case):
    """Fields in and out once, kappa (or the velocity) once; the operations of the shell form."""
    N = float(np.prod(_shape(case)))
    w = 8 if case["prec"] == "c64" else 16
    nr = case["nrhs"]
    stencil = 2 * 26 + 16 + (40 / nr if case["op"] == "A" else 60 / nr)   # shell sums, four weights, coefficients
    if case["kind"] == "apply":
        return {"bytes": N * (2 * w * nr + w / 2), "flops": N * nr * stencil}
    if case["kind"] == "jacobi":
        return {"bytes": N * (2 * w * nr + w / 2), "flops": N * nr * (stencil + 30)}
    if case["kind"] == "resid":
        return {"bytes": N * (3 * w * nr + w / 2), "flops": N * nr * (stencil + 6)}
    # Algorithm 1 per fine node: 10 fine stencils; on 2h 20 steps of five stencils and about six
    # Gram-Schmidt terms twice over; on 4h 20 solves of eight stencils
    cycle = 10 * 100.0 + 20 * (5 * 110.0 + 12 * 16.0) / 8 + 20 * (8 * 110.0 + 240.0) / 64
    calls = {"precond": 1, "solve": 12, "grad": 20}[case["kind"]]
    out = {"precond": 2 * w * nr + w / 2, "solve": 2 * w * nr + w / 2, "grad": 16.0}[case["kind"]]
    return {"bytes": N * out, "flops": N * nr * cycle * calls}


# ----------------------------------------------------------------------------
# the same in 64 bits, plainly
# ----------------------------------------------------------------------------
def _axis_factors(n, p):
    """abar and achk of one axis: half sum and half difference of the two PML second-difference weights."""
    i = np.arange(-1, n + 2, dtype=np.float64)
    d = np.clip(np.maximum(np.maximum(p - i, i - (n - p)), 0.0), 0.0, p)
    g = GAMMA_MAX * (1 - np.cos(math.pi * d / (2 * p))) if p else np.zeros_like(i)
    node, half = 1 / (1 + 1j * g[1:-1]), 1 / (1 + 0.5j * (g[1:] + g[:-1]))
    dp, dm = node * half[1:], node * half[:-1]
    return 0.5 * (dp + dm), 0.5 * (dp - dm)


def _tables(eta):
    """The eight tabulated functions (alpha_1..5, beta_1..3), cubic Hermite in eta."""
    rows = np.loadtxt(os.path.join(os.path.dirname(hz.__file__), "tables", "iofd_tables.txt"), comments="#")
    T = torch.tensor(rows, dtype=torch.float64, device=eta.device)
    ds = float(rows[1, 0] - rows[0, 0])
    k = torch.clamp((eta / ds).floor().long(), 0, len(rows) - 2)
    t = eta / ds - k
    out = []
    for v, d in [(1 + j, 6 + j) for j in range(5)] + [(11 + j, 14 + j) for j in range(3)]:
        v0, v1, d0, d1 = T[:, v][k], T[:, v][k + 1], T[:, d][k] * ds, T[:, d][k + 1] * ds
        out.append(v0 + t * (d0 + t * (3 * (v1 - v0) - 2 * d0 - d1 + t * (d0 + d1 - 2 * (v1 - v0)))))
    return out


class _Operator64:
    """Rows of A, B or Q of one level, evaluated offset by offset in complex128."""

    def __init__(self, case, seed):
        c = _velocity(case, seed)
        h, omega = _spacing(case, c)
        f, p, n = 2 ** case["level"], case["pml"], _n(case)
        idx = [torch.clamp(torch.arange(0, m + 1, f, device="cuda"), p, m - p) for m in reversed(n)]
        c = c[idx[0]][:, idx[1]][:, :, idx[2]]
        self.ell = h * f
        self.k2 = (omega * self.ell / c) ** 2
        a1, a2, a3, a4, a5, b1, b2, b3 = _tables(torch.clamp(torch.sqrt(self.k2) / (2 * math.pi), max=0.4))
        self.t = [a4, a5 / 4, (1 - a4 - a5) / 4]
        self.m = [a1, a2 / 6, a3 / 12, (1 - a1 - a2 - a3) / 8]
        self.q = [b1, b2 / 6, b3 / 12, (1 - b1 - b2 - b3) / 8]
        self.op = case["op"][0]
        self.shift = 1 + 1j * SIGMA if self.op == "B" else 1.0
        self.ax = []
        for j, m in enumerate(reversed(n)):   # z, y, x
            ab, ac = _axis_factors(m // f, p // f)
            view = [1, 1, 1]
            view[j] = -1
            self.ax.append(tuple(torch.tensor(v, device="cuda").view(view) for v in (-2 * ab, ab + ac, ab - ac)))

    def coeff(self, d):
        """Coefficient of x[i + d] in row i, d = (dz, dy, dx)."""
        far = sum(v != 0 for v in d)
        if self.op == "Q":
            return self.q[far].to(torch.complex128)
        S = 0.0
        for j in range(3):
            S = S + self.t[far - (d[j] != 0)] * self.ax[j][d[j]]   # index -1: the weight of offset -1
        return -(S + self.shift * self.k2 * self.m[far]) / self.ell ** 2

    def apply(self, x, adjoint=False):
        y = torch.zeros_like(x)
        sl = lambda o, s: tuple(slice(max(0, v), n + min(0, v)) for v, n in zip(o, s))
        for d in [(a, b, e) for a in (-1, 0, 1) for b in (-1, 0, 1) for e in (-1, 0, 1)]:
            C = self.coeff(d)
            here, there = sl([-v for v in d], C.shape), sl(d, C.shape)
            if adjoint:
                y[there] += torch.conj(C[here]) * x[here]
            else:
                y[here] += C[here] * x[there]
        return y


def exact(case, seed):
    """None for the whole calls: Algorithm 1 in 64 bits takes minutes in plain host code at these sizes."""
    if case["kind"] in ("precond", "solve", "grad"):
        return None
    H = _Operator64(case, seed)
    x = _field(case, seed, 3).to(torch.complex128)
    adj = case["op"].endswith("ADJ")
    if case["kind"] == "jacobi":
        w, D = OMEGA_J[case["level"]], H.coeff((0, 0, 0))
        out = torch.empty_like(x)
        for r in range(x.shape[0]):
            y1 = w * x[r] / D
            out[r] = y1 + w * (x[r] - H.apply(y1)) / D
        return out
    for r in range(x.shape[0]):
        x[r] = H.apply(x[r], adj)
    if case["kind"] == "apply":
        return x
    x = _field(case, seed, 4).to(torch.complex128) - x
    return x, torch.stack([torch.linalg.vector_norm(v) ** 2 for v in x])
