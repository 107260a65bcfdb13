"""What users of this library have it do, as cases that can be timed and checked.

Every case is one call (or the few calls that belong together) of the public
binding on seeded synthetic geometries: a random smooth free surface, a flat or
bumped bottom and up to four ellipses, split about 1/2, 1/4, 1/4 over the
unknowns as in the repository's workloads.  `exact` restates each result from
the definitions (Table 1 and Secs. 2-5 of arXiv 2108.01786) in FP64 torch.

Kinds:
  solve    node data -> operator -> omega, U, psi (one stage of a time stepper)
  host     the same from host buffers, copies included
  grad     U as an autograd function: forward and backward, all gradients
  evolve   Runge-Kutta steps of the graph formulation
  batch    many geometries of uneven size in one call
  multi    several right-hand sides on one assembled operator
  product  full-accuracy operator times a block of vectors
  targets  velocity at points of the fluid, near and far from the boundaries
  pressure auxiliary Dirichlet problem and its boundary values
"""
import math

import numpy as np
import torch

import paper_2108_01786_gb300 as P

TWO_PI = 2.0 * math.pi
PREC = ("fp64", "fp32_ir", "bf16_ir", "fp16_ir")


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # a small solve (the repository's 640-unknown problem size), where launches and latency count
        {"name": "solve_640_fp32", "kind": "solve", "n": 640, "obstacles": 1, "precision": "fp32_ir"},
        # plain FP64 GMRES on an odd, ragged size: the reference scheme on a desk-top problem
        {"name": "solve_1001_fp64", "kind": "solve", "n": 1001, "obstacles": 3, "precision": "fp64"},
        # a middle-sized stage of a time stepper, odd in every block, BF16 inner storage
        {"name": "solve_4099_bf16", "kind": "solve", "n": 4099, "obstacles": 2, "precision": "bf16_ir"},
        # the repository's headline size and storage
        {"name": "solve_16383_fp16", "kind": "solve", "n": 16383, "obstacles": 3, "precision": "fp16_ir"},
        # a caller without device buffers (size of the paper's finest problem-1 run)
        {"name": "host_8256_fp32", "kind": "host", "n": 8256, "obstacles": 3, "precision": "fp32_ir"},
        # shape and surface gradients of one step of an optimisation (forward and backward)
        {"name": "grad_4096_fp32", "kind": "grad", "n": 4096, "obstacles": 2, "precision": "fp32_ir"},
        # time evolution at four times the paper's coarsest problem-1 resolution
        {"name": "evolve_2944_fp16", "kind": "evolve", "n": 2944, "obstacles": 3, "steps": 2,
         "precision": "fp16_ir"},
        # a parameter ensemble: uneven problems in one call
        {"name": "batch_24_fp32", "kind": "batch", "n": 1024, "nmax": 6144, "problems": 24,
         "obstacles": 3, "precision": "fp32_ir"},
        # several surface potentials on one geometry
        {"name": "multi_5887x12_fp16", "kind": "multi", "n": 5887, "nrhs": 12, "obstacles": 3,
         "precision": "fp16_ir"},
        # the operator applied to a block of vectors (an eigenvalue or a block method of the user's own)
        {"name": "product_8191x24", "kind": "product", "n": 8191, "nrhs": 24, "obstacles": 3,
         "precision": "fp32_ir"},
        # a velocity field: a grid of the fluid and points close to the boundaries
        {"name": "targets_12288", "kind": "targets", "n": 12288, "obstacles": 4, "grid": 200000,
         "near": 20000},
        # pressure on the boundaries of a solved state
        {"name": "pressure_6001_fp32", "kind": "pressure", "n": 6001, "obstacles": 2,
         "precision": "fp32_ir"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "host", "grad", "evolve", "batch", "multi",
                       "product", "targets", "pressure"])
    c = {"kind": kind, "obstacles": rng.randint(0, 4) if kind == "solve" else rng.randint(1, 4)}
    ir = rng.choice(["fp32_ir", "bf16_ir", "fp16_ir"])
    if kind == "solve":
        c["precision"] = rng.choice(["fp64", "fp32_ir", "fp32_ir", "bf16_ir", "fp16_ir", "fp16_ir"])
        c["n"] = _log_int(rng, 512, 6000 if c["precision"] == "fp64" else 16383)
    elif kind == "host":
        c.update(precision=ir, n=_log_int(rng, 640, 10000))
    elif kind == "grad":
        c.update(precision=rng.choice(["fp32_ir", "fp16_ir"]), n=_log_int(rng, 640, 4096))
    elif kind == "evolve":
        c.update(precision=ir, n=_log_int(rng, 640, 5000), steps=rng.randint(1, 2))
    elif kind == "batch":
        c.update(precision=ir, n=_log_int(rng, 512, 1500), problems=rng.randint(4, 24))
        c["nmax"] = _log_int(rng, 2 * c["n"], 6144)
    elif kind == "multi":
        c.update(precision=rng.choice(["bf16_ir", "fp16_ir"]), n=_log_int(rng, 700, 8191),
                 nrhs=_log_int(rng, 2, 40))
    elif kind == "product":
        c.update(precision=ir, n=_log_int(rng, 700, 8191), nrhs=_log_int(rng, 1, 40))
    elif kind == "targets":
        c.update(n=_log_int(rng, 700, 12288), grid=_log_int(rng, 2000, 200000))
        c["near"] = _log_int(rng, 100, 20000)
    else:
        c.update(precision=ir, n=_log_int(rng, 700, 8191))
    return c


# ---------------------------------------------------------------------------
# seeded inputs (numpy; analytic derivatives)
# ---------------------------------------------------------------------------

class Geom:
    """Node data in block order (surface, bottom, obstacles) and the flow."""

    def __init__(self, M, curves, ell, V1, a):
        self.M, self.ell, self.V1, self.a = M, ell, V1, a
        self.zeta, self.dzeta, self.d2zeta = (np.concatenate([c[i] for c in curves]) for i in range(3))
        self.zc = np.array([e[0] + 1j * e[1] for e in ell], dtype=np.complex128)
        self.N = len(self.zeta)


def _alphas(M):
    return TWO_PI * np.arange(M) / M


def _series(M, A, B):
    """sum_k A_k cos(k alpha) + B_k sin(k alpha), k = 1.., and two derivatives."""
    k = np.arange(1, len(A) + 1)
    a = _alphas(M)[:, None]
    c, s = np.cos(k * a), np.sin(k * a)
    return c @ A + s @ B, (-s * k) @ A + (c * k) @ B, (-c * k * k) @ A + (-s * k * k) @ B


def _noise(rng, M, amp, kmax):
    """Band-limited noise of the given size (|k| <= kmax)."""
    kmax = min(kmax, max(1, M // 8))
    k = np.arange(1, kmax + 1)
    A, B = rng.standard_normal(kmax), rng.standard_normal(kmax)
    return _series(M, amp / math.sqrt(kmax) * A, amp / math.sqrt(kmax) * B)[0]


def _surface(rng, M, amp, kmax):
    kmax = min(kmax, max(2, M // 16))
    k = np.arange(1, kmax + 1, dtype=np.float64)
    A, B = rng.standard_normal(kmax) * k ** -2.0, rng.standard_normal(kmax) * k ** -2.0
    e = np.abs(_series(2048, A, B)[0]).max()
    return _series(M, amp / e * A, amp / e * B)


def _geometry(rng, n, obstacles):
    M0, M1 = ((n + 1) // 2, (n + 1) // 4) if obstacles else (n - n // 2, n // 2)
    rest = n - M0 - M1
    M = [M0, M1] + [rest // obstacles] * (obstacles - 1) if obstacles else [M0, M1]
    if obstacles:
        M.append(n - sum(M))
    a0, a1 = _alphas(M0), _alphas(M1)
    e, de, d2e = _surface(rng, M0, rng.uniform(0.08, 0.14), 32)
    h, w = (0.25, 0.4) if rng.random() < 0.5 else (0.0, 0.4)
    g = h * np.exp(-(a1 - math.pi) ** 2 / w)
    dg = g * (-2.0 * (a1 - math.pi) / w)
    d2g = g * ((2.0 * (a1 - math.pi) / w) ** 2 - 2.0 / w)
    curves = [(a0 + 1j * e, 1.0 + 1j * de, 1j * d2e), (a1 + 1j * (g - 1.3), 1.0 + 1j * dg, 1j * d2g)]
    ell = []
    for j in range(obstacles):   # one ellipse per slot of the period, clear of surface and bottom
        x = TWO_PI * (j + 0.5 + rng.uniform(-0.15, 0.15)) / obstacles
        ell.append((x, rng.uniform(-0.62, -0.5), rng.uniform(0.1, 0.22), rng.uniform(0.08, 0.16),
                    rng.uniform(0.0, math.pi)))
        a = _alphas(M[2 + j])
        q, b, r = ell[-1][2], ell[-1][3], np.exp(1j * ell[-1][4])
        curves.append((x + 1j * ell[-1][1] + r * (q * np.cos(a) - 1j * b * np.sin(a)),
                       r * (-q * np.sin(a) - 1j * b * np.cos(a)),
                       r * (-q * np.cos(a) + 1j * b * np.sin(a))))
    return Geom(M, curves, ell, rng.uniform(0.5, 1.5), rng.uniform(-0.5, 0.5, size=obstacles))


def _height(g, k, x):
    o = sum(g.M[:k])
    z = g.zeta[o:o + g.M[k]]
    return np.interp(x, np.append(z.real, z.real[0] + TWO_PI), np.append(z.imag, z.imag[0]))


def _targets(rng, g, grid, near):
    """`grid` points of a uniform grid of the fluid (spread over those it has) and
    `near` points within two node spacings of a boundary, on the fluid side."""
    side = int(math.sqrt(grid / 0.5))
    nx, ny = max(4, 2 * side), max(4, side // 2)
    X, Y = np.meshgrid((np.arange(nx) + rng.random()) * TWO_PI / nx, -1.3 + (np.arange(ny) + 0.5) * 1.45 / ny)
    z = (X + 1j * Y).ravel()
    ok = (z.imag < _height(g, 0, z.real) - 0.005) & (z.imag > _height(g, 1, z.real) + 0.005)
    for x, y, q, b, th in g.ell:
        w = (z - (x + 1j * y)) * np.exp(-1j * th)
        ok &= (w.real / (q + 0.005)) ** 2 + (w.imag / (b + 0.005)) ** 2 > 1.0
    z = z[ok][np.linspace(0, np.count_nonzero(ok) - 1, grid).astype(np.int64)]
    blk = np.repeat(np.arange(len(g.M)), g.M)
    i = rng.integers(0, g.N, near)
    t = g.dzeta[i]
    h = np.abs(t) * TWO_PI / np.asarray(g.M)[blk[i]]
    t = t / np.abs(t)
    off = np.where(blk[i] == 0, -1.0, 1.0) * rng.uniform(0.05, 2.0, near)
    return np.concatenate([z, g.zeta[i] + h * (1j * off * t + rng.uniform(-0.5, 0.5, near) * t)])


def _inputs(case, seed):
    """(geometry or list of geometries, dict of numpy arrays) of a case."""
    rng = np.random.default_rng([seed, case["n"]])
    kind = case["kind"]
    if kind == "batch":
        lo, hi, p = math.log(case["n"]), math.log(case["nmax"]), case["problems"]
        sizes = [int(round(math.exp(lo + (hi - lo) * i / (p - 1)))) for i in range(p)]
        gs = [_geometry(rng, n, 1 + (i + case["obstacles"]) % 4) for i, n in enumerate(sizes)]
        return gs, {"phit": np.concatenate([_noise(rng, g.M[0], 0.05, 20) for g in gs])}
    g = _geometry(rng, case["n"], case["obstacles"])
    M0 = g.M[0]
    d = {}
    if kind in ("solve", "host", "grad"):
        d["phit"] = _noise(rng, M0, 0.05, 48)
    if kind == "grad":
        d["gU"] = _noise(rng, M0, 0.1, 8)
    if kind == "evolve":
        d["eta"], d["phit"] = _surface(rng, M0, 0.08, 6)[0], _noise(rng, M0, 0.05, 6)
    if kind == "multi":
        d["phit"] = np.stack([_noise(rng, M0, 0.05, 8 + r) for r in range(case["nrhs"])])
    if kind == "product":
        d["x"] = np.stack([np.concatenate([_noise(rng, m, 0.3, 24) for m in g.M]) for _ in range(case["nrhs"])])
    if kind == "targets":
        d["omega"] = np.concatenate([_noise(rng, m, 0.3, 24) for m in g.M])
        d["z"] = _targets(rng, g, case["grid"], case["near"])
    if kind == "pressure":
        d["phit"], d["U"] = _noise(rng, M0, 0.05, 20), _noise(rng, M0, 0.3, 20)
    return g, d


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

class State:
    """What a program holds between calls; releases its handle with itself."""

    def __init__(self, kind):
        self.kind, self.ctx, self.batch = kind, None, None

    def __del__(self):
        if self.ctx is not None:
            P.bie_destroy(self.ctx)
        if self.batch is not None:
            P.bie_batch_destroy(self.batch)


def _dev(x):
    return torch.as_tensor(x, device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    g, d = _inputs(case, seed)
    s = State(kind)
    s.case, s.prec = case, case.get("precision")
    if kind == "batch":
        s.batch = P.bie_batch_create(0, torch.cuda.current_stream())
        for p, q in enumerate(g):
            P.bie_batch_set_problem(s.batch, p, q.M, _dev(q.zeta), _dev(q.dzeta), _dev(q.d2zeta), q.zc, q.V1, q.a)
        s.N, s.M0 = sum(q.N for q in g), sum(q.M[0] for q in g)
        s.phit = _dev(d["phit"])
        return s
    s.M, s.V1, s.a, s.zc, s.N = g.M, g.V1, g.a, g.zc, g.N
    if kind == "host":
        pin = lambda x: torch.as_tensor(x).pin_memory()  # noqa: E731
        s.node = [pin(x) for x in (g.zeta, g.dzeta, g.d2zeta)]
        s.phit = pin(d["phit"])
        s.out = [pin(np.zeros(n)) for n in (g.N, g.M[0], max(1, len(g.M) - 2))]
        s.ctx = P.bie_create(0, torch.cuda.current_stream())
        return s
    s.node = [_dev(x) for x in (g.zeta, g.dzeta, g.d2zeta)]
    s.d = {k: _dev(v).contiguous() for k, v in d.items()}
    if kind == "grad":
        s.solver = P.Solver(g.M, g.V1, g.a, precision=s.prec)
        s.leaf = [x.requires_grad_(True) for x in s.node] + [torch.as_tensor(g.zc).requires_grad_(True),
                                                            s.d["phit"].requires_grad_(True)]
        return s
    s.ctx = P.bie_create(0, torch.cuda.current_stream())
    P.bie_set_geometry(s.ctx, s.M, *s.node, s.zc)
    P.bie_set_flow(s.ctx, s.V1, s.a)
    if kind in ("multi", "product", "pressure"):
        P.bie_assemble(s.ctx, s.prec)
    return s


def _new(*shape, dtype=torch.float64):
    return torch.empty(shape, dtype=dtype, device="cuda")


def run(s):
    kind = s.kind
    if kind == "batch":
        omega, U = _keep(s, "omega", s.N), _keep(s, "U", s.M0)
        P.bie_batch_run(s.batch, s.case["problems"], s.phit, omega, U, s.prec)
        return {"omega": omega, "U": U}
    M0 = s.M[0]
    if kind == "host":
        P.bie_solve_host(s.ctx, s.M, *s.node, s.zc, s.V1, s.a, s.phit, s.prec, *s.out)
        return {"omega": s.out[0], "U": s.out[1], "psi": s.out[2]}
    if kind == "grad":
        U = P.solve_u(*s.leaf, s.solver)
        return {"U": U.detach(), "grads": list(torch.autograd.grad(U, s.leaf, s.d["gU"]))}
    if kind == "solve":
        omega, U, psi = _new(s.N), _new(M0), torch.zeros(max(1, len(s.M) - 2), dtype=torch.float64, device="cuda")
        P.bie_set_geometry(s.ctx, s.M, *s.node, s.zc)
        P.bie_set_flow(s.ctx, s.V1, s.a)
        P.bie_assemble(s.ctx, s.prec)
        P.bie_solve(s.ctx, s.d["phit"], omega, U, psi)
        return {"omega": omega, "U": U, "psi": psi}
    if kind == "evolve":
        eta, phit = s.d["eta"].clone(), s.d["phit"].clone()
        E, _ = P.bie_evolve(s.ctx, eta, phit, 1e-3, s.case["steps"], formulation="graph", integrator="rk4",
                            filter=True, precision=s.prec)
        return {"eta": eta, "phit": phit, "energy": E}
    if kind == "multi":
        nr = s.case["nrhs"]
        omega, U = _new(nr, s.N), _new(nr, M0)
        P.bie_solve_multi(s.ctx, s.d["phit"], omega, U)
        return {"omega": omega, "U": U}
    if kind == "product":
        y = _new(s.case["nrhs"], s.N)
        P.bie_matmat_full(s.ctx, s.d["x"], y)
        return {"y": y}
    if kind == "targets":
        uv = _new(s.d["z"].numel(), dtype=torch.complex128)
        P.bie_eval_velocity(s.ctx, s.d["omega"], s.d["z"], uv, mode=P.VEL_AUTO, near_spacings=4.0)
        return {"uv": uv}
    b, omega, phi = _new(s.N), _new(s.N), _new(s.N, dtype=torch.complex128)
    P.bie_pressure_rhs(s.ctx, s.d["phit"], s.d["U"], b, tau=0.1, g=1.0)
    P.bie_solve_b(s.ctx, b, omega)
    P.bie_boundary_potential(s.ctx, omega, phi)
    return {"omega": omega, "phi": phi}


def _keep(s, name, n):
    """An output buffer that the program keeps from call to call (a batch records its pointers)."""
    if not hasattr(s, name):
        setattr(s, name, _new(n))
    return getattr(s, name)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

# FP32-class operations of one kernel entry 1/2 cot of a node difference times
# zeta' (complex product, reciprocal, complex product) in plain arithmetic, and
# Krylov products a solve to 1e-14 takes
ENTRY, STEPS = 24, 16


def work(case):
    kind, n = case["kind"], case["n"]
    if kind == "batch":
        p = case["problems"]
        sizes = [n * (case["nmax"] / n) ** (i / max(1, p - 1)) for i in range(p)]
    else:
        sizes = [n]
    solve = sum(q * q * (ENTRY + 2.0 * STEPS) + q * q for q in sizes)
    io = sum(8.0 * (6 * q + 0.5 * q + 1.5 * q) for q in sizes)   # node data, phi~ in; omega, U out
    if kind in ("solve", "host", "batch"):
        return {"bytes": io, "flops": solve}
    if kind == "grad":   # two solves, and one pass over the pairs for the kernel derivatives
        return {"bytes": 2 * io, "flops": 2 * solve + 2.0 * ENTRY * n * n}
    if kind == "evolve":
        return {"bytes": 16.0 * n, "flops": (4 * case["steps"] + 1) * solve}
    if kind == "multi":
        nr = case["nrhs"]
        return {"bytes": 8.0 * nr * 2 * n, "flops": 2.0 * STEPS * nr * n * n}
    if kind == "product":
        nr = case["nrhs"]
        return {"bytes": 8.0 * n * n + 16.0 * nr * n, "flops": 2.0 * nr * n * n}
    if kind == "targets":
        t = case["grid"] + case["near"]
        return {"bytes": 32.0 * t + 56.0 * n, "flops": 16.0 * t * n + ENTRY * n * n}
    return {"bytes": 32.0 * n, "flops": 2.0 * STEPS * n * n + 2.0 * ENTRY * n * n}


# ---------------------------------------------------------------------------
# the same results from the definitions, in FP64 torch
# ---------------------------------------------------------------------------

def _half_cot(x, y):
    """Real and imaginary part of 1/2 cot((x + iy)/2) without cancellation."""
    s, c, sh, ch = torch.sin(0.5 * x), torch.cos(0.5 * x), torch.sinh(0.5 * y), torch.cosh(0.5 * y)
    n = 0.5 / (s * s + sh * sh)
    return s * c * n, -sh * ch * n


class Exact:
    """The discrete method on one geometry: nodes as FP64 / complex128 tensors."""

    def __init__(self, M, zeta, dzeta, d2zeta, zc, V1, a):
        self.M, self.z, self.dz, self.d2z, self.zc, self.V1, self.a = M, zeta, dzeta, d2zeta, zc, V1, a
        dev = zeta.device
        self.N, self.M0 = zeta.numel(), M[0]
        self.o = np.concatenate([[0], np.cumsum(M)]).tolist()
        self.blk = torch.repeat_interleave(torch.arange(len(M), device=dev), torch.tensor(M, device=dev))
        self.Mf = torch.tensor(M, dtype=torch.float64, device=dev)[self.blk]

    def parts(self, v):
        return [v[..., self.o[k]:self.o[k + 1]] for k in range(len(self.M))]

    @staticmethod
    def symbol(v, f):
        M = v.shape[-1]
        k = torch.fft.fftfreq(M, d=1.0 / M, device=v.device, dtype=torch.float64)
        if M % 2 == 0:
            k[M // 2] = 0.0
        return torch.fft.ifft(f(k) * torch.fft.fft(v)).real

    def d(self, v):
        return self.symbol(v, lambda k: 1j * k)

    def hil(self, v):
        return self.symbol(v, lambda k: -1j * torch.sign(k))

    def diff(self, rows):
        """1/2 cot((zeta_l - zeta_m)/2) for rows m (a range), zero on the diagonal."""
        x = self.z.real[None, :] - self.z.real[rows, None]
        y = self.z.imag[None, :] - self.z.imag[rows, None]
        r = torch.arange(rows.start, rows.stop, device=x.device)
        eye = r[:, None] == torch.arange(self.N, device=x.device)[None, :]
        hr, hi = _half_cot(torch.where(eye, torch.ones_like(x), x), torch.where(eye, torch.zeros_like(y), y))
        return hr.masked_fill(eye, 0.0), hi.masked_fill(eye, 0.0), eye

    def matrix_rows(self, rows):
        hr, hi, eye = self.diff(rows)
        F_re = self.dz.real * hr - self.dz.imag * hi
        F_im = self.dz.real * hi + self.dz.imag * hr
        kr, js = self.blk[rows, None], self.blk[None, :]
        A = torch.where((kr == 0) == (js == 0), F_im, torch.where(kr == 0, F_re, -F_re))
        lim = (self.d2z[rows] / (2.0 * self.dz[rows])).imag
        A = torch.where(eye, lim[:, None], A) / self.Mf
        A = A + eye * torch.where(kr == 0, -0.5, 0.5)
        return A - ((kr == js) & (kr >= 2)) / self.Mf

    def matrix(self, step=1024):
        return torch.cat([self.matrix_rows(slice(i, min(self.N, i + step))) for i in range(0, self.N, step)])

    def rhs(self, phit):
        zs = self.z[self.M0:]
        psi = self.V1 * zs.imag
        for aj, zj in zip(self.a, self.zc):
            psi = psi - float(aj) * torch.log(torch.abs(1.0 - torch.exp(1j * (zs - zj))))
        return torch.cat([phit, -psi])

    def dphi_mv(self, z):
        out = self.V1 + 0.0 * z
        for aj, zj in zip(self.a, self.zc):
            hr, hi = _half_cot((z - zj).real, (z - zj).imag)
            out = out + float(aj) * (0.5 - 1j * torch.complex(hr, hi))
        return out

    def reg(self, k, rows):
        """1/2 cot((beta_l - alpha_m)/2) of boundary k's parameters, zero on the diagonal."""
        M = self.M[k]
        i = torch.arange(M, device=self.z.device)
        q = (i[None, :] - i[rows, None]) % M
        t = torch.zeros(M, dtype=torch.float64, device=self.z.device)
        t[1:] = 0.5 / torch.tan(math.pi * torch.arange(1, M, device=t.device, dtype=torch.float64) / M)
        return t[q]

    def velocity(self, omega, step=1024):
        """Normal velocity of the surface (omega: one vector)."""
        w = torch.cat([self.d(v) for v in self.parts(omega)]) / self.Mf
        dz0, out = self.dz[:self.M0], []
        for i in range(0, self.M0, step):
            r = slice(i, min(self.M0, i + step))
            hr, hi, eye = self.diff(r)
            a, b = dz0.real[r, None], dz0.imag[r, None]
            im = -(a * hi + b * hr)                          # Im{zeta_m' 1/2 cot((zeta_m - zeta_l)/2)}
            re = -(a * hr - b * hi)[:, :self.M0] + self.reg(0, r)
            re = re + eye[:, :self.M0] * (self.d2z[r] / (2.0 * self.dz[r])).real[:, None]
            out.append(im[:, self.M0:] @ w[self.M0:] - re @ w[:self.M0])
        t = torch.cat(out) - 0.5 * self.hil(w[:self.M0] * self.Mf[:self.M0])
        t = t - (self.V1 + 0.5 * float(np.sum(self.a))) * dz0.imag
        for aj, zj in zip(self.a, self.zc):
            u = self.z[:self.M0] - zj
            hr, hi = _half_cot(u.real, u.imag)
            t = t + float(aj) * (hr * dz0.real - hi * dz0.imag)
        return t / torch.abs(dz0)

    def psi(self, omega):
        p = self.parts(omega)[2:]
        return torch.stack([v.mean() for v in p]) if p else torch.zeros(1, dtype=torch.float64, device=omega.device)

    def solve(self, phit):
        omega = torch.linalg.solve(self.matrix(), self.rhs(phit))
        return omega, self.velocity(omega), self.psi(omega)

    def curvature(self):
        z1, z2 = self.dz[:self.M0], self.d2z[:self.M0]
        return (z2 * z1.conj()).imag / torch.abs(z1) ** 3

    def phi_s(self, phit):
        return self.d(phit) + (self.dphi_mv(self.z[:self.M0]) * self.dz[:self.M0]).real

    def boundary_potential(self, omega, A, step=1024):
        """Phi~ on every boundary from the fluid side (Plemelj)."""
        y, parts = A @ omega, self.parts(omega)
        hil = torch.cat([self.hil(v) for v in parts])
        w, other = omega / self.Mf, []
        for i in range(0, self.N, step):
            rows = slice(i, min(self.N, i + step))
            hr, hi, eye = self.diff(rows)
            F_re = self.dz.real * hr - self.dz.imag * hi
            F_im = self.dz.real * hi + self.dz.imag * hr
            kr, js = self.blk[rows, None], self.blk[None, :]
            lim = (self.d2z[rows] / (2.0 * self.dz[rows])).real
            T = torch.where((kr == 0) == (js == 0), F_re, F_im)
            T = torch.where(eye, lim[:, None], T)
            for k in range(len(self.M)):   # the own boundary less its 1/2 cot
                a, b = max(i, self.o[k]), min(rows.stop, self.o[k + 1])
                if a < b:
                    T[a - i:b - i, self.o[k]:self.o[k + 1]] -= self.reg(k, slice(a - self.o[k], b - self.o[k]))
            # surface rows: Im = 1/2 H omega_0 - G omega_0 + K omega_j; solid rows: Re = K omega_0 + G omega_j - 1/2 H
            sg = torch.where((kr == 0) & (js == 0), -1.0, 1.0)
            other.append((T * sg) @ w)
        t = torch.cat(other) + torch.where(self.blk == 0, 0.5, -0.5) * hil
        add = torch.cat([torch.zeros_like(v) if k < 2 else v.mean().expand_as(v) for k, v in enumerate(parts)])
        return torch.where(self.blk == 0, torch.complex(y, t), torch.complex(t, y + add))

    def boundary_values(self, omega, step=1024):
        """Phi' at every node from the fluid side."""
        dw = [self.d(v) for v in self.parts(omega)]
        gam = torch.cat([-dw[0]] + dw[1:])
        hg = torch.cat([self.hil(v) for v in self.parts(gam)])
        c, dmv, out = gam / self.Mf, self.dphi_mv(self.z), []
        sn, ss = (dmv * 1j * self.dz).real, (dmv * self.dz).real
        for i in range(0, self.N, step):
            r = slice(i, min(self.N, i + step))
            hr, hi, eye = self.diff(r)
            a, b = self.dz.real[r, None], self.dz.imag[r, None]
            re, im = -(a * hr - b * hi), -(a * hi + b * hr)
            for k in range(len(self.M)):
                p, q = max(i, self.o[k]), min(r.stop, self.o[k + 1])
                if p < q:
                    re[p - i:q - i, self.o[k]:self.o[k + 1]] += self.reg(k, slice(p - self.o[k], q - self.o[k]))
            lim = self.d2z[r] / (2.0 * self.dz[r])
            re, im = torch.where(eye, lim.real[:, None], re), torch.where(eye, lim.imag[:, None], im)
            m = self.M0
            sn_r = sn[r] + re[:, :m] @ c[:m] + im[:, m:] @ c[m:]
            ss_r = ss[r] + im[:, :m] @ c[:m] - re[:, m:] @ c[m:]
            surf = self.blk[r] == 0
            sn_r = sn_r + torch.where(surf, 0.5 * hg[r], -0.5 * gam[r])
            ss_r = ss_r + torch.where(surf, 0.5 * gam[r], -0.5 * hg[r])
            out.append(torch.complex(ss_r, -sn_r) / self.dz[r])
        return torch.cat(out)

    def helsing(self, f, z, step=512):
        """Boundary values f taken into the fluid (Helsing-Ojala ratio)."""
        w = torch.where(self.blk == 0, -1.0, 1.0) * self.dz / self.Mf
        out = []
        for i in range(0, z.numel(), step):
            x = self.z.real[None, :] - z.real[i:i + step, None]
            y = self.z.imag[None, :] - z.imag[i:i + step, None]
            lam = torch.complex(*_half_cot(x, y)) * w
            out.append((lam @ f) / lam.sum(dim=1))
        return torch.cat(out)


def _exact_of(g, dev):
    t = lambda x: torch.as_tensor(x, device=dev)  # noqa: E731
    return Exact(g.M, t(g.zeta), t(g.dzeta), t(g.d2zeta), [complex(z) for z in g.zc], g.V1, g.a)


def _graph_rates(g, eta, phit, dev, grav=1.0, tau=0.1):
    x = _exact_of(g, dev)
    M0 = g.M[0]
    ea = x.d(eta)
    eaa = x.d(ea)
    al = torch.as_tensor(_alphas(M0), device=dev)
    x.z = torch.cat([torch.complex(al, eta), x.z[M0:]])
    x.dz = torch.cat([torch.complex(torch.ones_like(ea), ea), x.dz[M0:]])
    x.d2z = torch.cat([torch.complex(torch.zeros_like(eaa), eaa), x.d2z[M0:]])
    _, U, _ = x.solve(phit)
    s = torch.sqrt(1.0 + ea * ea)
    dmv = x.dphi_mv(x.z[:M0])
    mvn = (dmv * 1j * x.dz[:M0]).real / s
    pa = x.d(phit)
    grad2 = ((pa + (dmv * x.dz[:M0]).real) / s) ** 2 + U * U
    th = eaa / (1.0 + ea * ea)
    return s * U, (pa / s) * (ea * U) + (U - mvn) * U - 0.5 * grad2 - grav * eta + tau * th / s


def _filter(v):
    M = v.numel()
    k = torch.fft.fftfreq(M, d=1.0 / M, device=v.device, dtype=torch.float64).abs()
    return torch.fft.ifft(torch.exp(-36.0 * (k / (M / 2.0)) ** 36) * torch.fft.fft(v)).real


def exact(case, seed):
    kind, dev = case["kind"], "cuda" if torch.cuda.is_available() else "cpu"
    g, d = _inputs(case, seed)
    d = {k: torch.as_tensor(v, device=dev) for k, v in d.items()}
    if kind == "batch":
        om, U, at = [], [], 0
        for q in g:
            o, u, _ = _exact_of(q, dev).solve(d["phit"][at:at + q.M[0]])
            at += q.M[0]
            om.append(o)
            U.append(u)
        return {"omega": torch.cat(om), "U": torch.cat(U)}
    x = _exact_of(g, dev)
    if kind in ("solve", "host"):
        omega, U, psi = x.solve(d["phit"])
        return {"omega": omega, "U": U, "psi": psi}
    if kind == "grad":
        leaf = [v.clone().requires_grad_(True) for v in (x.z, x.dz, x.d2z)]
        zc = torch.as_tensor(g.zc, device=dev).requires_grad_(True)
        phit = d["phit"].clone().requires_grad_(True)
        e = Exact(g.M, *leaf, list(zc), g.V1, g.a)
        U = e.velocity(torch.linalg.solve(e.matrix(g.N), e.rhs(phit)), step=g.M[0])
        return {"U": U.detach(), "grads": list(torch.autograd.grad(U, leaf + [zc, phit], d["gU"]))}
    if kind == "evolve":
        eta, phit, h = d["eta"], d["phit"], 1e-3
        for _ in range(case["steps"]):
            k = [_graph_rates(g, eta, phit, dev)]
            for c in (0.5 * h, 0.5 * h, h):
                k.append(_graph_rates(g, eta + c * k[-1][0], phit + c * k[-1][1], dev))
            eta, phit = (_filter(v + h / 6.0 * (k[0][i] + 2.0 * k[1][i] + 2.0 * k[2][i] + k[3][i]))
                         for i, v in ((0, eta), (1, phit)))
        return {"eta": eta, "phit": phit, "energy": None}
    if kind == "multi":
        B = torch.stack([x.rhs(p) for p in d["phit"]], dim=1)
        omega = torch.linalg.solve(x.matrix(), B).T.contiguous()
        return {"omega": omega, "U": torch.stack([x.velocity(o) for o in omega])}
    if kind == "product":
        return {"y": (d["x"] @ x.matrix().T).contiguous()}
    if kind == "targets":
        if 1.0 * case["n"] * (case["grid"] + case["near"]) > 3e9:
            return None
        return {"uv": x.helsing(x.boundary_values(d["omega"]), d["z"])}
    z0, M0 = x.z[:g.M[0]], g.M[0]
    s = torch.abs(x.dz[:M0])
    b = torch.zeros(g.N, dtype=torch.float64, device=dev)
    b[:M0] = 0.1 * x.curvature() - 0.5 * ((x.phi_s(d["phit"]) / s) ** 2 + d["U"] ** 2) - z0.imag
    A = x.matrix()
    omega = torch.linalg.solve(A, b)
    return {"omega": omega, "phi": x.boundary_potential(omega, A)}
