"""What a user of this library has it do, as cases that can be timed and checked.

A case is a dict of plain values.  `listed()` gives the standing ones, `draw()`
more of the same ranges, `prepare()` what a program holds before the call,
`run()` one pass through the public entry points, `work()` the least bytes and
operations of a pass, `exact()` its result in 64 bits by plain torch (the PML
discretisation and the recursive sweep written out again, a direct solve where
the grid is small enough), without this library's code.

Kinds:
  apply     z = M r, one preconditioner apply on a set-up handle: the inner call
            of every Krylov iteration, by far the largest part of a solve
  batch     one batched apply over uneven problems (a server's mixed queue)
  matvec    y = A x in complex FP32 (each Krylov iteration) or FP64 (residuals)
  solve     helm_solve on a set-up handle: GMRES to 1e-6 for several sources
  setup     a new velocity model: set up, apply once, release (one step of an
            outer iteration over models, or an operator for another solver)
  gradient  a loss on receivers and its velocity gradient through autograd
            (set up, solve, adjoint solve, gradient kernel)
"""
import math

import torch

from paper_1502_07266_gb300 import helm
from paper_1502_07266_gb300.autograd import helmholtz_solve

TOL = 1e-6          # GMRES tolerance of the solves
PML_C = 10.0


# ------------------------------------------------------------------- the cases

def _apply(name, n, nrhs, form, precision, schedule, b_aux, velocity, b=6, d=1):
    return {"name": name, "kind": "apply", "n": n, "b": b, "d": d, "nrhs": nrhs, "form": form,
            "precision": precision, "schedule": schedule, "b_aux": b_aux, "velocity": velocity}


def listed():
    return [
        # the 64-source workload of the benchmark: split FP16 operators, two fronts, 2-layer auxiliary PML
        _apply("apply_two_127x64", 127, 64, "dense", "split_fp16", "two_front", 2, "random"),
        # the same preconditioner serving one source at the mid size: latency is all that counts
        _apply("apply_two_63x1", 63, 1, "dense", "split_fp16", "two_front", 2, "lens"),
        # the sweep as Algorithms 4 and 6 print it (one front, b_aux = b), operators and products in FP32
        _apply("apply_one_47x16_fp32", 47, 16, "dense", "fp32", "one_front", 6, "lens"),
        # half-size storage, an even grid and a ragged number of sources
        _apply("apply_one_50x33_fp16", 50, 33, "dense", "fp16", "one_front", 3, "random"),
        # the library's default options (chain form, FP32) on the lens with one source
        _apply("apply_chain_63x1", 63, 1, "chain", "fp32", "one_front", 6, "lens"),
        # a mixed queue: three problems of different size, b = 5, in one launch
        {"name": "apply_batch_uneven", "kind": "batch", "n": 47, "n2": 31, "n3": 39, "b": 5, "d": 1, "nrhs": 16,
         "nrhs2": 8, "nrhs3": 32, "precision": "split_fp16"},
        # the operator on the 64-source workload's vectors
        {"name": "matvec_127x64", "kind": "matvec", "n": 127, "b": 6, "nrhs": 64, "fp64": False},
        # the smallest call: one vector of the small grid
        {"name": "matvec_31x1", "kind": "matvec", "n": 31, "b": 6, "nrhs": 1, "fp64": False},
        # the FP64 operator of the residuals
        {"name": "matvec64_63x16", "kind": "matvec", "n": 63, "b": 6, "nrhs": 16, "fp64": True},
        # a shot gather: 16 sources solved to 1e-6 on a set-up handle
        {"name": "solve_two_63x16", "kind": "solve", "n": 63, "b": 6, "d": 1, "nrhs": 16, "form": "dense",
         "precision": "split_fp16", "schedule": "two_front", "b_aux": 2, "velocity": "lens"},
        # a new model: factors, restricted operators, packing, and the first apply
        {"name": "setup_two_95x1", "kind": "setup", "n": 95, "b": 6, "d": 1, "nrhs": 1, "form": "dense",
         "precision": "split_fp16", "schedule": "two_front", "b_aux": 2, "velocity": "random"},
        # one loss and its velocity gradient for 16 sources
        {"name": "gradient_23x16", "kind": "gradient", "n": 23, "b": 6, "d": 1, "nrhs": 16, "precision": "fp32",
         "b_aux": 0, "velocity": "bump"},
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["two", "two", "two", "one", "one", "chain", "batch", "matvec", "matvec", "solve", "setup",
                       "gradient"])
    velocity = rng.choice(["lens", "random", "waveguide", "constant"])
    if kind == "two":
        d = rng.choice([1, 1, 1, 2])
        b = rng.choice([4, 5, 6, 8])
        n = _log(rng, 15, 111)
        c = _apply("", n, _log(rng, 1, 64), "dense", rng.choice(["split_fp16", "split_fp16", "fp16", "fp32"]),
                   "two_front", rng.choice([1, 2, 2, 3]) if d == 1 else rng.choice([1, 2]), velocity, b=b, d=d)
    elif kind == "one":
        d = rng.choice([1, 1, 1, 2])
        c = _apply("", _log(rng, 15, 55), _log(rng, 1, 64), "dense", rng.choice(["split_fp16", "fp16", "fp32"]),
                   "one_front", rng.choice([2, 3, 4, 5, 6]), velocity, b=rng.choice([5, 6]), d=d)
    elif kind == "chain":
        c = _apply("", _log(rng, 11, 50), _log(rng, 1, 64), "chain", rng.choice(["fp32", "fp16", "split_fp16"]),
                   "one_front", rng.choice([0, 2, 3, 4]), velocity, b=rng.choice([5, 6]), d=rng.choice([1, 1, 2]))
    elif kind == "batch":
        c = {"kind": "batch", "n": _log(rng, 13, 47), "n2": _log(rng, 13, 47), "n3": _log(rng, 13, 47), "b": 5, "d": 1,
             "nrhs": _log(rng, 1, 24), "nrhs2": _log(rng, 1, 24), "nrhs3": _log(rng, 1, 24),
             "precision": rng.choice(["fp32", "fp16", "split_fp16"])}
    elif kind == "matvec":
        fp64 = rng.random() < 0.4
        c = {"kind": "matvec", "n": _log(rng, 15, 79 if fp64 else 120), "b": rng.choice([4, 5, 6, 8]),
             "nrhs": _log(rng, 1, 32 if fp64 else 64), "fp64": fp64}
    elif kind == "solve":
        c = {"kind": "solve", "n": _log(rng, 15, 55), "b": rng.choice([5, 6]), "d": 1, "nrhs": _log(rng, 1, 24),
             "form": "dense", "precision": rng.choice(["split_fp16", "split_fp16", "fp32"]), "schedule": "two_front",
             "b_aux": rng.choice([2, 3]), "velocity": velocity}
    elif kind == "setup":
        c = {"kind": "setup", "n": _log(rng, 21, 80), "b": rng.choice([5, 6]), "d": 1, "nrhs": _log(rng, 1, 16),
             "form": "dense", "precision": rng.choice(["split_fp16", "fp32"]), "schedule": "two_front",
             "b_aux": rng.choice([2, 3]), "velocity": velocity}
    else:
        c = {"kind": "gradient", "n": _log(rng, 11, 23), "b": rng.choice([4, 5, 6]), "d": 1,
             "nrhs": _log(rng, 1, 16), "precision": rng.choice(["fp32", "split_fp16"]), "b_aux": rng.choice([0, 3]),
             "velocity": "bump"}
    c.pop("name", None)
    return c


# ------------------------------------------------------------------ the inputs

def _omega(n):
    return 2.0 * math.pi * n / 8.0                   # 8 points per wavelength at c = 1


def _gen(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 1000003 + 7919 * salt + 12345)
    return g


def _axis(n, b, clamp):
    g = torch.arange(n + 2 * b, device="cuda", dtype=torch.float64)
    if clamp:
        g = g.clamp(b, b + n - 1)
    return (g - b + 1) / (n + 1)


def _velocity(kind, n, b, seed, salt=0):
    """float32 velocity on the padded grid ([z, y, x]), nearest value in the padding; the seed moves the model."""
    x = _axis(n, b, True)
    N = n + 2 * b
    u = torch.rand(4, generator=_gen(seed, 100 + salt), device="cuda", dtype=torch.float64)
    if kind == "random":                             # a smooth random medium in [1, 2]: a 16^3 lattice, trilinear
        v = torch.randn((1, 1, 16, 16, 16), generator=_gen(seed, 200 + salt), device="cuda", dtype=torch.float64)
        v = 1.0 + (v - v.min()) / (v.max() - v.min())
        t = 2.0 * x - 1.0
        Z, Y, X = torch.meshgrid(t, t, t, indexing="ij")
        c = torch.nn.functional.grid_sample(v, torch.stack((X, Y, Z), -1)[None], mode="bilinear", align_corners=True)
        return c.reshape(N, N, N).float().contiguous()
    ctr = 0.45 + 0.1 * u[:3]
    r2 = (x - ctr[0])[None, None, :] ** 2 + (x - ctr[1])[None, :, None] ** 2
    if kind == "waveguide":                          # a slow vertical guide
        inside = ((x - ctr[0]).abs() < 0.1)[None, None, :] & ((x - ctr[1]).abs() < 0.1)[None, :, None]
        return torch.where(inside, 0.7, 1.0).expand(N, N, N).float().contiguous()
    if kind == "constant":
        return torch.full((N, N, N), 1.0 + 0.1 * float(u[0]), device="cuda", dtype=torch.float32)
    r2 = r2 + (x - ctr[2])[:, None, None] ** 2
    c = (4.0 / 3.0) * (1.0 - 0.5 * torch.exp(-32.0 * r2))
    if kind == "bump":                               # the lens and a small perturbation
        p = 0.35 + 0.3 * u[1:4]
        q2 = ((x - p[0])[None, None, :] ** 2 + (x - p[1])[None, :, None] ** 2 + (x - p[2])[:, None, None] ** 2)
        c = c + 0.05 * torch.exp(-32.0 * q2)
    return c.float().contiguous()


def _centres(R, seed, salt=0):
    """Source positions near the plane z = 0.1 on a jittered grid, (R, 3) as x, y, z."""
    p = math.ceil(math.sqrt(R))
    u = torch.rand((R, 3), generator=_gen(seed, 300 + salt), device="cuda", dtype=torch.float64)
    i = torch.arange(R, device="cuda")
    xy = torch.stack(((i % p + 0.25 + 0.5 * u[:, 0]) / p, (i // p + 0.25 + 0.5 * u[:, 1]) / p), 1)
    return torch.cat((xy, 0.08 + 0.04 * u[:, 2:3]), 1)


def _sources(n, b, R, seed, salt=0):
    """Gaussian point sources exp(-(4 omega/pi)^2 |x - x_s|^2), zero in the padding: complex64 (R, N, N, N)."""
    a = (4.0 * _omega(n) / math.pi) ** 2
    x = _axis(n, b, False)
    N = n + 2 * b
    phys = torch.zeros(N, device="cuda", dtype=torch.float64)
    phys[b:b + n] = 1.0
    s = _centres(R, seed, salt)
    e = [torch.exp(-a * (x[None, :] - s[:, q:q + 1]) ** 2) * phys for q in range(3)]
    f = torch.empty((R, N, N, N), device="cuda", dtype=torch.complex64)
    for r in range(R):
        f[r] = e[2][r][:, None, None] * e[1][r][None, :, None] * e[0][r][None, None, :]
    return f


def _vectors(n, b, R, seed, salt=0):
    """Vectors an apply or a matvec meets: unit-norm sources (a first residual) in turn with
    oscillating fields of every direction (later basis vectors)."""
    f = _sources(n, b, R, seed, salt)
    om = _omega(n)
    x = _axis(n, b, False)
    u = torch.rand((R, 4), generator=_gen(seed, 400 + salt), device="cuda", dtype=torch.float64)
    for r in range(R):
        if r % 2:
            k = torch.nn.functional.normalize(u[r, :3] - 0.5, dim=0) * om
            w = [torch.polar(0.5 + u[r, 3] * torch.sin(math.pi * x.clamp(0, 1)), k[q] * x) for q in range(3)]
            f[r] = (w[2][:, None, None] * w[1][None, :, None] * w[0][None, None, :]).to(torch.complex64)
        f[r] /= torch.linalg.vector_norm(f[r])
    return f


def _solver(case, c, **over):
    p = dict(case, **over)
    return helm.Solver(c, _omega(p["n"]), p["n"], p["b"], p["d"], b_aux=p["b_aux"], precision=p["precision"],
                       apply_form=p["form"], schedule=p["schedule"])


class _State:
    pass


class _Batch:
    """Three handles served by one batched launch; released together."""

    def __init__(self, case, cs):
        self.S = [helm.Solver(c, _omega(n), n, case["b"], case["d"], precision=case["precision"])
                  for c, (n, _) in zip(cs, _members(case))]


def _members(case):
    return [(case["n"], case["nrhs"]), (case["n2"], case["nrhs2"]), (case["n3"], case["nrhs3"])]


def _receivers(n, b):
    return b - 1 + int(round(0.9 * (n + 1)))         # the grid plane nearest z = 0.9


def _observed(n, b, R, seed):
    """Receiver data of a homogeneous medium: the free-space field of each Gaussian source on the plane."""
    om = _omega(n)
    a = (4.0 * om / math.pi) ** 2
    x = _axis(n, b, False)
    s = _centres(R, seed)
    z = float(x[_receivers(n, b)])
    r = torch.sqrt((x[None, None, :] - s[:, 0, None, None]) ** 2 + (x[None, :, None] - s[:, 1, None, None]) ** 2
                   + (z - s[:, 2, None, None]) ** 2)
    amp = -((math.pi / a) ** 1.5) * math.exp(-om * om / (4.0 * a)) / (4.0 * math.pi * r)
    return torch.polar(amp.abs(), om * r + math.pi).to(torch.complex64)


def prepare(case, seed):
    s = _State()
    s.case, s.kind = case, case["kind"]
    n, b, R = case["n"], case["b"], case["nrhs"]
    if s.kind == "apply":
        s.S = _solver(case, _velocity(case["velocity"], n, b, seed))
        s.r = _vectors(n, b, R, seed)
    elif s.kind == "batch":
        s.B = _Batch(case, [_velocity(v, m, b, seed, q)
                            for q, ((m, _), v) in enumerate(zip(_members(case), ("lens", "waveguide", "random")))])
        s.r = [_vectors(m, b, k, seed, q) for q, (m, k) in enumerate(_members(case))]
    elif s.kind == "matvec":
        # a handle with the cheapest stored form: only its coefficients are used
        s.S = helm.Solver(_velocity("random", n, b, seed), _omega(n), n, b, 1, b_aux=1, precision="fp16")
        s.r = _vectors(n, b, R, seed)
        if case["fp64"]:
            s.r = s.r.to(torch.complex128)
    elif s.kind == "solve":
        s.S = _solver(case, _velocity(case["velocity"], n, b, seed))
        s.r = _sources(n, b, R, seed)
    elif s.kind == "setup":
        s.c = _velocity(case["velocity"], n, b, seed)
        s.r = _vectors(n, b, R, seed)
    else:
        s.c = _velocity(case["velocity"], n, b, seed).requires_grad_(True)
        s.r = _sources(n, b, R, seed)
        s.obs = _observed(n, b, R, seed)
        s.plane = _receivers(n, b)
    return s


# -------------------------------------------------------------------- the pass

def run(s):
    case = s.case
    if s.kind == "apply":
        return s.S.apply(s.r)
    if s.kind == "batch":
        z = [torch.empty_like(r) for r in s.r]
        helm.helm_apply_batch([S.handle for S in s.B.S], [r.data_ptr() for r in s.r], [t.data_ptr() for t in z],
                              [r.shape[0] for r in s.r], torch.cuda.current_stream().cuda_stream)
        return z
    if s.kind == "matvec":
        return s.S.matvec(s.r)
    if s.kind == "solve":
        return s.S.solve(s.r, tol=TOL)[0]
    if s.kind == "setup":
        S = _solver(case, s.c)
        z = S.apply(s.r)
        S.close()
        return z
    u = helmholtz_solve(s.c, s.r, _omega(case["n"]), case["n"], case["b"], case["d"], TOL, case["precision"],
                        case["b_aux"])
    misfit = u[:, s.plane] - s.obs
    loss = 0.5 * (misfit.real.square().sum() + misfit.imag.square().sum())
    (grad,) = torch.autograd.grad(loss, s.c)
    return {"grad": grad, "u": u.detach()}


# -------------------------------------------- the least bytes and operations

def _blocks(N, b, d, two):
    """(first layer, end, role) of the swept-axis blocks, and the index of the centre."""
    if two:
        q = (N - 2 * b - 1) // (2 * d)
        lo = [(0, b, "L")] + [(b + i * d, b + (i + 1) * d, "L") for i in range(q)]
        hi = [(N - b - (i + 1) * d, N - b - i * d, "U") for i in range(q - 1, -1, -1)] + [(N - b, N, "U")]
        return lo + [(b + q * d, N - b - q * d, "C")] + hi, q + 1
    out, m = [(0, b, "L")], b
    while m < N:
        out.append((m, min(m + d, N), "L"))
        m += d
    out[-1] = out[-1][:2] + ("C",)
    return out, len(out) - 1


def _windows(N, b, d, b_aux, two):
    """Per block: (lo, L, ia, ib, moving low side, moving high side)."""
    out = []
    blocks, cen = _blocks(N, b, d, two)
    for m, e, role in blocks:
        ml, mh = role != "U" and m > 0, role != "L" and e < N
        lo, hi = (m - b_aux if ml else m), (e + b_aux if mh else e)
        if lo < 0:
            lo, ml = 0, False
        if hi > N:
            hi, mh = N, False
        out.append((lo, hi - lo, m - lo, e - lo, ml, mh))
    return out, cen


def _sweep_work(n, b, d, b_aux, two, form, precision, R):
    """Stored bytes of the preconditioner (each read at least once) and the flops of one apply."""
    N = n + 2 * b
    win, cen = _windows(N, b, d, b_aux or b, two)
    B = len(win)
    stored = flops = 0
    for M, (_, Lz, za, zb, _, _) in enumerate(win):
        slab_uses = 1 if M == cen else 2
        for Mp, (_, Ly, ya, yb, _, _) in enumerate(win):
            uses = 1 if Mp == cen else 2
            if form == "chain":
                k = Ly * Lz
                stored += N * k * k * (4 if precision == "fp16" else 8)
                flops += slab_uses * uses * 2 * N * k * k * 8 * R
                continue
            per = 4 if precision == "fp16" else 8
            nl = yb - ya
            if Mp == 0 or (two and Mp == B - 1):     # a boundary block's two maps
                n_in, n_out = nl * (zb - za) * N, ((nl - 1) * (zb - za) + Lz) * N
                b_in, b_out = Lz * N, nl * (zb - za) * N
                stored += per * (n_in * n_out + b_in * b_out)
                flops += slab_uses * 8 * R * (n_in * n_out + b_in * b_out)
            else:
                m = nl * Lz * N
                stored += per * m * m
                flops += slab_uses * uses * 8 * R * m * m
    return stored, flops


def work(case):
    n, b, R, kind = case["n"], case["b"], case["nrhs"], case["kind"]
    N3 = (n + 2 * b) ** 3
    if kind == "matvec":
        e = 16 if case["fp64"] else 8
        return {"bytes": 2 * e * N3 * R + e // 2 * N3, "flops": 62 * N3 * R}
    if kind == "batch":
        by = fl = 0
        for m, k in _members(case):
            s, f = _sweep_work(m, b, case["d"], 0, False, "chain", case["precision"], k)
            by, fl = by + s + 16 * k * (m + 2 * b) ** 3, fl + f
        return {"bytes": by, "flops": fl}
    form = case.get("form", "chain")
    s, f = _sweep_work(n, b, case["d"], case["b_aux"], case.get("schedule") == "two_front", form, case["precision"], R)
    if kind == "apply":
        return {"bytes": s + 16 * R * N3, "flops": f}
    if kind == "setup":                              # operators written once; the first apply reads them
        return {"bytes": 2 * s + 4 * N3 + 16 * R * N3, "flops": f}
    # a solve takes about n/4 + 3 iterations: each reads the operators and the new vectors, and the basis twice
    its = n // 4 + 3
    one = its * (s + 16 * R * N3) + 16 * R * N3 * its * (its + 1) // 2
    fl = its * f
    if kind == "solve":
        return {"bytes": one, "flops": fl}
    return {"bytes": 2 * one + s + 12 * N3, "flops": 2 * fl}


# ------------------------------------------------------- the result in 64 bits

class _Exact:
    """The PML operator and the recursive sweep in complex128, slab by slab: every quasi-1D problem's
    restricted inverse as a dense matrix, formed for all line blocks of a slab at once."""

    def __init__(self, c, n, b, d=1, b_aux=0, two=False):
        self.n, self.b, self.N, self.omega = n, b, n + 2 * b, _omega(n)
        self.h, self.b_aux = 1.0 / (n + 1), b_aux or b
        self.kappa = (self.omega / c.double()) ** 2
        g = torch.arange(self.N, device="cuda", dtype=torch.float64)
        self.cdn, self.cup = self._couplings(g, self._sigma_global)
        self.win, self.cen = _windows(self.N, b, d, self.b_aux, two)
        self.blk, _ = _blocks(self.N, b, d, two)
        self.ycpl = self._line_couplings()

    def _pml(self, t, eta):
        return torch.where((t >= 0) & (t <= eta), PML_C / eta * ((t - eta) / eta) ** 2, torch.zeros_like(t))

    def _sigma_global(self, p):
        eta = self.b * self.h
        return self._pml((p + 1) * self.h, eta) + self._pml((self.N - p) * self.h, eta)

    def _sigma_window(self, w):
        lo, L, _, _, ml, mh = w
        eta, aux = self.b * self.h, self.b_aux * self.h

        def fn(p):
            low = self._pml((p - (lo - 1)) * self.h, aux) if ml else self._pml((p + 1) * self.h, eta)
            return low + (self._pml((lo + L - p) * self.h, aux) if mh else self._pml((self.N - p) * self.h, eta))
        return fn

    def _s(self, sigma):
        return 1.0 / (1.0 + 1j * sigma / self.omega)

    def _couplings(self, g, fn):
        s = self._s(fn(g))
        return s * self._s(fn(g - 0.5)) / self.h ** 2, s * self._s(fn(g + 0.5)) / self.h ** 2

    def matvec(self, u):
        out = self.kappa * u
        for ax in (1, 2, 3):
            sh = [1, 1, 1, 1]
            sh[ax] = self.N
            up, dn = self.cup.reshape(sh), self.cdn.reshape(sh)
            z = torch.zeros_like(u.narrow(ax, 0, 1))
            out = out + up * (torch.cat((u.narrow(ax, 1, self.N - 1), z), ax) - u)
            out = out - dn * (u - torch.cat((z, u.narrow(ax, 0, self.N - 1)), ax))
        return out

    def _line_couplings(self):
        """(ydn, yup) over the window of every line block."""
        out = []
        for w in self.win:
            y = torch.arange(w[0], w[0] + w[1], device="cuda", dtype=torch.float64)
            out.append(self._couplings(y, self._sigma_window(w)))
        return out

    def _operators(self, M):
        """[line block] -> matrix over (line, window z, x) of the block's own lines."""
        lo, Lz = self.win[M][:2]
        z = torch.arange(lo, lo + Lz, device="cuda", dtype=torch.float64)
        zdn, zup = self._couplings(z, self._sigma_window(self.win[M]))
        kz = torch.diag(zup[:-1], 1) + torch.diag(zdn[1:], -1)
        eye = torch.eye(Lz, dtype=torch.complex128, device="cuda")
        out, groups = {}, {}
        for Mp, w in enumerate(self.win):
            groups.setdefault((w[1], w[2], w[3]), []).append(Mp)
        for (Ly, ya, yb), Mps in groups.items():
            k, nb, N = Ly * Lz, len(Mps), self.N
            ydn = torch.stack([self.ycpl[Mp][0] for Mp in Mps])
            yup = torch.stack([self.ycpl[Mp][1] for Mp in Mps])
            ky = torch.diag_embed(yup[:, :-1], 1) + torch.diag_embed(ydn[:, 1:], -1)
            eyy = torch.eye(Ly, dtype=torch.complex128, device="cuda")
            base = (torch.einsum("nab,ij->naibj", ky, eye) + torch.einsum("ab,ij->aibj", eyy, kz)).reshape(nb, k, k)
            lines = torch.tensor([self.win[Mp][0] for Mp in Mps], device="cuda")[:, None] + torch.arange(Ly, device="cuda")
            diag = (self.kappa[lo:lo + Lz][:, lines].permute(1, 2, 0, 3) - (self.cdn + self.cup)
                    - (ydn + yup)[:, :, None, None] - (zdn + zup)[:, None]).reshape(nb, k, N)
            rows = torch.arange(ya * Lz, yb * Lz, device="cuda")
            m = len(rows)
            ncol = m * N
            y = torch.zeros((N, nb, k, ncol), dtype=torch.complex128, device="cuda")
            T = None
            Ts = []
            for i in range(N):
                S = base + torch.diag_embed(diag[:, :, i])
                if i:
                    S = S - self.cdn[i] * self.cup[i - 1] * T
                T = torch.linalg.inv(S)
                Ts.append(T)
                if i:                                 # columns of x < i carry the elimination, x = i the unit entries
                    y[i, :, :, :i * m] = T @ (-self.cdn[i] * y[i - 1, :, :, :i * m])
                y[i, :, :, i * m:(i + 1) * m] = T[:, :, rows]
            G = torch.empty((nb, m, N, ncol), dtype=torch.complex128, device="cuda")
            x = y[N - 1]
            G[:, :, N - 1] = x[:, rows]
            for i in range(N - 2, -1, -1):
                x = y[i] - self.cup[i] * (Ts[i] @ x)
                G[:, :, i] = x[:, rows]
            # columns (x, line, z) -> (line, z, x)
            G = G.reshape(nb, m * N, N, m).transpose(2, 3).reshape(nb, m * N, m * N)
            for q, Mp in enumerate(Mps):
                out[Mp] = G[q]
        return out

    def _pass(self, solve, g):
        """One block sweep over the leading axis of g (block axis first), v the same shape."""
        v = torch.zeros_like(g)
        B, c = len(self.blk), self.cen
        for M in list(range(c)) + list(range(B - 1, c, -1)) + [c]:
            m, e, _ = self.blk[M]
            r = g[m:e].clone()
            if 0 < M <= c:
                r[0] -= self.cdn[m] * v[m - 1]
            if c <= M < B - 1:
                r[-1] -= self.cup[e - 1] * v[e]
            v[m:e] = solve(M, r)
        for M in list(range(c - 1, -1, -1)) + list(range(c + 1, B)):
            m, e, _ = self.blk[M]
            r = torch.zeros_like(g[m:e])
            if M < c:
                r[-1] = self.cup[e - 1] * v[e]
            else:
                r[0] = self.cdn[m] * v[m - 1]
            v[m:e] -= solve(M, r)
        return v

    def apply(self, f):
        """M f for f (R, z, y, x)."""
        R, N = f.shape[0], self.N
        keep = {}
        per = 16.0 * (max(w[3] - w[2] for w in self.win[1:-1]) * max(w[1] for w in self.win[1:-1]) * N) ** 2
        cache = per * len(self.win) ** 2 < 60e9      # both visits of a slab share its operators where they fit

        def slab(M, r):                               # r: (own layers, y, x, R)
            G = keep.get(M) or self._operators(M)
            if cache:
                keep[M] = G
            _, Lz, za, zb, _, _ = self.win[M]
            g = torch.zeros((N, Lz, N, R), dtype=torch.complex128, device="cuda")
            g[:, za:zb] = r.transpose(0, 1)
            v = self._pass(lambda Mp, t: (G[Mp] @ t.reshape(-1, R)).reshape(t.shape), g)
            return v[:, za:zb].transpose(0, 1)
        return self._pass(slab, f.permute(1, 2, 3, 0).contiguous()).permute(3, 0, 1, 2)

    def _planes(self):
        """Block elimination along z: the inverses of the plane Schur complements."""
        N = self.N
        P = N * N
        plane = torch.zeros((N, N, N, N), dtype=torch.complex128, device="cuda")
        i = torch.arange(N, device="cuda")
        for q in range(N):
            plane[q, i[:-1], q, i[1:]] += self.cup[:-1]
            plane[q, i[1:], q, i[:-1]] += self.cdn[1:]
            plane[i[:-1], q, i[1:], q] += self.cup[:-1]
            plane[i[1:], q, i[:-1], q] += self.cdn[1:]
        plane = plane.reshape(P, P)
        s = self.cdn + self.cup
        T = []
        for z in range(N):
            S = plane.clone()
            S.diagonal().add_((self.kappa[z] - s[z] - s[:, None] - s[None, :]).reshape(P))
            if z:
                S -= self.cdn[z] * self.cup[z - 1] * T[-1]
            T.append(torch.linalg.inv(S))
        return T

    def solve(self, f, adjoint=False, T=None):
        """A^-1 f, or A^-T f (the same elimination transposed)."""
        R, N = f.shape[0], self.N
        T = T or self._planes()
        q = f.reshape(R, N, N * N).permute(1, 2, 0)
        dn, up = (self.cup.roll(1), self.cdn.roll(-1)) if adjoint else (self.cdn, self.cup)
        y = []
        for z in range(N):
            t = q[z] if z == 0 else q[z] - dn[z] * y[-1]
            y.append((T[z].transpose(0, 1) if adjoint else T[z]) @ t)
        x = [y[-1]]
        for z in range(N - 2, -1, -1):
            x.append(y[z] - (T[z].transpose(0, 1) if adjoint else T[z]) @ (up[z] * x[-1]))
        return torch.stack(x[::-1]).permute(2, 0, 1).reshape(R, N, N, N), T


def exact(case, seed):
    kind, n, b = case["kind"], case["n"], case["b"]
    if kind == "solve" and n + 2 * b > 43:           # the direct solve of a larger grid takes minutes
        return None
    if kind == "batch":
        out = []
        for q, ((m, k), v) in enumerate(zip(_members(case), ("lens", "waveguide", "random"))):
            X = _Exact(_velocity(v, m, b, seed, q), m, b, case["d"])
            out.append(X.apply(_vectors(m, b, k, seed, q).to(torch.complex128)))
        return out
    if kind == "matvec":
        return _Exact(_velocity("random", n, b, seed), n, b).matvec(
            _vectors(n, b, case["nrhs"], seed).to(torch.complex128))
    c = _velocity(case["velocity"], n, b, seed)
    if kind in ("apply", "setup"):
        X = _Exact(c, n, b, case["d"], case["b_aux"], case["schedule"] == "two_front")
        return X.apply(_vectors(n, b, case["nrhs"], seed).to(torch.complex128))
    X = _Exact(c, n, b)
    u, T = X.solve(_sources(n, b, case["nrhs"], seed).to(torch.complex128))
    if kind == "solve":
        return u
    g = torch.zeros_like(u)
    plane = _receivers(n, b)
    g[:, plane] = (u[:, plane] - _observed(n, b, case["nrhs"], seed)).conj()
    lam, _ = X.solve(g, adjoint=True, T=T)
    return {"grad": (lam * u).real.sum(0) * 2.0 * X.omega ** 2 / c.double() ** 3, "u": u}
