"""What a user of this framework has it do, as measurable cases.

Every case goes through the public binding (``paper_2005_13425_gb300.nekgb``):
the operator on one box, CG solves (plain FP64, Jacobi from host buffers,
mixed precision), and the batched engine.  ``prepare`` sets up what a user's
program holds before the call (context or engine, inputs on the device, or on
the host where the entry point takes host buffers), ``run`` is one call or
one served batch, and ``exact`` restates the mathematics (GLL nodes, box
geometry, operator, CG) in 64 bits with plain torch and numpy.  ``iters`` of
a case that runs to a tolerance is about what it takes (``work`` counts it).

Inputs are those of the framework's own workloads: a unit-cube box whose mesh
is perturbed by 0.05 s_d sin sin sin, fields uniform in [-1, 1], right-hand
sides continuous and masked.
"""
import math
import os
import random
import tempfile

import numpy as np
import torch

from paper_2005_13425_gb300 import nekgb

AMP = 0.05
DEGREES = (6, 8, 10, 12)     # GLL points per direction of served requests


def listed():
    return [
        # one operator application on the smallest configured box (Nekbone's
        # 64-element run): launches and latency count
        dict(name="apply_4x4x4_n8", kind="apply", ex=4, ey=4, ez=4, n=8),
        # the paper's headline operator: 4096 elements of degree 9
        dict(name="apply_16x16x16_n10", kind="apply", ex=16, ey=16, ez=16, n=10),
        # a ragged box of odd order, the element operator alone
        dict(name="ax_13x11x7_n9", kind="ax", ex=13, ey=11, ez=7, n=9),
        # the largest box that is served
        dict(name="apply_32x32x32_n12", kind="apply", ex=32, ey=32, ez=32, n=12),
        # the highest supported order
        dict(name="apply_9x8x7_n16", kind="apply", ex=9, ey=8, ez=7, n=16),
        # the single-precision operator (ax_e and dssum) of mixed solves
        dict(name="ax_f32_16x16x8_n10", kind="ax_f32", ex=16, ey=16, ez=8, n=10),
        # Nekbone's own run: 100 fixed CG iterations on 64 elements
        dict(name="cg_4x4x4_n8", kind="cg", ex=4, ey=4, ez=4, n=8, iters=100),
        # the headline solve: fixed CG iterations, 4096 elements of degree 9
        dict(name="cg_16x16x16_n10", kind="cg", ex=16, ey=16, ez=16, n=10, iters=100),
        # a Jacobi-preconditioned solve to a tolerance on a ragged box, from
        # and to host buffers
        dict(name="jacobi_host_9x7x5_n7", kind="jacobi_host", ex=9, ey=7, ez=5, n=7, tol=1e-10, iters=290),
        # mixed precision to an FP64 tolerance at full size
        dict(name="mixed_16x16x16_n8", kind="mixed", ex=16, ey=16, ez=16, n=8, tol=1e-10, iters=1210),
        # a batch of uneven FP64 requests: submit, advance, retire
        dict(name="engine_fp64_32", kind="engine", mixed=False, count=32, list_seed=4, e_lo=64, e_hi=4096, iters=100),
        # served mixed-precision requests, stepped until each has converged
        dict(name="engine_mixed_12", kind="engine", mixed=True, count=12, list_seed=5, e_lo=64, e_hi=1024,
             tol=1e-10, iters=900),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _dims(rng, elements):
    """Box dimensions of about `elements` elements, sides within a factor of two of a cube's."""
    side = max(1.0, elements) ** (1.0 / 3.0)
    ex = max(1, round(side * 2.0 ** rng.uniform(-0.7, 0.7)))
    ey = max(1, round(side * 2.0 ** rng.uniform(-0.7, 0.7)))
    ez = max(1, round(elements / (ex * ey)))
    return ex, ey, ez


def draw(rng):
    kind = rng.choice(["apply", "apply", "ax", "ax_f32", "cg", "cg", "jacobi_host", "mixed", "engine"])
    if kind in ("apply", "ax", "ax_f32"):
        n = rng.randint(2, 16)
        ex, ey, ez = _dims(rng, min(30000.0, _log_uniform(rng, 1.5e4, 3e7) / n ** 3))
        return dict(kind=kind, ex=ex, ey=ey, ez=ez, n=n)
    if kind == "cg":
        n = rng.randint(4, 14)
        ex, ey, ez = _dims(rng, max(27.0, _log_uniform(rng, 2e4, 4e6) / n ** 3))
        return dict(kind=kind, ex=ex, ey=ey, ez=ez, n=n, iters=rng.randint(20, 100))
    if kind in ("jacobi_host", "mixed"):
        n = rng.randint(5, 12)
        ex, ey, ez = _dims(rng, max(27.0, _log_uniform(rng, 2e4, 1e6) / n ** 3))
        return dict(kind=kind, ex=ex, ey=ey, ez=ez, n=n, tol=1e-10, iters=4 * n * max(ex, ey, ez) + 60)
    mixed = rng.random() < 0.5
    case = dict(kind="engine", mixed=mixed, count=rng.randint(4, 12 if mixed else 32), list_seed=rng.randrange(1 << 20),
                e_lo=64, e_hi=1024 if mixed else 4096, iters=900 if mixed else rng.randint(24, 100))
    if mixed:
        case["tol"] = 1e-10
    return case


def _problems(case):
    """Boxes and orders of an engine case: element counts log-uniform, rounded to
    powers of two per side, orders from DEGREES."""
    rng = random.Random(case["list_seed"])
    out = []
    for _ in range(case["count"]):
        k = round(math.log2(_log_uniform(rng, case["e_lo"], case["e_hi"])))
        c = k // 3
        a, b = c + (k % 3 >= 1), c + (k % 3 >= 2)
        out.append(((1 << a, 1 << b, 1 << c), rng.choice(DEGREES)))
    return out


# ------------------------------------------------------------------ inputs
def _coeffs(seed):
    return np.random.default_rng(seed).uniform(-1.0, 1.0, size=3)


def _uniform(shape, seed, dtype=torch.float64):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.empty(shape, dtype=dtype, device="cuda").uniform_(-1.0, 1.0, generator=g)


def _unique_field(dims, n, seed):
    """Uniform values per unique node, x fastest, zero on the faces of the box."""
    nz, ny, nx = (dims[2] * (n - 1) + 1, dims[1] * (n - 1) + 1, dims[0] * (n - 1) + 1)
    f = torch.zeros(nz, ny, nx, dtype=torch.float64, device="cuda")
    f[1:-1, 1:-1, 1:-1] = _uniform((nz - 2, ny - 2, nx - 2), seed)
    return f.reshape(-1)


def _gid(dims, n):
    """Unique-node index of every local point, [E * n^3]."""
    ex, ey, ez = dims
    ax = [(torch.arange(e, device="cuda")[:, None] * (n - 1) + torch.arange(n, device="cuda")) for e in (ex, ey, ez)]
    nx, ny = ex * (n - 1) + 1, ey * (n - 1) + 1
    gx = ax[0][None, None, :, None, None, :]
    gy = ax[1][None, :, None, None, :, None]
    gz = ax[2][:, None, None, :, None, None]
    return (gx + nx * (gy + ny * gz)).reshape(-1)


class _Context:
    """A context of the library, destroyed with its owner."""

    def __init__(self, dims, n, s, prec, stream):
        self.h = nekgb.nb_setup_box(dims, n, AMP, s, prec, stream)

    def __del__(self):
        nekgb.nb_destroy(self.h)


class _Engine:
    def __init__(self, arena, stream):
        self.h = nekgb.nb_engine_create(arena, stream)

    def __del__(self):
        nekgb.nb_engine_destroy(self.h)


def prepare(case, seed):
    kind = case["kind"]
    stream = torch.cuda.Stream()
    st = dict(case=case, stream=stream)
    if kind == "engine":
        # a serving program keeps the tuner's choices in a file
        os.environ.setdefault("NEKGB_TUNE_CACHE",
                              os.path.join(tempfile.gettempdir(), "nekgb_tune_%d" % os.getpid()))
        prec = nekgb.NB_MIXED if case["mixed"] else nekgb.NB_FP64
        probs = _problems(case)
        st["prec"], st["probs"] = prec, probs
        st["s"] = [_coeffs((seed, i)) for i in range(len(probs))]
        st["f"] = [_unique_field(d, n, seed * 1009 + i) for i, (d, n) in enumerate(probs)]
        st["x"] = [torch.empty(d[0] * d[1] * d[2], n ** 3, dtype=torch.float64, device="cuda") for d, n in probs]
        need = sum(nekgb.nb_engine_footprint(d, n, prec) for d, n in probs)
        torch.cuda.synchronize()
        st["eng"] = _Engine(need + need // 8 + (64 << 20), stream)
        for n in sorted({n for _, n in probs}):      # each order's first request chooses its layout
            i = next(k for k, p in enumerate(probs) if p[1] == n)
            _, rid = nekgb.nb_engine_submit_unique(st["eng"].h, probs[i][0], n, AMP, st["s"][i], 0.0, 8,
                                                   st["f"][i], prec=prec)
            nekgb.nb_engine_step(st["eng"].h, 8)
            nekgb.nb_engine_retire(st["eng"].h, rid)
        return st
    dims, n = (case["ex"], case["ey"], case["ez"]), case["n"]
    E = dims[0] * dims[1] * dims[2]
    mixed = kind in ("mixed", "ax_f32")
    st["ctx"] = _Context(dims, n, _coeffs(seed), nekgb.NB_MIXED if mixed else nekgb.NB_FP64, stream)
    if kind in ("apply", "ax", "ax_f32"):
        dtype = torch.float32 if kind == "ax_f32" else torch.float64
        st["u"] = _uniform((E, n ** 3), seed, dtype)
        st["w"] = torch.empty_like(st["u"])
    else:
        st["f"] = _unique_field(dims, n, seed)[_gid(dims, n)].reshape(E, n ** 3)
        if kind == "jacobi_host":
            nekgb.nb_set_preconditioner(st["ctx"].h, 1)
            st["f"] = st["f"].cpu().pin_memory().numpy()
            st["x"] = torch.zeros(E, n ** 3, dtype=torch.float64).pin_memory().numpy()
    torch.cuda.synchronize()
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "engine":
        return _serve(st)
    ctx = st["ctx"].h
    if kind == "apply":
        nekgb.nb_apply(ctx, st["u"], st["w"])
        return st["w"]
    if kind == "ax":
        nekgb.nb_ax(ctx, st["u"], st["w"])
        return st["w"]
    if kind == "ax_f32":
        nekgb.nb_ax_f32(ctx, st["u"], st["w"])
        nekgb.nb_dssum_f32(ctx, st["w"])
        return st["w"]
    if kind == "jacobi_host":
        st["x"].fill(0.0)
        nekgb.nb_cg_solve_host(ctx, st["f"], st["x"], tol=case["tol"], maxit=20000)
        return st["x"]
    with torch.cuda.stream(st["stream"]):
        x = torch.zeros_like(st["f"])
        if kind == "mixed":
            nekgb.nb_cg_solve(ctx, st["f"], x, tol=case["tol"], maxit=20000)
        else:
            nekgb.nb_cg_solve(ctx, st["f"], x, tol=0.0, maxit=case["iters"])
    return x


def _serve(st):
    """All requests submitted, advanced together and retired into the user's buffers."""
    case, eng = st["case"], st["eng"].h
    tol, maxit = (case["tol"], 20000) if case["mixed"] else (0.0, case["iters"])
    ids = []
    for (dims, n), s, f in zip(st["probs"], st["s"], st["f"]):
        ids.append(nekgb.nb_engine_submit_unique(eng, dims, n, AMP, s, tol, maxit, f, prec=st["prec"])[1])
    if case["mixed"]:
        live = set(range(len(ids)))
        while live:
            nekgb.nb_engine_step(eng, 16)
            for k in sorted(live):
                if nekgb.nb_engine_poll(eng, ids[k])[0]:
                    nekgb.nb_engine_retire(eng, ids[k], st["x"][k])
                    live.discard(k)
    else:
        nekgb.nb_engine_step(eng, case["iters"])
        for rid, x in zip(ids, st["x"]):
            nekgb.nb_engine_retire(eng, rid, x)
    return st["x"]


# ------------------------------------------------------------------ work
ON_CHIP = 120e6     # bytes of solver state that stay in L2 between iterations


def _solve_work(points, n, iters, single):
    """CG with the geometric factors (6 values), r, p and x per point: from memory
    in every iteration, or once where the whole state stays on chip."""
    size = 4 if single else 8
    passes = iters if 10 * size * points > ON_CHIP else 1
    return dict(bytes=points * (passes * 12 * size + 16), flops=points * iters * (12 * n + 25))


def work(case):
    kind = case["kind"]
    if kind == "engine":
        probs = _problems(case)
        total = sum(d[0] * d[1] * d[2] * n ** 3 for d, n in probs)
        size = 4 if case["mixed"] else 8
        passes = case["iters"] if 10 * size * total > ON_CHIP else 1
        return dict(bytes=total * (passes * 12 * size + 16),
                    flops=sum(d[0] * d[1] * d[2] * n ** 3 * case["iters"] * (12 * n + 25) for d, n in probs))
    n = case["n"]
    points = case["ex"] * case["ey"] * case["ez"] * n ** 3
    if kind in ("apply", "ax", "ax_f32"):
        size = 4 if kind == "ax_f32" else 8
        return dict(bytes=8 * size * points, flops=points * (12 * n + 15))
    return _solve_work(points, n, case["iters"], kind == "mixed")


# ------------------------------------------------------------------ exact
def _gll(n):
    """GLL nodes, weights and derivative matrix on [-1, 1]."""
    L = np.polynomial.legendre.Legendre.basis(n - 1)
    d1, d2 = L.deriv(), L.deriv(2)
    x = np.concatenate([[-1.0], np.sort(d1.roots().real) if n > 2 else [], [1.0]])
    for _ in range(3):
        x[1:-1] -= d1(x[1:-1]) / d2(x[1:-1])
    w = 2.0 / (n * (n - 1) * L(x) ** 2)
    D = np.zeros((n, n))
    for i in range(n):
        for j in range(n):
            if i != j:
                D[i, j] = L(x[i]) / (L(x[j]) * (x[i] - x[j]))
    D[0, 0], D[-1, -1] = -n * (n - 1) / 4.0, n * (n - 1) / 4.0
    return x, w, D


def _derivatives(D, u, n):
    """(d/dr, d/ds, d/dt) of u [E, n, n, n] (t, s, r)."""
    return (torch.matmul(u, D.T), torch.matmul(D, u),
            torch.matmul(D, u.reshape(-1, n, n * n)).reshape(u.shape))


class _Box:
    """The assembled Poisson operator of a perturbed box in 64 bits."""

    def __init__(self, dims, n, s):
        self.dims, self.n = dims, n
        x, w, D = _gll(n)
        self.D = torch.from_numpy(D).cuda()
        xt, wt = torch.from_numpy(x).cuda(), torch.from_numpy(w).cuda()
        ex, ey, ez = dims
        ax = [(torch.arange(e, device="cuda", dtype=torch.float64)[:, None] + (xt + 1.0) / 2.0) / e for e in dims]
        shape = (ez, ey, ex, n, n, n)
        X = [ax[0][None, None, :, None, None, :].expand(shape), ax[1][None, :, None, None, :, None].expand(shape),
             ax[2][:, None, None, :, None, None].expand(shape)]
        bump = torch.sin(math.pi * X[0]) * torch.sin(math.pi * X[1]) * torch.sin(math.pi * X[2])
        J = [_derivatives(self.D, (X[d] + AMP * float(s[d]) * bump).reshape(-1, n, n, n), n) for d in range(3)]
        c = [[J[(d + 1) % 3][(k + 1) % 3] * J[(d + 2) % 3][(k + 2) % 3] -
              J[(d + 1) % 3][(k + 2) % 3] * J[(d + 2) % 3][(k + 1) % 3] for d in range(3)] for k in range(3)]
        det = J[0][0] * c[0][0] + J[1][0] * c[0][1] + J[2][0] * c[0][2]
        scale = (wt[:, None, None] * wt[:, None] * wt) / det
        del J, det, bump
        self.g = [[sum(c[a][d] * c[b][d] for d in range(3)) * scale if a <= b else None for b in range(3)]
                  for a in range(3)]

    def ax(self, u):
        n = self.n
        u = u.reshape(-1, n, n, n)
        v = _derivatives(self.D, u, n)
        f = [sum(self.g[min(a, b)][max(a, b)] * v[b] for b in range(3)) for a in range(3)]
        out = torch.matmul(f[0], self.D) + torch.matmul(self.D.T, f[1])
        out += torch.matmul(self.D.T, f[2].reshape(-1, n, n * n)).reshape(out.shape)
        return out.reshape(-1)

    def numbering(self):
        self.gid = _gid(self.dims, self.n)
        self.nodes = math.prod(e * (self.n - 1) + 1 for e in self.dims)

    def assemble(self, w):
        return torch.zeros(self.nodes, dtype=torch.float64, device="cuda").index_add_(0, self.gid, w)

    def mask(self, g):
        nx, ny, nz = (e * (self.n - 1) + 1 for e in self.dims)
        v = g.view(nz, ny, nx)
        for face in (v[0], v[-1], v[:, 0], v[:, -1], v[:, :, 0], v[:, :, -1]):
            face.zero_()
        return g

    def apply(self, g):
        """On unique-node values."""
        return self.mask(self.assemble(self.ax(g[self.gid])))


def _cg(A, f, iters, tol=0.0):
    """Plain CG from zero; `iters` iterations, or fewer once the residual is below tol."""
    x, r = torch.zeros_like(f), f.clone()
    p, rho, f2 = torch.zeros_like(f), torch.dot(f, f), float(torch.dot(f, f))
    old = None
    for k in range(iters):
        if tol and k % 16 == 0 and float(rho) <= tol * tol * f2:
            break
        p = r + (rho / old) * p if old is not None else r.clone()
        w = A(p)
        alpha = rho / torch.dot(w, p)
        x += alpha * p
        r -= alpha * w
        old, rho = rho, torch.dot(r, r)
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "engine":
        out = []
        for i, (dims, n) in enumerate(_problems(case)):
            box = _Box(dims, n, _coeffs((seed, i)))
            box.numbering()
            f = _unique_field(dims, n, seed * 1009 + i)
            x = _cg(box.apply, f, 4000, 1e-13) if case["mixed"] else _cg(box.apply, f, case["iters"])
            out.append(x[box.gid].reshape(-1, n ** 3))
        return out
    dims, n = (case["ex"], case["ey"], case["ez"]), case["n"]
    E = dims[0] * dims[1] * dims[2]
    box = _Box(dims, n, _coeffs(seed))
    if kind in ("apply", "ax", "ax_f32"):
        u = _uniform((E, n ** 3), seed, torch.float32 if kind == "ax_f32" else torch.float64)
        w = box.ax(u.double())
        if kind != "ax":
            box.numbering()
            g = box.assemble(w)
            w = (box.mask(g) if kind == "apply" else g)[box.gid]
        return w.reshape(E, n ** 3)
    box.numbering()
    f = _unique_field(dims, n, seed)
    x = _cg(box.apply, f, case["iters"]) if kind == "cg" else _cg(box.apply, f, 4000, 1e-13)
    return x[box.gid].reshape(E, n ** 3)
