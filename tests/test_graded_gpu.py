"""The fixed-point operator on graded elements (an entry, a corner or a factor far
above the rest), which it computes in double-float arithmetic.

Tolerance.  Double-float pairs hold 46 bits of an input and 47 of D and gxyz, and
a compensated product sum of n terms rounds at about 2^-47 of its terms' absolute
sum.  Through the three stages (derivative, contraction, transposed derivative) at
most nine such errors add up at a point, each relative to the operator of
absolute values there (with even-odd lines those of the mirrored entries
too): 9 2^-46 < 2^-42.8.  2^-42 of that operator is the bound.  One scale for an
element gives an absolute error of about 2^-52 of the largest result instead,
which at 1e-3 of the peak is already ten times the bound, at 1e-12 all of the result.
"""
import numpy as np
import pytest

from paper_2005_13425_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BOUND = 2.0 ** -42


@pytest.fixture(scope="module")
def nek():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_13425_gb300 import build as b
    b.build()
    from paper_2005_13425_gb300 import nekgb
    nekgb.load()
    torch.cuda.set_stream(torch.cuda.Stream())
    return nekgb


def absolute_operator(D, gxyz, u, mirrored):
    """The operator of absolute values, [E, n^3]; mirrored: of the even-odd lines."""
    n = D.shape[0]
    A = np.abs(D)
    if mirrored:
        A = A + A[::-1] + A[:, ::-1] + A[::-1, ::-1]
    g = np.abs(gxyz).reshape(-1, 6, n, n, n)
    v = np.abs(u).reshape(-1, n, n, n)
    d = [np.einsum("il,etsl->etsi", A, v), np.einsum("il,etlr->etir", A, v), np.einsum("il,elsr->eisr", A, v)]
    f = [g[:, 0] * d[0] + g[:, 1] * d[1] + g[:, 2] * d[2], g[:, 1] * d[0] + g[:, 3] * d[1] + g[:, 4] * d[2],
         g[:, 2] * d[0] + g[:, 4] * d[1] + g[:, 5] * d[2]]
    out = np.einsum("li,etsl->etsi", A, f[0]) + np.einsum("li,etlr->etir", A, f[1]) + \
        np.einsum("li,elsr->eisr", A, f[2])
    return out.reshape(u.shape)


def graded(kind, P, n):
    """D, gxyz and an input; the elements with an even index are graded."""
    D, g = P["D"].copy(), P["gxyz"].reshape(P["E"], 6, n ** 3).copy()
    u = inputs.local_field(P["E"], n, seed=n + 5)
    even = np.arange(0, P["E"], 2)
    t = np.linspace(0.0, 1.0, n)
    ramp = (t[:, None, None] + t[:, None] + t).reshape(-1)      # 0 at one corner, 3 at the other
    if kind == "spike":
        u[even] *= np.array([1e-3, 1e-6, 1e-12])[even // 2 % 3, None]
        u[even, (n // 2) * (n * n + n + 1)] = 1.0
    elif kind == "corner":
        u[even] *= 10.0 ** (-6 * ramp)
    elif kind == "tiny":                                         # the largest entry is below 2^-958
        u[even] *= 1e-295
        g *= 1e40                                                # w itself stays a normal number
    elif kind == "flat":                                         # t sides 512 times as long: weak factors
        u[even] *= np.repeat(2.0 ** (-30 * t), n * n)
        g[even] *= np.array([512.0, 512.0, 1.0, 512.0, 1.0, 1.0 / 512.0])[:, None]
    elif kind == "jacobian":
        g[even] *= 2.0 ** (10 * ramp)
    elif kind == "matrix":
        D = np.random.default_rng(n).uniform(-3, 3, (n, n))
        D[:, n // 2] *= 1e-8
    return D, g.reshape(P["gxyz"].shape), u


def boxes(n, few):
    """A few elements (three threads per column), or more than two groups per SM
    (152), no multiple of the group size."""
    if few:
        return (3, 1, 1)
    return (61, 5, 1) if n == 8 or n >= 10 else ((61, 15, 1) if n >= 6 else (199, 3, 17))


@pytest.mark.parametrize("kind", ["spike", "corner", "tiny", "flat", "jacobian", "matrix"])
@pytest.mark.parametrize("few", [False, True])
@pytest.mark.parametrize("n", [2, 5, 8, 10, 16])
def test_operator(nek, oracle, n, few, kind):
    dims = boxes(n, few)
    P = oracle.box_problem(*dims, n, inputs.PERTURB_AMP, inputs.perturbation_coeffs(n))
    D, g, u = graded(kind, P, n)
    want = oracle.ax_e(D, g, u)
    h = nek.nb_setup(dims, n, D, g, stream=torch.cuda.current_stream())
    try:
        w = torch.empty(u.shape, dtype=torch.float64, device="cuda")
        nek.nb_ax(h, torch.from_numpy(u).cuda(), w)
        torch.cuda.current_stream().synchronize()
        got = w.cpu().numpy()
    finally:
        nek.nb_destroy(h)
    limit = BOUND * absolute_operator(D, g, u, kind != "matrix")
    even = slice(None) if kind == "matrix" else slice(0, None, 2)
    assert (np.abs(got - want) <= limit)[even].all()
    err = np.abs(got - want).max(axis=1) / np.abs(want).max(axis=1)
    assert err[1::2].max() <= (1e-12 if kind == "matrix" else 2e-14)


@pytest.mark.parametrize("n,few", [(4, False), (8, True), (10, False)])
def test_operator_beside_itself(nek, oracle, n, few):
    """nb_ax keeps nothing between its launches: two captured calls of one context,
    replayed on two streams at a time, give the bits they give alone."""
    dims = boxes(n, few)
    P = oracle.box_problem(*dims, n, inputs.PERTURB_AMP, inputs.perturbation_coeffs(n))
    stream = torch.cuda.current_stream()
    h = nek.nb_setup(dims, n, P["D"], P["gxyz"], stream=stream)
    try:
        us = [torch.from_numpy(graded(kind, P, n)[2]).cuda() for kind in ("spike", "corner")]
        alone, outs, graphs = [], [], []
        for u in us:
            w = torch.empty_like(u)
            nek.nb_ax(h, u, w)
            stream.synchronize()
            alone.append(w.clone())
            outs.append(w)
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=stream, capture_error_mode="thread_local"):
                nek.nb_ax(h, u, w)
            graphs.append(g)
        sides = [torch.cuda.Stream(), torch.cuda.Stream()]
        for w in outs:
            w.fill_(7.0)
        torch.cuda.synchronize()
        for _ in range(20):
            for g, side in zip(graphs, sides):
                with torch.cuda.stream(side):
                    g.replay()
        torch.cuda.synchronize()
        for w, want in zip(outs, alone):
            assert torch.equal(w.view(torch.int64), want.view(torch.int64))
    finally:
        nek.nb_destroy(h)


@pytest.mark.parametrize("jacobi", [False, True])
@pytest.mark.parametrize("n,dims", [(8, (13, 7, 5)), (13, (11, 7, 5))])
def test_cg_heads(nek, oracle, n, dims, jacobi):
    """Two CG iterations from a right-hand side that falls by 1e-9 and more within an
    element, point by point: x = a0 p0 + a1 (r1 + b1 p0) with r1 = f - a0 A p0."""
    P = oracle.box_problem(*dims, n, inputs.PERTURB_AMP, inputs.perturbation_coeffs(n))
    gid = oracle.gid(*dims, n).reshape(-1)
    shape = tuple(e * (n - 1) + 1 for e in reversed(dims))
    z, y, x = np.meshgrid(*(np.linspace(0, e, s) for e, s in zip(reversed(dims), shape)), indexing="ij")
    fall = np.exp(-7.0 * (np.abs(x - 0.43 * dims[0]) + np.abs(y - 0.4 * dims[1]) + np.abs(z - 0.45 * dims[2])))
    f = (inputs.unique_field(*dims, n, seed=n) * fall.reshape(-1))[gid].reshape(P["E"], -1)
    f = oracle.apply_mask(P["mask"], f)
    minv = oracle.jacobi_inverse(*dims, n, P["D"], P["gxyz"], P["mask"]) if jacobi else np.ones_like(f)
    apply = lambda v: oracle.apply_A(*dims, n, P["D"], P["gxyz"], P["mask"], v)
    dot = lambda a, b: oracle.dot_c(*dims, n, a, b)
    p0 = minv * f
    A0 = apply(p0)
    rho0 = dot(f, p0)
    a0 = rho0 / dot(p0, A0)
    r1 = f - a0 * A0
    z1 = minv * r1
    b1 = dot(r1, z1) / rho0
    p1 = z1 + b1 * p0
    a1 = dot(r1, z1) / dot(p1, apply(p1))
    want = a0 * p0 + a1 * p1
    B = np.bincount(gid, absolute_operator(P["D"], P["gxyz"], p0, True).reshape(-1))[gid].reshape(f.shape)
    # the scalars carry 1e-11 at most (the oracle's own sums, R r and w p at 2^-42)
    limit = 1e-11 * (abs(a0 * p0) + abs(a1) * minv * (abs(f) + abs(a0 * A0)) + abs(a1 * b1 * p0)) + \
        abs(a1) * minv * abs(a0) * BOUND * B
    h = nek.nb_setup(dims, n, P["D"], P["gxyz"], stream=torch.cuda.current_stream())
    try:
        if jacobi:
            nek.nb_set_preconditioner(h, 1)
        xd = torch.zeros(P["E"], n ** 3, dtype=torch.float64, device="cuda")
        nek.nb_cg_solve(h, torch.from_numpy(f).cuda(), xd, tol=0.0, maxit=2)
        torch.cuda.current_stream().synchronize()
        got = xd.cpu().numpy()
    finally:
        nek.nb_destroy(h)
    assert (np.abs(got - want) <= limit + 1e-300).all()
