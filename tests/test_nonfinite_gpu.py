"""A NaN or an Inf in the input or in the operator's data does not disappear in
the fixed-point arithmetic: the results of its element are not finite, those
of the other elements keep their bits, nb_apply carries it to the neighbours'
shared nodes, and a CG solve ends with a breakdown.  On both thread layouts and
both CG heads."""
import numpy as np
import pytest

from paper_2005_13425_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FEW, MANY = (3, 2, 2), (9, 9, 9)


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


def problem(oracle, dims, n, what):
    """D, gxyz, a field and the index of the element that has the bad value."""
    P = oracle.box_problem(*dims, n, inputs.PERTURB_AMP, inputs.perturbation_coeffs(n))
    D, g = P["D"].copy(), P["gxyz"].copy()
    u = inputs.local_field(P["E"], n, seed=n)
    bad = P["E"] // 2
    value = {"nan": np.nan, "inf": np.inf}[what.split("_")[1]]
    point = (n // 2) * (n * n + n + 1)
    if what[0] == "u":
        u[bad, point] = value
    elif what[0] == "g":
        g.reshape(P["E"], 6, -1)[bad, 3, point] = value
    else:
        D[1, 2] = value
    return P, D, g, u, bad


def call(nek, f, dims, n, D, g, u):
    h = nek.nb_setup(dims, n, D, g, stream=torch.cuda.current_stream())
    try:
        w = torch.empty(u.shape, dtype=torch.float64, device="cuda")
        f(h, torch.from_numpy(u).cuda(), w)
        torch.cuda.current_stream().synchronize()
        return w.cpu().numpy()
    finally:
        nek.nb_destroy(h)


@pytest.mark.parametrize("what", ["u_nan", "u_inf", "g_nan", "g_inf", "D_nan", "D_inf"])
@pytest.mark.parametrize("dims", [FEW, MANY])
@pytest.mark.parametrize("n", [4, 8, 13])
def test_operator(nek, oracle, n, dims, what):
    P, D, g, u, bad = problem(oracle, dims, n, what)
    got = call(nek, nek.nb_ax, dims, n, D, g, u)
    if what[0] == "D":
        assert not np.isfinite(got).any()
        return
    assert not np.isfinite(got[bad]).any()
    clean = call(nek, nek.nb_ax, dims, n, P["D"], P["gxyz"], inputs.local_field(P["E"], n, seed=n))
    others = np.arange(P["E"]) != bad
    assert np.array_equal(got[others].view(np.int64), clean[others].view(np.int64))


@pytest.mark.parametrize("what", ["u_nan", "g_inf"])
def test_apply_reaches_the_neighbours(nek, oracle, what):
    dims, n = (3, 3, 3), 8
    P, D, g, u, bad = problem(oracle, dims, n, what)          # the middle element
    got = call(nek, nek.nb_apply, dims, n, D, g, u).reshape(P["E"], n, n, n)
    assert not np.isfinite(got[bad]).any()
    assert not np.isfinite(got[bad + 1][:, :, 0]).any() and np.isfinite(got[bad + 1][:, :, 1:]).all()
    assert (got[0][0] == 0.0).all()                           # box faces


@pytest.mark.parametrize("what", ["u_nan", "g_nan", "g_inf"])
@pytest.mark.parametrize("jacobi", [False, True])
@pytest.mark.parametrize("dims", [FEW, MANY])
def test_cg_breaks_down(nek, oracle, dims, jacobi, what):
    n = 8
    P, D, g, u, bad = problem(oracle, dims, n, what)
    f = oracle.apply_mask(P["mask"], oracle.scatter_unique(*dims, n, inputs.unique_field(*dims, n, seed=n)))
    if what[0] == "u":
        f[bad, (n // 2) * (n * n + n + 1)] = np.nan
    h = nek.nb_setup(dims, n, D, g, stream=torch.cuda.current_stream())
    try:
        if jacobi:
            nek.nb_set_preconditioner(h, 1)
        x = torch.zeros(P["E"], n ** 3, dtype=torch.float64, device="cuda")
        with pytest.raises(nek.NekgbError) as err:
            nek.nb_cg_solve(h, torch.from_numpy(f).cuda(), x, tol=0.0, maxit=10)
        assert err.value.status == nek.NB_ERR_BREAKDOWN
        assert "range" not in str(err.value)
    finally:
        nek.nb_destroy(h)
