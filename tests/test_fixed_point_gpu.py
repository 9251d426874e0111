"""The fixed-point-pair operator where its layouts change: one column per
thread (more elements than two per SM) with ragged groups of elements, three
threads per column (fewer), plain line products, and scales outside the range
of one power of two.

Tolerance: the pairs carry 30 + 24 bits, their small sums round at 2^-25 of a
unit; a bit-level emulation of the kernel gives 1e-15 to 2.5e-15 of max|w| on
random data for n = 2..16.  2e-14 is ten times that, and a twentieth of what a
lost term of the small sums would cost (2^-31 of the terms, which are 30-60
times the result).
"""
import numpy as np
import pytest

from paper_2005_13425_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 2e-14


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


def run_ax(nek, dims, n, D, g, u):
    h = nek.nb_setup(dims, n, D, g, stream=torch.cuda.current_stream())
    try:
        w = torch.empty(u.shape, dtype=torch.float64, device="cuda")
        nek.nb_ax(h, torch.from_numpy(u).cuda(), w)
        torch.cuda.current_stream().synchronize()
        return w.cpu().numpy()
    finally:
        nek.nb_destroy(h)


def rel(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


def many(n):
    """A box with more than two groups of elements per SM (152), no multiple of
    the group size."""
    return (61, 5, 1) if n == 8 or n >= 10 else ((61, 15, 1) if n >= 6 else (199, 3, 17))


@pytest.mark.parametrize("n", range(2, 17))
@pytest.mark.parametrize("few", [False, True])
def test_operator_layouts(nek, oracle, few, n):
    dims = (3, 1, 1) if few else many(n)
    P = oracle.box_problem(*dims, n, inputs.PERTURB_AMP, inputs.perturbation_coeffs(n))
    u = inputs.local_field(P["E"], n, seed=n + 50)
    u[1] *= 1e-9                              # the scale is an element's own
    want = oracle.ax_e(P["D"], P["gxyz"], u)
    got = run_ax(nek, dims, n, P["D"], P["gxyz"], u)
    assert rel(got, want) <= TOL
    assert rel(got[1], want[1]) <= TOL


@pytest.mark.parametrize("n", [4, 7, 13])
def test_plain_lines_many_elements(nek, oracle, n):
    dims = many(n)
    P = oracle.box_problem(*dims, n, inputs.PERTURB_AMP, inputs.perturbation_coeffs(n))
    D = np.random.default_rng(n).uniform(-3, 3, (n, n))
    u = inputs.local_field(P["E"], n, seed=n + 60)
    want = oracle.ax_e(D, P["gxyz"], u)
    assert rel(run_ax(nek, dims, n, D, P["gxyz"], u), want) <= TOL


@pytest.mark.parametrize("su,sg", [(1e-200, 1e-90), (1e200, 1e95), (1e-150, 1e150)])
def test_scales_beyond_one_factor(nek, oracle, su, sg):
    dims, n = (3, 2, 1), 6
    P = oracle.box_problem(*dims, n, inputs.PERTURB_AMP, inputs.perturbation_coeffs(2))
    u = inputs.local_field(P["E"], n, seed=70)
    want = oracle.ax_e(P["D"], P["gxyz"], u)          # w is linear in u and gxyz
    got = run_ax(nek, dims, n, P["D"], P["gxyz"] * sg, u * su)
    assert np.all(np.isfinite(got))
    assert rel(got / su / sg, want) <= TOL


@pytest.mark.parametrize("n", [3, 6, 9, 13, 16])
def test_cg_head_many_elements(nek, oracle, n):
    """Ten iterations of the two-kernel CG in the throughput layout (with and
    without the kept input) against the oracle's."""
    dims = many(n)
    P = oracle.box_problem(*dims, n, inputs.PERTURB_AMP, inputs.perturbation_coeffs(n))
    f = oracle.apply_mask(P["mask"], oracle.scatter_unique(*dims, n, inputs.unique_field(*dims, n, seed=n)))
    x_ref, it_ref, _, hist_ref, _ = oracle.cg(*dims, n, P["D"], P["gxyz"], P["mask"], f, tol=0.0, maxit=10)
    h = nek.nb_setup(dims, n, P["D"], P["gxyz"], stream=torch.cuda.current_stream())
    try:
        x = torch.zeros(P["E"], n ** 3, dtype=torch.float64, device="cuda")
        _, it, _ = nek.nb_cg_solve(h, torch.from_numpy(f).cuda(), x, tol=0.0, maxit=10)
        hist = nek.nb_cg_history(h)
        torch.cuda.current_stream().synchronize()
        xg = x.cpu().numpy()
    finally:
        nek.nb_destroy(h)
    assert it == it_ref == 10
    assert np.abs(hist - hist_ref).max() <= 1e-10 * hist_ref.max()
    assert rel(xg, x_ref) <= 1e-10
