"""The CG heads of large boxes (fixed-point pairs, one column per thread): every CTA
takes three groups of elements or more, the last group ragged, so that the loop
over the groups, the dynamic schedule and the reuse of the shared arrays run;
and the properties that the solves promise, bit for bit, on boxes beyond those
of the head for few elements.

E is above three times the groups that 152 SMs can hold (2048 threads or 64
registers a thread bound them) times the elements of a group.  The tolerance is
the one of the CG parity tests at few iterations: 1e-10 of the largest value.
"""
import numpy as np
import pytest

from paper_2005_13425_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LOOPS = {3: (61, 29, 29), 4: (61, 31, 16), 6: (37, 17, 18), 7: (41, 19, 11), 10: (31, 13, 7), 13: (29, 11, 7)}
LARGE = (13, 7, 5)      # 455 elements: more than two per SM


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


def problem(oracle, dims, n):
    P = oracle.box_problem(*dims, n, inputs.PERTURB_AMP, inputs.perturbation_coeffs(n))
    f = oracle.apply_mask(P["mask"], oracle.scatter_unique(*dims, n, inputs.unique_field(*dims, n, seed=n)))
    return P, f


def solve(nek, h, f, maxit, stream, **kw):
    """x, history and status of a solve from zero."""
    with torch.cuda.stream(stream):
        x = torch.zeros(f.shape, dtype=torch.float64, device="cuda")
        st, it, _ = nek.nb_cg_solve(h, torch.from_numpy(f).cuda(), x, tol=0.0, maxit=maxit, **kw)
        hist = nek.nb_cg_history(h)
        stream.synchronize()
        return x.cpu().numpy(), hist, st, it


def rel(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


@pytest.mark.parametrize("n", sorted(LOOPS))
def test_two_kernel_head_over_many_groups(nek, oracle, n):
    dims = LOOPS[n]
    P, f = problem(oracle, dims, n)
    x_ref, _, _, hist_ref, _ = oracle.cg(*dims, n, P["D"], P["gxyz"], P["mask"], f, tol=0.0, maxit=4)
    stream = torch.cuda.current_stream()
    h = nek.nb_setup(dims, n, P["D"], P["gxyz"], stream=stream)
    try:
        x, hist, st, it = solve(nek, h, f, 4, stream)
        again = solve(nek, h, f, 4, stream)
    finally:
        nek.nb_destroy(h)
    assert it == 4 and rel(x, x_ref) <= 1e-10 and np.abs(hist - hist_ref).max() <= 1e-10 * hist_ref.max()
    assert np.array_equal(x, again[0]) and np.array_equal(hist, again[1])     # whatever the schedule


@pytest.mark.parametrize("form", ["jacobi", "mask"])
@pytest.mark.parametrize("n", [4, 7, 10, 13])
def test_other_heads_over_many_groups(nek, oracle, n, form):
    """Jacobi, and a mask of the caller's."""
    dims = LOOPS[n]
    P, f = problem(oracle, dims, n)
    stream = torch.cuda.current_stream()
    mask = None
    if form == "mask":
        # one interior node per element more, at the element's centre
        mask = P["mask"].copy().reshape(P["E"], n, n, n)
        mask[:, n // 2, n // 2, n // 2] = 0
        mask = mask.reshape(P["mask"].shape)
        f = oracle.apply_mask(mask, f)
        ref = oracle.cg(*dims, n, P["D"], P["gxyz"], mask, f, tol=0.0, maxit=4)
    else:
        minv = oracle.jacobi_inverse(*dims, n, P["D"], P["gxyz"], P["mask"])
        ref = oracle.pcg(*dims, n, P["D"], P["gxyz"], P["mask"], minv, f, tol=0.0, maxit=4)
    h = nek.nb_setup(dims, n, P["D"], P["gxyz"], mask=mask, stream=stream)
    try:
        if form == "jacobi":
            nek.nb_set_preconditioner(h, 1)
        x, _, _, it = solve(nek, h, f, 4, stream)
        again = solve(nek, h, f, 4, stream)
    finally:
        nek.nb_destroy(h)
    assert it == 4 and rel(x, ref[0]) <= 1e-10
    assert np.array_equal(x, again[0])


def test_range_check_stops_the_solve(nek, oracle, monkeypatch):
    """Shares beyond the exact sum's range (the scale shifted at set-up)."""
    n = 8
    P, f = problem(oracle, LARGE, n)
    stream = torch.cuda.current_stream()
    monkeypatch.setenv("NEKGB_TEST_DOT_SHIFT", "60")
    h = nek.nb_setup(LARGE, n, P["D"], P["gxyz"], stream=stream)
    monkeypatch.delenv("NEKGB_TEST_DOT_SHIFT")
    try:
        *_, st, _ = solve(nek, h, f, 20, stream, allow=(nek.NB_ERR_BREAKDOWN,))
        assert st == nek.NB_ERR_BREAKDOWN and "range" in nek.nb_last_error()
    finally:
        nek.nb_destroy(h)


@pytest.mark.parametrize("n,k", [(8, 200), (10, -180), (13, 37)])
def test_powers_of_two_keep_the_bits(nek, oracle, n, k):
    P, f = problem(oracle, LARGE, n)
    stream = torch.cuda.current_stream()
    h = nek.nb_setup(LARGE, n, P["D"], P["gxyz"], stream=stream)
    try:
        x0, h0, *_ = solve(nek, h, f, 20, stream)
        x1, h1, *_ = solve(nek, h, f * 2.0 ** k, 20, stream)
    finally:
        nek.nb_destroy(h)
    assert np.array_equal(x1, x0 * 2.0 ** k) and np.array_equal(h1, h0 * 2.0 ** (2 * k))


def test_launch_forms_keep_the_bits(nek, oracle):
    """Graphs, plain launches (the default stream) and sampled timing."""
    n = 9
    dims = (13, 11, 7)
    P, f = problem(oracle, dims, n)
    out = []
    for stream, timing in ((torch.cuda.current_stream(), 0), (torch.cuda.default_stream(), 0),
                           (torch.cuda.current_stream(), 2)):
        with torch.cuda.stream(stream):
            h = nek.nb_setup(dims, n, P["D"], P["gxyz"], stream=stream)
            try:
                if timing:
                    nek.nb_timing_enable(h, timing)
                out.append(solve(nek, h, f, 37, stream))
            finally:
                nek.nb_destroy(h)
    for x, hist, *_ in out[1:]:
        assert np.array_equal(x, out[0][0]) and np.array_equal(hist, out[0][1])
