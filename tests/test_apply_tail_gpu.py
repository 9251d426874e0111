"""nb_apply's tail (dssum and box mask in one launch) against the separate
operator, dssum and mask calls, bit for bit: boxes with one element in some or
all directions (no shared nodes there), n = 2 (every point on an element face)
and boxes whose every shared node lies on a box face or none does.  No
tolerance: each point is the same sum or the same +0.0 either way."""
import numpy as np
import pytest

from paper_2005_13425_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", (2, 3, 8, 9, 16))
@pytest.mark.parametrize("dims", ((1, 1, 1), (2, 1, 1), (1, 3, 2), (2, 2, 2), (5, 3, 4)))
@pytest.mark.parametrize("kind", ("random", "nan"))
def test_apply_is_ax_dssum_mask(dims, n, kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_13425_gb300 import build as b
    b.build()
    from paper_2005_13425_gb300 import nekgb
    nekgb.load()
    stream = torch.cuda.Stream()
    torch.cuda.set_stream(stream)
    h = nekgb.nb_setup_box(dims, n, inputs.PERTURB_AMP, (0.3, -0.5, 0.7), nekgb.NB_FP64, stream)
    try:
        E = dims[0] * dims[1] * dims[2]
        u = np.random.default_rng(7).uniform(-1.0, 1.0, (E, n ** 3))
        if kind == "nan":   # an element that is not finite reaches its neighbours, never the faces
            u[E // 2, n ** 3 // 2] = np.nan
        u = torch.from_numpy(u).cuda()
        w = torch.full_like(u, 7.0)
        v = torch.full_like(u, 7.0)
        nekgb.nb_apply(h, u, w)
        nekgb.nb_ax(h, u, v)
        nekgb.nb_dssum(h, v)
        nekgb.nb_mask(h, v)
        stream.synchronize()
        assert torch.equal(w.view(torch.int64), v.view(torch.int64))
    finally:
        nekgb.nb_destroy(h)
