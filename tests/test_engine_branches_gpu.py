"""A step whose groups run as graph branches, one of them big enough to share
the in-turn branch: every request's solution has the bits it has alone (no
tolerance: a request's arithmetic does not depend on the batch)."""
import pytest

from paper_2005_13425_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def solve(nek, reqs, stream):
    need = sum(nek.nb_engine_footprint(d, n, prec) for d, n, prec in reqs)
    eng = nek.nb_engine_create(int(need * 1.1) + (64 << 20), stream)
    try:
        ids = []
        for k, (d, n, prec) in enumerate(reqs):
            fu = torch.from_numpy(inputs.unique_field(*d, n, seed=d[0] + n)).cuda()
            _, rid = nek.nb_engine_submit_unique(eng, d, n, inputs.PERTURB_AMP, (0.3, -0.5, 0.7), 0.0, 16, fu,
                                                 prec=prec)
            ids.append(rid)
        for _ in range(4):
            nek.nb_engine_step(eng, 8)
        out = []
        for (d, n, _), rid in zip(reqs, ids):
            x = torch.empty(d[0] * d[1] * d[2], n ** 3, dtype=torch.float64, device="cuda")
            nek.nb_engine_retire(eng, rid, x)
            out.append(x)
        stream.synchronize()
        return out
    finally:
        nek.nb_engine_destroy(eng)


@pytest.mark.parametrize("big", ((28, 28, 28), (4, 4, 3)))
def test_branches_keep_the_bits(big, monkeypatch, tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_13425_gb300 import build as b
    b.build()
    from paper_2005_13425_gb300 import nekgb as nek
    nek.load()
    monkeypatch.setenv("NEKGB_TUNE_CACHE", str(tmp_path / "tune.txt"))
    stream = torch.cuda.Stream()
    torch.cuda.set_stream(stream)
    reqs = [(big, 3, nek.NB_FP64), ((3, 2, 2), 4, nek.NB_FP64), ((2, 2, 3), 4, nek.NB_MIXED),
            ((4, 3, 2), 6, nek.NB_FP64)]
    together = solve(nek, reqs, stream)
    for q, x in zip(reqs, together):
        alone, = solve(nek, [q], stream)
        assert torch.equal(alone.view(torch.int64), x.view(torch.int64)), q
