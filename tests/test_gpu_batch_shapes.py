"""Launch shapes of a batch: what hpg_batch_tune or a caller chose survives
hpg_batch_tune_solve, which solves from zero and reports a time."""

import pytest

torch = pytest.importorskip("torch")

import paper_2507_11512_gb300 as hpg  # noqa: E402
from paper_2507_11512_gb300 import batch  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available()


@pytest.mark.parametrize("nrhs", [1, 2, 4, 8])
def test_tune_solve_keeps_the_spmv_block(nrhs):
    edges = (16, 24)
    probs = [hpg.Problem(e, e, e, beta=0.5) for e in edges]
    g = torch.Generator(device="cuda").manual_seed(2)
    Bs = [torch.randn(nrhs, e ** 3, dtype=torch.float64, device="cuda", generator=g) for e in edges]
    try:
        for p in probs:
            batch.set_shape(p.h, 0, batch.KIND_SPMV, nrhs, 0, 128)
        with batch.BatchSolver(probs, nrhs) as solver:
            ref = [torch.zeros_like(b) for b in Bs]
            solver.solve(Bs, ref, tol=1e-9)
            Xs = [torch.ones_like(b) for b in Bs]
            times = solver.tune(Bs, Xs, tol=1e-9)
            assert sorted(times) == sorted({1, min(2, nrhs), nrhs})
            assert all(t > 0.0 for t in times.values())
            assert all(torch.equal(a, b) for a, b in zip(Xs, ref))
            Xs = [torch.zeros_like(b) for b in Bs]
            solver.solve(Bs, Xs, tol=1e-9)
            assert all(torch.equal(a, b) for a, b in zip(Xs, ref))
        for p in probs:
            assert batch.get_shape(p.h, 0, batch.KIND_SPMV, nrhs) == (1, 128)
    finally:
        for p in probs:
            p.close()
