"""Launches of a batch: the shapes that hpg_batch_tune or a caller chose survive
hpg_batch_tune_solve, which solves from zero and reports a time; programmatic
launches (HPG_OPT_PDL) change no value, on levels that start the next kernel early
and on those that do not."""

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


@pytest.mark.parametrize("dims", [(16, 16, 16), (40, 40, 8), (64, 64, 8), (64, 48, 40),
                                  (96, 96, 96)])
def test_programmatic_launches_change_nothing(dims):
    n = dims[0] * dims[1] * dims[2]
    g = torch.Generator(device="cuda").manual_seed(2)
    B = torch.randn(8, n, dtype=torch.float64, device="cuda", generator=g)
    with hpg.Problem(*dims, beta=0.6) as p:
        X = {R: torch.stack([p.to_storage(B[q], dtype=torch.float32) for q in range(R)],
                            dim=1).contiguous() for R in (2, 8)}
        out = []
        for on in (1, 0):
            hpg.set_option(p.h, hpg.HPG_OPT_PDL, on)
            got = [p.vcycle(p.to_storage(B[0])), p.vcycle(p.to_storage(B[0], dtype=torch.float32))]
            for R in (2, 8):
                for _ in range(2):
                    Y = torch.empty_like(X[R])
                    batch.vcycle_batch(p.h, 0, X[R], Y)
                    got.append(Y)
            S = torch.zeros_like(B[:2])
            infos = batch.solve_batch(p.h, B[:2].contiguous(), S, tol=1e-8)
            got += [S, torch.tensor([i["iterations"] for i in infos])]
            x, info = p.solve(B[0].contiguous(), tol=1e-8)
            got += [x, torch.tensor(info["iterations"])]
            out.append(got)
        for a, b in zip(*out):
            assert torch.equal(a, b)
