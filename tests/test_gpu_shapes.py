"""Grids far from a cube -- long lines, few planes, single planes -- and vectors of
several right-hand sides on them: values bit for bit those of the stored-matrix or
the single-vector kernels, and times near those of a compact grid of about the
same number of points (each ratio stood at 1.6 or more where a rule looked at the
number of points alone, or a kernel was slow on such a grid)."""

import pytest

torch = pytest.importorskip("torch")

import paper_2507_11512_gb300 as hpg  # noqa: E402
from paper_2507_11512_gb300 import batch  # noqa: E402

pytestmark = pytest.mark.gpu

DEV = "cuda"
STORED = 3   # HPG_OPT_GS_PIPELINE: every sweep on the stored matrix
DTYPE = {"fp32": torch.float32, "fp64": torch.float64}


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available()


def vec(p, dtype, seed):
    g = torch.Generator(device="cpu").manual_seed(seed)
    nat = torch.randn(p.info[0]["n"], generator=g, dtype=torch.float64).to(DEV)
    return p.to_storage(nat, dtype=dtype)


def graph_us(call):
    """Device time of a call: 32 of them in a CUDA graph, the fastest of eleven replays."""
    call()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        for _ in range(32):
            call()
    best = float("inf")
    for _ in range(11):
        e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        e0.record()
        g.replay()
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1) * 1e3 / 32)
    return best


def case_us(op, prec, dims):
    with hpg.Problem(*dims, beta=0.4, levels=1 if op == "smooth" else 4) as p:
        r = vec(p, DTYPE[prec], 1)
        z = torch.zeros_like(r)
        if op == "spmv":
            return graph_us(lambda: hpg.spmv(p.h, 0, r, z))
        if op == "smooth":
            return graph_us(lambda: hpg.mg_smooth(p.h, 0, r, z, 1, False))
        return graph_us(lambda: hpg.mg_vcycle(p.h, 0, r, z))


# (what, precision, grid, compact grid, bound on the ratio of their times)
TIMES = [
    # lines that no plane takes: colour phases whose addresses are formed before the wait
    # (47 us; 25 now) against 26 us by planes
    ("smooth", "fp32", (2000, 4, 4), (1000, 8, 8), 1.4),
    # few planes, in FP64 few busy SMs: colours instead (136, 92 and 47 us; 43, 19 and 32
    # now, against 42, 26 and 15 by planes)
    ("smooth", "fp64", (128, 128, 8), (64, 64, 32), 1.6),
    ("smooth", "fp64", (200, 200, 1), (40, 40, 40), 1.6),
    ("smooth", "fp32", (300, 300, 4), (72, 72, 72), 2.6),
    # lines of one point (82 us; 29 now, against 28)
    ("smooth", "fp32", (1, 1000, 1000), (104, 104, 104), 1.6),
    # few planes are few CTAs of the small levels' cluster (120 and 34 us; 65 and 12 now,
    # against 66 and 13)
    ("vcycle", "fp32", (90, 88, 4), (32, 32, 32), 1.4),
    ("smooth", "fp32", (64, 64, 4), (32, 32, 32), 1.6),
    # a small product's launch and latency (4.1 us; 2.8 now, against 15.6)
    ("spmv", "fp64", (16, 16, 16), (64, 64, 64), 0.245),
]


@pytest.mark.parametrize("op,prec,dims,compact,bound", TIMES)
def test_time_against_a_compact_grid(op, prec, dims, compact, bound):
    t, ref = case_us(op, prec, dims), case_us(op, prec, compact)
    assert t <= bound * ref, (t, ref)


# lines that no plane takes; grids on both sides of the choice between planes and colours
@pytest.mark.parametrize("dims", [(2000, 4, 4), (3100, 3, 2), (1700, 5, 7),
                                  (200, 200, 1), (128, 128, 8), (150, 150, 2), (1, 300, 300),
                                  (2, 300, 300), (72, 71, 72), (64, 64, 64), (16, 2000, 4)])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("theta", [False, True])
def test_sweeps_equal_stored_matrix(dims, prec, theta):
    n = dims[0] * dims[1] * dims[2]
    g = torch.Generator(device="cpu").manual_seed(3)
    th = (0.9 + 0.2 * torch.rand(n, generator=g, dtype=torch.float64)).numpy() if theta else None
    with hpg.Problem(*dims, beta=-0.4, levels=1, theta=th) as p:
        r, z0 = vec(p, DTYPE[prec], 1), vec(p, DTYPE[prec], 2)
        out = []
        for pipe in (1, STORED):
            hpg.set_option(p.h, hpg.HPG_OPT_GS_PIPELINE, pipe)
            for zero in (True, False):
                z = z0.clone()
                hpg.mg_smooth(p.h, 0, r, z, 1, zero)
                out.append(z)
        assert torch.equal(out[0], out[2]) and torch.equal(out[1], out[3])


# lines longer than a plane's CTA takes, even and odd edges
@pytest.mark.parametrize("dims", [(1600, 3, 4), (801, 5, 3)])
@pytest.mark.parametrize("R", [2, 4, 8])
@pytest.mark.parametrize("theta", [False, True])
def test_rvector_colour_phases_equal_single_vector(dims, R, theta):
    n = dims[0] * dims[1] * dims[2]
    g = torch.Generator(device="cpu").manual_seed(3)
    th = (0.9 + 0.2 * torch.rand(n, generator=g, dtype=torch.float64)).numpy() if theta else None
    with hpg.Problem(*dims, beta=0.5, levels=1, theta=th) as p:
        X = torch.stack([vec(p, torch.float32, 20 + q) for q in range(R)], dim=1).contiguous()
        Y = torch.empty_like(X)
        batch.vcycle_batch(p.h, 0, X, Y)
        for q in range(R):
            assert torch.equal(Y[:, q], p.vcycle(X[:, q].contiguous())), q


@pytest.mark.parametrize("dims", [(128, 128, 128), (160, 128, 104), (96, 96, 96)])
def test_default_sweeps_read_no_stored_matrix(dims):
    """By the profile's byte model: vectors alone, at every size (the pipelined sweep on
    the stored matrix, 15/8 x 27 x 12 bytes a point, was the default in a band of sizes)."""
    with hpg.Problem(*dims, beta=0.4, levels=1) as p:
        r, z = vec(p, torch.float64, 1), vec(p, torch.float64, 2)
        hpg.set_profiling(p.h, True)
        hpg.mg_smooth(p.h, 0, r, z, 1, False)
        torch.cuda.synchronize()
        total = sum(k["bytes"] for k in hpg.profile_report(p.h))
    assert 0 < total < 100.0 * p.info[0]["n"]


# V-cycles that leave the small levels' cluster: planes and colours with a diagonal per
# cell, two and four elements a thread (600,000 elements), odd edges
@pytest.mark.parametrize("dims", [(45, 37, 41), (64, 64, 8), (64, 64, 2), (46, 44, 40),
                                  (45, 44, 40), (56, 56, 52), (57, 56, 50)])
@pytest.mark.parametrize("R", [2, 4, 8])
def test_rvector_vcycle_with_cell_diagonals_equals_single_vector(dims, R):
    n = dims[0] * dims[1] * dims[2]
    g = torch.Generator(device="cpu").manual_seed(3)
    th = (0.9 + 0.2 * torch.rand(n, generator=g, dtype=torch.float64)).numpy()
    with hpg.Problem(*dims, beta=0.5, theta=th) as p:
        X = torch.stack([vec(p, torch.float32, 20 + q) for q in range(R)], dim=1).contiguous()
        Y = torch.empty_like(X)
        batch.vcycle_batch(p.h, 0, X, Y)
        for q in range(R):
            assert torch.equal(Y[:, q], p.vcycle(X[:, q].contiguous())), q
        batch.spmv_batch(p.h, 0, X, Y)
        for q in range(R):
            assert torch.equal(Y[:, q], p.spmv(X[:, q].contiguous())), q


# R-vectors anywhere on a 4-byte boundary: the product and the V-cycle (small levels'
# cluster, planes, colours) give what aligned vectors give and write nothing beside them
@pytest.mark.parametrize("dims", [(24, 20, 28), (64, 48, 40), (45, 37, 41), (64, 64, 8)])
@pytest.mark.parametrize("R", [2, 4, 8])
@pytest.mark.parametrize("off", [1, 2, 3])
def test_rvectors_off_a_vector_boundary(dims, R, off):
    with hpg.Problem(*dims, beta=0.5) as p:
        X = torch.stack([vec(p, torch.float32, 20 + q) for q in range(R)], dim=1).contiguous()
        n = X.numel()
        for f in (batch.spmv_batch, batch.vcycle_batch):
            ref = torch.empty_like(X)
            f(p.h, 0, X, ref)
            xb, yb = (torch.zeros(n + 4, dtype=torch.float32, device=DEV) for _ in range(2))
            xb[off:off + n] = X.reshape(-1)
            f(p.h, 0, xb[off:off + n].view(-1, R), yb[off:off + n].view(-1, R))
            assert torch.equal(yb[off:off + n].view(-1, R), ref)
            assert not yb[:off].any() and not yb[off + n:].any()


# FP64 products by single points, by rows and by lines, with a diagonal per cell
@pytest.mark.parametrize("dims", [(16, 16, 16), (33, 17, 24), (5, 1, 3), (1, 1, 40), (45, 37, 41),
                                  (64, 63, 30), (130, 128, 100)])
@pytest.mark.parametrize("theta", [False, True])
def test_fp64_product_against_plain_torch(dims, theta):
    nx, ny, nz = dims
    n, beta = nx * ny * nz, -0.4
    g = torch.Generator(device="cpu").manual_seed(3)
    th = 0.9 + 0.2 * torch.rand(n, generator=g, dtype=torch.float64)
    x = torch.randn(n, generator=g, dtype=torch.float64).to(DEV)

    def product(v, b, diag):
        vp = torch.nn.functional.pad(v.view(nz, ny, nx), (1, 1, 1, 1, 1, 1))
        y = (diag * v).view(nz, ny, nx).clone()
        for q in range(27):
            dx, dy, dz = q % 3, q // 3 % 3, q // 9
            if q != 13:
                y += (-1.0 + b * (dx + dy + dz - 3) / 3.0) * vp[dz:dz + nz, dy:dy + ny, dx:dx + nx]
        return y.reshape(-1)

    diag = 26.0 * th.to(DEV) if theta else torch.full_like(x, 26.0)
    with hpg.Problem(*dims, beta=beta, levels=1, theta=th.numpy() if theta else None) as p:
        y = p.to_natural(p.spmv(p.to_storage(x)))
        # padding rows are identity rows
        pad = torch.ones(p.n_store(0), dtype=torch.float64, device=DEV)
        pad[p.to_storage(torch.ones_like(x)) != 0] = 0
        assert torch.equal(p.spmv(pad), pad)
    # |A||x|: 26 theta and at most 1.4 a neighbour; 27 FMAs and the rounding of a
    # coefficient make 28 u of it, twice that with the reference's own
    scale = diag * x.abs() - 1.4 * product(x.abs(), 0.0, torch.zeros_like(x))
    assert ((y - product(x, beta, diag)).abs() <= 2 * 28 * 2.0 ** -53 * scale).all()
