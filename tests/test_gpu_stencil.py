"""Kernels that evaluate the operator straight from the grid against the
stored-matrix ones, bit for bit: sweeps by planes and by colours against the
pipelined sweep (HPG_OPT_GS_PIPELINE 3), the small levels' one-cluster V-cycle
against it too, on odd, aligned, misaligned, long and degenerate grids, with
per-cell diagonals and with infinities; the product against plain torch."""

import pytest

torch = pytest.importorskip("torch")

import paper_2507_11512_gb300 as hpg  # noqa: E402
from paper_2507_11512_gb300 import batch  # noqa: E402

pytestmark = pytest.mark.gpu

DEV = "cuda"
STORED = 3   # HPG_OPT_GS_PIPELINE: every sweep on the stored matrix


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available()


def vec(p, dtype, seed, level=0):
    g = torch.Generator(device="cpu").manual_seed(seed)
    nat = torch.randn(p.info[level]["n"], generator=g, dtype=torch.float64).to(DEV)
    return p.to_storage(nat, level=level, dtype=dtype)


def theta_of(dims, seed):
    g = torch.Generator(device="cpu").manual_seed(seed)
    n = dims[0] * dims[1] * dims[2]
    return (0.9 + 0.2 * torch.rand(n, generator=g, dtype=torch.float64)).numpy()


# whole groups of 4, of 2 and ragged parts, small and large (four elements a thread from
# 600,000 points), one and several CTAs per plane, lines longer than a CTA takes (1538 FP32),
# single planes, lines and columns
GRIDS = [(128, 96, 72), (130, 100, 80), (100, 92, 80), (130, 82, 78), (34, 18, 10), (40, 37, 3), (5, 3, 7),
         (1538, 3, 2), (3100, 2, 3), (1, 9, 4), (6, 1, 5), (7, 6, 1), (2, 2, 2)]


@pytest.mark.parametrize("dims", GRIDS)
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("theta", [False, True])
def test_sweeps_equal_stored_matrix(dims, dtype, theta):
    th = theta_of(dims, 3) if theta else None
    with hpg.Problem(*dims, beta=-0.4, levels=1, theta=th) as p:
        r, z0 = vec(p, dtype, 1), vec(p, dtype, 2)
        out = {}
        for pipe in (1, STORED):
            hpg.set_option(p.h, hpg.HPG_OPT_GS_PIPELINE, pipe)
            for sweeps, zero in [(1, True), (2, True), (1, False), (3, False)]:
                z = z0.clone()
                hpg.mg_smooth(p.h, 0, r, z, sweeps, zero)
                out[pipe, sweeps, zero] = z
        for key in [(1, True), (2, True), (1, False), (3, False)]:
            assert torch.equal(out[(1,) + key], out[(STORED,) + key]), key


@pytest.mark.parametrize("dims", [(128, 96, 72), (32, 16, 12)])
def test_sweeps_on_vectors_off_a_vector_boundary(dims):
    with hpg.Problem(*dims, beta=0.3, levels=1) as p:
        n = p.n_store(0)
        r, z0 = vec(p, torch.float32, 1), vec(p, torch.float32, 2)
        ref = z0.clone()
        hpg.mg_smooth(p.h, 0, r, ref, 1, False)
        y = p.spmv(r)
        for off in (1, 2):
            rb, zb, yb = (torch.zeros(n + 4, dtype=torch.float32, device=DEV) for _ in range(3))
            rb[off:off + n], zb[off:off + n] = r, z0
            hpg.mg_smooth(p.h, 0, rb[off:off + n], zb[off:off + n], 1, False)
            assert torch.equal(zb[off:off + n], ref)
            hpg.spmv(p.h, 0, rb[off:off + n], yb[off:off + n])
            assert torch.equal(yb[off:off + n], y)
            assert not zb[:off].any() and not zb[off + n:].any()


@pytest.mark.parametrize("dims", [(16, 16, 16), (24, 20, 28), (32, 32, 32), (2, 4, 8), (40, 8, 48)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("theta", [False, True])
@pytest.mark.parametrize("pre,post", [(1, 1), (0, 2), (2, 0)])
def test_small_level_vcycle_equals_stored_matrix(dims, dtype, theta, pre, post):
    th = theta_of(dims, 5) if theta else None
    with hpg.Problem(*dims, beta=0.5, theta=th, pre_sweeps=pre, post_sweeps=post) as p:
        for level in range(p.levels):
            r = vec(p, dtype, 7 + level, level)
            zs = []
            for pipe in (1, STORED):
                hpg.set_option(p.h, hpg.HPG_OPT_GS_PIPELINE, pipe)
                zs.append(p.vcycle(r, level=level))
            assert torch.equal(zs[0], zs[1]), level


@pytest.mark.parametrize("dims", [(20, 12, 10), (16, 16, 16)])
@pytest.mark.parametrize("R", [2, 4, 8])
def test_rvector_vcycle_columns_with_cell_diagonals(dims, R):
    with hpg.Problem(*dims, beta=0.5, theta=theta_of(dims, 9)) as p:
        X = torch.stack([vec(p, torch.float32, 20 + r) for r in range(R)], dim=1).contiguous()
        Y = torch.empty_like(X)
        batch.vcycle_batch(p.h, 0, X, Y)
        for r in range(R):
            assert torch.equal(Y[:, r], p.vcycle(X[:, r].contiguous())), r


@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan"), 3.4e38, 1e-38, 0.0])
@pytest.mark.parametrize("where", [(0, 0, 0), (5, 0, 3), (9, 7, 5), (4, 3, 2)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_special_values_equal_stored_matrix(value, where, dtype):
    """An infinite or NaN entry at a corner, a face and inside, and entries at
    the ends of the range that the division by 26 treats apart."""
    dims = (10, 8, 6)
    with hpg.Problem(*dims, beta=0.5, levels=1) as p:
        nat = torch.randn(480, dtype=torch.float64, device=DEV,
                          generator=torch.Generator(device=DEV).manual_seed(4))
        nat[where[0] + 10 * (where[1] + 8 * where[2])] = value
        special, plain = p.to_storage(nat, dtype=dtype), vec(p, dtype, 6)
        for r, z0 in [(special, plain), (plain, special)]:
            zs = []
            for pipe in (1, STORED):
                hpg.set_option(p.h, hpg.HPG_OPT_GS_PIPELINE, pipe)
                z = z0.clone()
                hpg.mg_smooth(p.h, 0, r, z, 1, False)
                zs.append(z)
            assert torch.equal(torch.isnan(zs[0]), torch.isnan(zs[1]))
            assert torch.equal(torch.nan_to_num(zs[0], nan=1.0), torch.nan_to_num(zs[1], nan=1.0))


def product(x, dims, beta):
    """A x in FP64 on the natural grid."""
    nx, ny, nz = dims
    xp = torch.nn.functional.pad(x.view(nz, ny, nx), (1, 1, 1, 1, 1, 1))
    y = 26.0 * x.view(nz, ny, nx)
    for dz in range(3):
        for dy in range(3):
            for dx in range(3):
                if (dx, dy, dz) != (1, 1, 1):
                    y = y + (-1.0 + beta * (dx + dy + dz - 3) / 3.0) * \
                        xp[dz:dz + nz, dy:dy + ny, dx:dx + nx]
    return y.reshape(-1)


@pytest.mark.parametrize("dims", GRIDS)
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_product_against_plain_torch(dims, dtype):
    beta = -0.4
    with hpg.Problem(*dims, beta=beta, levels=1) as p:
        x = vec(p, dtype, 1)
        nat = p.to_natural(x).double()
        y = p.to_natural(p.spmv(x)).double()
        scale = 26.0 * nat.abs() + (product(nat.abs(), dims, 0.0) - 26.0 * nat.abs()).abs() * 1.4
        # 27 FMAs and the rounding of a coefficient: 28 u (|A||x|)_i, twice that for the reference
        u = 2.0 ** (-24 if dtype == torch.float32 else -53)
        assert ((y - product(nat, dims, beta)).abs() <= 2 * 28 * u * scale).all()
        # padding rows are identity rows
        pad = torch.ones(p.n_store(0), dtype=dtype, device=DEV)
        pad[p.to_storage(torch.ones_like(nat)) != 0] = 0
        assert torch.equal(p.spmv(pad), pad)
