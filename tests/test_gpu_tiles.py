"""Elements per block: every tile that fr_set_tile takes runs and gives the bits of the default one, the default tile is
about as fast as the best fixed one, meshes with walls run about as fast as periodic ones, and fr_autotune times the
tile in use beside its candidates."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_05709_gb300 import build as B
    B.build()


def _load(dim, n, p, prec, visc=True, walls=False, curve=0.0):
    from paper_2501_05709_gb300 import fr as F
    from paper_2501_05709_gb300 import workloads as W
    mesh = W.box_mesh(dim, n, 0.0, 1.0, q=2 if curve else 1, curve=curve, walls_y=walls)
    ctx = F.fr_mesh_load(mesh, F.options(order=p, precision=prec, viscous=visc, mu=0.001 if visc else 0.0, dt=1e-9))
    g = torch.Generator(device="cuda").manual_seed(1)
    r = 0.05 * (2 * torch.rand((ctx.nelem, ctx.nvar, ctx.nsp), generator=g, device="cuda", dtype=torch.float64) - 1)
    u = r.clone()
    u[:, 0] += 1.0
    u[:, 1:-1] += 0.3
    u[:, -1] += 3.0
    return ctx, u.to(torch.float64 if prec == F.FR_FP64 else torch.float32)


def _residual_us(ctx, u):
    from paper_2501_05709_gb300 import fr as F
    R = torch.empty_like(u)
    best = 1e18
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        F.fr_residual(ctx, u, R)
        a.record()
        for _ in range(10):
            F.fr_residual(ctx, u, R)
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) * 100.0)
    return best


# orders, precisions and meshes whose kernels hold the most registers
@pytest.mark.parametrize("prec, dim, p, walls, curve", [
    ("fp64", 3, 2, True, 0.0), ("fp64", 3, 2, False, 0.0), ("fp64", 3, 4, True, 0.0), ("fp64", 2, 4, True, 0.0),
    ("fp64", 3, 2, False, 0.05), ("fp32", 3, 2, False, 0.0), ("fp32", 3, 4, False, 0.0), ("fp32", 3, 4, False, 0.05),
    ("fp32", 2, 4, True, 0.0), ("tf32", 3, 4, False, 0.0), ("tf32", 3, 3, True, 0.0)])
def test_every_tile_that_is_taken_runs(prec, dim, p, walls, curve):
    from paper_2501_05709_gb300 import fr as F
    ctx, u = _load(dim, [3, 4, 3][:dim], p, {"fp64": F.FR_FP64, "fp32": F.FR_FP32, "tf32": F.FR_TF32_TC}[prec], True, walls,
                   curve)
    with ctx:
        ref, R = torch.empty_like(u), torch.empty_like(u)
        F.fr_residual(ctx, u, ref)
        taken = 0
        for tile in range(1, 33):
            try:
                F.fr_set_tile(ctx, tile)
            except F.FrError:
                continue
            taken += 1
            F.fr_residual(ctx, u, R.zero_())
            assert torch.equal(R, ref), tile
        assert taken >= 4


@pytest.mark.parametrize("dim, n, p, visc", [(2, [250, 256], 2, False), (3, [14, 15, 11], 4, True), (3, [28, 28, 28], 1, False)])
def test_the_default_tile_is_about_the_best(dim, n, p, visc):
    from paper_2501_05709_gb300 import fr as F
    ctx, u = _load(dim, n, p, F.FR_FP32, visc)
    with ctx:
        default = _residual_us(ctx, u)
        fixed = []
        for tile in (2, 4, 8):
            F.fr_set_tile(ctx, tile)
            fixed.append(_residual_us(ctx, u))
    assert default <= 1.1 * min(fixed)


def test_walls_cost_little():
    # 22,000 elements at p = 4: two faces in 84 carry a boundary state
    from paper_2501_05709_gb300 import fr as F
    us = []
    for walls in (False, True):
        ctx, u = _load(3, [27, 28, 29], 4, F.FR_FP32, True, walls)
        with ctx:
            us.append(_residual_us(ctx, u))
    assert us[1] <= 1.25 * us[0]


def test_autotune_times_the_tile_in_use():
    from paper_2501_05709_gb300 import fr as F
    ctx, u = _load(3, [6, 6, 6], 2, F.FR_FP32)
    with ctx:
        F.fr_state_set(ctx, u.double())
        count = []
        for tile in (4, 3):                  # one of the candidates, and one that is none
            F.fr_set_tile(ctx, tile)
            before = F.fr_launch_count(ctx)
            F.fr_autotune(ctx)
            count.append(F.fr_launch_count(ctx) - before)
    assert count[1] == count[0] // 5 * 6
