"""The default tile of a mesh with reduced-degree elements beside the others is about as fast as the best fixed one."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_default_tile_beside_reduced_elements():
    # 2,400 curved elements in FP64, a fifth of them reduced: 1,571 us a step with one element a block, 1,458 with four
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_05709_gb300 import build as B
    from paper_2501_05709_gb300 import cases as C
    from paper_2501_05709_gb300 import fr as F
    from paper_2501_05709_gb300 import workloads as W
    B.build()
    nodes, conn, opts, (rho, vel, pr) = C.naca_setup((0.02, 0.4, 0.12), 60, 20, 2, first_cell=2e-2, order=3,
                                                     precision=F.FR_FP64)
    opts.dt = 1e-7
    u = W.perturbed_uniform(len(nodes), 64, rho, vel, pr, amplitude=0.01, seed=0)
    us = {}
    for tile in (0, 1, 2, 4):
        with F.fr_mesh_load((nodes, conn), opts) as ctx:
            F.fr_set_element_order(ctx, W.sponge_orders(nodes, 3))
            F.fr_state_set(ctx, u)
            if tile:
                F.fr_set_tile(ctx, tile)
            F.fr_rk_step_graph(ctx, 4)
            us[tile] = 1e18
            for _ in range(6):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                F.fr_rk_step_graph(ctx, 4)
                b.record()
                b.synchronize()
                us[tile] = min(us[tile], a.elapsed_time(b) * 250.0)
    assert us[0] <= 1.05 * min(us[1], us[2], us[4])
