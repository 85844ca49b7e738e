"""The adaptive step costs a small part of a step whatever the state: in FP64, where every element's rate is evaluated,
and in FP32 on a uniform flow, where the FP32 bounds leave no element out."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _step_us(F, mesh, opts, u, cfl):
    best = 1e18
    with F.fr_mesh_load(mesh, opts) as ctx:
        if cfl:
            F.fr_set_adaptive_dt(ctx, cfl)
        F.fr_state_set(ctx, u)
        F.fr_rk_step_graph(ctx, 8)
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            F.fr_rk_step_graph(ctx, 8)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b) * 125.0)
    return best


# rates of 1,000 elements take 15 us beside a step of 250 us (FP64, p = 3) and 10 us beside one of 20 us (FP32, p = 2)
@pytest.mark.parametrize("prec, p, most", [("fp64", 3, 1.3), ("fp32", 2, 2.5)])
def test_rates_of_a_uniform_flow(prec, p, most):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_05709_gb300 import build as B
    from paper_2501_05709_gb300 import fr as F
    from paper_2501_05709_gb300 import workloads as W
    B.build()
    mesh = W.box_mesh(3, 10, 0.0, 1.0, q=1)
    opts = F.options(order=p, precision=F.FR_FP64 if prec == "fp64" else F.FR_FP32, dt=1e-12)
    u = W.perturbed_uniform(1000, (p + 1) ** 3, 1.0, [0.3, 0.2, 0.1], 1.0, amplitude=0.0)
    fixed, adaptive = (_step_us(F, mesh, opts, u, cfl) for cfl in (0.0, 1e-9))
    assert adaptive <= most * fixed
