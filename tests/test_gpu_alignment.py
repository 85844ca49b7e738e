"""Residuals of states at any multiple of their value's size: the staging copies 16 bytes at a time from any start, and
gives the same bits as from an aligned array."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("curve", [0.0, 0.1])
def test_residual_of_a_shifted_state(dim, p, prec, curve):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_05709_gb300 import build as B
    from paper_2501_05709_gb300 import fr as F
    from paper_2501_05709_gb300 import workloads as W
    B.build()
    mesh = W.box_mesh(dim, [3, 4, 5][:dim], 0.0, 1.0, q=2 if p > 1 else 1, curve=curve if p > 1 else 0.0, seed=1)
    dt = torch.float64 if prec == "fp64" else torch.float32
    opts = F.options(order=p, precision=F.FR_FP64 if prec == "fp64" else F.FR_FP32, viscous=True, mu=0.01)
    with F.fr_mesh_load(mesh, opts) as ctx:
        x = F.fr_sp_coords(ctx)
        u = torch.tensor(np.ascontiguousarray(np.moveaxis(W.random_smooth_state(x, seed=3), 0, 1)), dtype=dt, device="cuda")
        R = [torch.empty_like(u) for _ in range(4)]
        room = torch.empty(u.numel() + 4, dtype=dt, device="cuda")
        for k in range(4):
            v = room[k:k + u.numel()].view(u.shape)
            v.copy_(u)
            F.fr_residual(ctx, v, R[k])
        torch.cuda.synchronize()
        assert torch.isfinite(R[0]).all()
        assert all(torch.equal(R[0], R[k]) for k in (1, 2, 3))
