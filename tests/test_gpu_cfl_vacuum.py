"""The adaptive step of FP32 states where pressures are zero within FP32 rounding: a point whose pressure is negative in
double is left out of the maximum, so an FP32 pressure that rounds to a positive value must not rule other elements out."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

GAMMA = 1.4


@pytest.mark.parametrize("visc", [False, True])
@pytest.mark.parametrize("ulps", [1, 2, 4])
def test_points_of_vanishing_pressure_rule_nothing_out(ulps, visc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle.mesh import Mesh
    from oracle.timestep import element_length
    from paper_2501_05709_gb300 import build as B
    from paper_2501_05709_gb300 import fr as F
    from paper_2501_05709_gb300 import workloads as W
    B.build()
    p, mu, rng = 2, 0.02, np.random.default_rng(11)
    mesh = W.box_mesh(3, [5, 4, 3], 0.0, 1.0, q=1)
    E, nsp = 60, (p + 1) ** 3
    rho, V = np.ones((E, nsp)), np.full((3, E, nsp), 0.3)
    dead = slice(20, 40)                                     # elements of fast points at (almost) no pressure
    rho[dead] = 1.0 + rng.random((20, nsp))
    V[:, dead] = 50.0 * (1.0 + 0.1 * rng.random((3, 20, nsp)))
    u = np.concatenate([rho[None], rho * V, (1.0 / (GAMMA - 1) + 0.5 * rho * (V ** 2).sum(0))[None]])
    u = np.ascontiguousarray(np.moveaxis(u, 0, 1)).astype(np.float32)
    r64 = u.astype(np.float64)
    ke = 0.5 * (r64[dead, 1:4] ** 2).sum(1) / r64[dead, 0]
    e = ke.astype(np.float32)
    e = np.where(e.astype(np.float64) >= ke, np.nextafter(e, np.float32(0)), e)   # the last float below the kinetic energy
    for _ in range(ulps - 1):
        e = np.nextafter(e, np.float32(0))
    u[dead, 4] = e
    u = u.astype(np.float64)
    with F.fr_mesh_load(mesh, F.options(order=p, precision=F.FR_FP32, viscous=visc, mu=mu if visc else 0.0)) as ctx:
        F.fr_set_adaptive_dt(ctx, 1e-9)
        F.fr_state_set(ctx, u)
        F.fr_rk_step(ctx, 1)
        got = F.fr_cand_dt(ctx, 0)
    m2, k, gm1 = (u[:, 1:4] ** 2).sum(1), (p + 1) ** 2, float(np.float32(GAMMA - 1.0))
    pr = gm1 * (u[:, 4] - 0.5 * m2 / u[:, 0])
    assert np.all(pr[dead] < 0.0) and np.all(np.delete(pr, np.r_[dead], 0) > 0.0)
    v = np.sqrt(m2) / u[:, 0] + np.sqrt(float(np.float32(GAMMA)) * np.maximum(pr, 0.0) / u[:, 0])
    h = element_length(Mesh(*mesh, p)).astype(np.float32).astype(float)
    lam = np.where(pr < 0.0, 0.0, v).max(1) * k / h
    if visc:
        lam = lam + np.max(float(np.float32(mu)) / u[:, 0], axis=1) * k * k / (h * h)
    assert abs(got - 1e-9 / lam.max()) <= 1e-6 * got
