"""The adaptive step of FP32 states, whose FP32 bounds leave most elements out, against the rate of every point in
double: ties everywhere (a uniform state), one element that decides, hypersonic states (pressure a small difference),
and points without a positive pressure (left out of the maximum, their elements' other points not)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

GAMMA = 1.4


@pytest.mark.parametrize("visc", [False, True])
@pytest.mark.parametrize("kind", ["uniform", "noise", "one", "hypersonic", "negative"])
def test_step_is_the_double_maximum(kind, visc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle.mesh import Mesh
    from oracle.timestep import element_length
    from paper_2501_05709_gb300 import build as B
    from paper_2501_05709_gb300 import fr as F
    from paper_2501_05709_gb300 import workloads as W
    B.build()
    p, mu, rng = 2, 0.02, np.random.default_rng(5)
    meshes = [W.box_mesh(3, [5, 4, 3], 0.0, 1.0, q=2, curve=0.1, seed=k) for k in (1, 2)]
    E, nsp = 60, (p + 1) ** 3
    rho, V, pr = np.ones((2 * E, nsp)), np.full((3, 2 * E, nsp), 0.3), np.ones((2 * E, nsp))
    if kind == "noise":
        V = V + 1e-3 * rng.standard_normal(V.shape)
    if kind == "one":
        V[0, 77, 3] = 4.0
    if kind == "hypersonic":
        V = 50.0 * (1.0 + 0.1 * rng.random(V.shape))
        rho = 1.0 + 0.2 * rng.random(rho.shape)
    u = np.concatenate([rho[None], rho * V, (pr / (GAMMA - 1) + 0.5 * rho * (V ** 2).sum(0))[None]])
    if kind == "negative":
        u[4, 5, :] = 0.0
        u[4, 70, 2:9] = -1.0
    u = np.ascontiguousarray(np.moveaxis(u, 0, 1).astype(np.float32).astype(np.float64))
    with F.fr_mesh_load(meshes, F.options(order=p, precision=F.FR_FP32, viscous=visc, mu=mu if visc else 0.0)) as ctx:
        F.fr_set_adaptive_dt(ctx, 1e-9)        # the state stays what it is
        F.fr_state_set(ctx, u)
        F.fr_rk_step(ctx, 1)
        got = [F.fr_cand_dt(ctx, k) for k in (0, 1)]
    r, m2, k = u[:, 0], (u[:, 1:4] ** 2).sum(1), (p + 1) ** 2
    gm1 = float(np.float32(GAMMA - 1.0))
    with np.errstate(invalid="ignore"):
        v = np.sqrt(m2) / r + np.sqrt(float(np.float32(GAMMA)) * gm1 * (u[:, 4] - 0.5 * m2 / r) / r)
    vmax = np.max(np.where(np.isfinite(v), v, 0.0), axis=1)
    for c, mesh in enumerate(meshes):
        h = element_length(Mesh(*mesh, p)).astype(np.float32).astype(float)
        e = slice(c * E, (c + 1) * E)
        lam = vmax[e] * k / h
        if visc:
            lam = lam + np.max(float(np.float32(mu)) / r[e], axis=1) * k * k / (h * h)
        assert abs(got[c] - 1e-9 / lam.max()) <= 1e-6 * got[c]     # h in FP32: half a unit, and its order of rounding
        # no element is left out: every element's rate is at most the one taken
        assert np.all(lam <= 1e-9 / got[c] * (1 + 1e-6))
