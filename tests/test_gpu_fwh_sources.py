"""FW-H sources of panels along the mean flow, where V.n is the small difference of large products: p' against the same
sums with 1e-12 of the largest sample, although the disturbances are 1e-9 of the flow."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_panels_along_the_flow():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import fwh as O
    from paper_2501_05709_gb300 import build as B
    from paper_2501_05709_gb300 import fr as F
    B.build()
    c0, rho0, p0, dt, nt, npts = 340.75, 1.234, 1.0e5, 0.004, 150, 40
    M = np.array([0.3 * np.cos(0.4), 0.3 * np.sin(0.4), 0.0])
    rng = np.random.default_rng(3)
    y = np.stack([np.linspace(-1.0, 1.0, npts) * np.cos(0.4), np.linspace(-1.0, 1.0, npts) * np.sin(0.4), 0.0 * np.arange(npts)], 1)
    n = np.tile([-np.sin(0.4), np.cos(0.4), 0.0], (npts, 1))
    dS = np.full(npts, 0.05)
    U = c0 * M
    # disturbances on the grid of the flow's last bits, so that V - U is exact, and no pressure: Q and its derivative only
    V = U + 1e-7 * rng.standard_normal((nt, npts, 3)) * np.array([1.0, 1.0, 0.0])
    hist = np.concatenate([np.full((nt, npts, 1), rho0), V, np.full((nt, npts, 1), p0)], axis=-1)
    obs = np.array([[-12.0, 20.0, 1.0]])
    dev = [torch.tensor(np.ascontiguousarray(a), device="cuda") for a in (hist, y, n, dS)]
    p, k, _ = F.fwh_integrate(*dev, dt, 0.0, obs, M, c0, rho0, p0)
    # the oracle with Q in extended precision: u.n, since rho = rho0 leaves nothing else
    L = np.longdouble
    un = ((V.astype(L) - U.astype(L)) * n.astype(L)).sum(-1)
    src = O.source_terms
    try:
        O.source_terms = lambda *a: ((L(rho0) * un).astype(float), src(*a)[1])
        ref = O.fwh_integrate(hist, y, n, dS, dt, obs[0], M, c0, rho0, p0)[1]
    finally:
        O.source_terms = src
    got = p.cpu().numpy()[0, :k[0]]
    # Un = U.n is 1e-15 here: Q = rho0 (u.n + Un) - rho0 Un is off by some 1e-16 of |Un| and of u.n (1e-7), while U is 100
    assert len(ref) == k[0] and np.max(np.abs(got - ref)) <= 1e-12 * np.max(np.abs(ref))
