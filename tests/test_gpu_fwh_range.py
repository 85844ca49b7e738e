"""FW-H sums of records with a large range in time against the FP64 oracle, every observer sample relative to the samples
around it: a decay by ten orders of magnitude, and one finite outlier, which only the samples whose stencils reach it may
feel.  The bound is that of the other FW-H tests, 1e-12, of the local size instead of the largest sample: a double holds
sources, products and sums to some 1e-16 of it, and source times to some 1e-14 of a step."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

C0, RHO0, P0, DT = 340.75, 1.234, 1.0e5, 0.004


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_05709_gb300 import build as B
    B.build()


def _record(nt, env, polar=6, seed=0):
    """Disturbances of a medium at rest (every source is a product of disturbances, without cancellation)."""
    from paper_2501_05709_gb300 import workloads as W
    y, n, dS = W.sphere_surface(1.0, polar, 2 * np.pi / 9)
    rng = np.random.default_rng(seed)
    t = DT * np.arange(nt)[:, None]
    wave = lambda: env[:, None] * np.sin(20.0 * t * (1 + rng.random(len(y))) + 6.28 * rng.random(len(y)))
    hist = np.stack([RHO0 + 1e-3 * wave(), wave(), wave(), wave(), P0 + 400.0 * wave()], axis=-1)
    return hist, y, n, dS


def _both(hist, y, n, dS, obs, copies=1):
    from oracle import fwh as O
    from paper_2501_05709_gb300 import fr as F
    dev = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    p, nt, _ = F.fwh_integrate(dev(hist), dev(y), dev(n), dev(dS), DT, 0.0, obs, [0.0] * 3, C0, RHO0, P0, Lspan=0.4,
                               ncopies=copies)
    p = p.cpu().numpy()
    ref = [O.fwh_integrate(hist, y, n, dS, DT, o, [0.0] * 3, C0, RHO0, P0, Lspan=0.4, ncopies=copies)[1] for o in obs]
    assert [len(r) for r in ref] == list(nt)
    return [p[k, :nt[k]] for k in range(len(obs))], ref


OBS = np.array([[20.0, 3.0, 1.0], [0.0, -15.0, 2.0], [-7.0, 9.0, 30.0]])


@pytest.mark.parametrize("copies", [1, 3])
@pytest.mark.parametrize("grows", [False, True])
def test_decay_and_growth(grows, copies):
    nt = 700
    env = 10.0 ** (-10.0 * np.arange(nt) / nt)
    out, ref = _both(*_record(nt, env[::-1].copy() if grows else env), OBS, copies)
    for a, b in zip(out, ref):
        for i in range(0, len(b), 16):
            assert np.max(np.abs((a - b)[i:i + 16])) <= 1e-12 * np.max(np.abs(b[i:i + 16]))


@pytest.mark.parametrize("big", [1e12, 1e30, 1e200, 1e300])
def test_one_finite_outlier(big):
    hist, y, n, dS = _record(400, np.ones(400))
    clean, _ = _both(hist, y, n, dS, OBS)
    hist[150, 7, 4] = big
    out, ref = _both(hist, y, n, dS, OBS)
    for a, b, c in zip(out, ref, clean):
        far = np.abs(b - c) <= 1e-9 * np.max(np.abs(c))      # not reached by the outlier
        assert far.sum() >= len(b) - 12
        assert np.max(np.abs(a - b)[far]) <= 1e-12 * np.max(np.abs(b[far]))
        assert np.max(np.abs(a - b)[~far]) <= 1e-12 * np.max(np.abs(b))


def test_a_diverged_record_costs_no_more_than_the_sums_in_double():
    from paper_2501_05709_gb300 import fr as F
    hist, y, n, dS = _record(600, np.ones(600), polar=24)
    dev = [torch.tensor(np.ascontiguousarray(a), device="cuda") for a in (hist, y, n, dS)]
    a = np.linspace(0.0, 6.0, 24)
    obs = np.stack([20.0 * np.cos(a), 20.0 * np.sin(a), 0.0 * a], axis=1)

    def best():
        t = []
        for _ in range(6):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            F.fwh_integrate(*dev, DT, 0.0, obs, [0.0] * 3, C0, RHO0, P0, Lspan=0.4, ncopies=3)
            t.append(time.perf_counter() - t0)
        return min(t)

    clean = best()
    dev[0][60:] = float("nan")
    # the sums in double take about four times those in fixed point (FP64 pipe against integer pipe)
    assert best() <= 8.0 * clean
