"""FW-H calls of many observers and of long records: more observers than a launch takes, several batches of panels, and
an observer's result independent of the other observers of its call."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

M, C0, RHO0, P0, DT = [0.3, 0.05, 0.1], 340.75, 1.234, 1.0e5, 0.004


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_05709_gb300 import build as B
    B.build()


def _record(nt, polar, seed=0):
    from paper_2501_05709_gb300 import workloads as W
    y, n, dS = W.sphere_surface(1.0, polar, 2 * np.pi / 9)
    rng = np.random.default_rng(seed)
    w = lambda: rng.standard_normal((nt, len(y)))
    hist = np.stack([RHO0 + 1e-3 * w()] + [C0 * M[i] + w() for i in range(3)] + [P0 + 400.0 * w()], axis=-1)
    return hist, y, n, dS


def _gpu(rec, obs, copies=1):
    from paper_2501_05709_gb300 import fr as F
    dev = [torch.as_tensor(np.ascontiguousarray(a)).cuda() for a in rec]
    p, nt, t0 = F.fwh_integrate(*dev, DT, 0.0, obs, M, C0, RHO0, P0, Lspan=0.3, ncopies=copies)
    p = p.cpu().numpy()
    return [p[k, :nt[k]] for k in range(len(obs))]


def _oracle(rec, o, copies=1):
    # panel positions and step in extended precision carry over to delays and source times (t - R / c0) / dt, whose
    # rounding in double is 1e-12 of a step at the end of 30,000 steps; sources and sums stay in double
    from oracle import fwh as O
    hist, y, n, dS = rec
    return O.fwh_integrate(hist, y.astype(np.longdouble), n, dS, np.longdouble(DT), o, M, C0, RHO0, P0, Lspan=0.3,
                           ncopies=copies)[1]


def _circle(n):
    a = np.linspace(0.0, 2 * np.pi, n, endpoint=False)
    return np.stack([30.0 * np.cos(a), 30.0 * np.sin(a), 5.0 * np.sin(3 * a)], axis=1)


@pytest.mark.parametrize("polar, copies", [(5, 1), (24, 3), (120, 3)])
def test_an_observer_has_the_same_bits_in_any_call(polar, copies):
    rec, obs = _record(260, polar), _circle(40)
    out = _gpu(rec, obs, copies)
    for k in (0, 17, 39):
        assert np.array_equal(out[k], _gpu(rec, obs[k:k + 1], copies)[0])
        assert np.array_equal(out[k], _gpu(rec, obs[[3, k, 8]], copies)[1])


def test_more_observers_than_a_launch_takes():
    # with one that is summed in double in each launch: a panel's outlier reaches its window's end only there
    rec, obs = _record(60, 4), _circle(5000)
    rec[0][30, 2, 4] = 1e25
    out = _gpu(rec, obs)
    for k in (0, 1, 2047, 2048, 4095, 4096, 4999):
        ref = _oracle(rec, obs[k])
        m = np.abs(ref) < 1e12
        assert m.sum() > 30 and np.max(np.abs(out[k] - ref)[m]) <= 1e-12 * np.max(np.abs(ref[m]))
    rec[0][30, 2, 4] = P0
    out = _gpu(rec, obs)
    for k in (0, 1, 2047, 2048, 4095, 4096, 4999):
        ref = _oracle(rec, obs[k])
        assert np.max(np.abs(out[k] - ref)) <= 1e-12 * np.max(np.abs(ref))


@pytest.mark.parametrize("outlier", [False, True])
def test_several_batches_of_panels(outlier):
    # 160 MiB of series hold 96 panels of such a record: three batches
    rec, obs = _record(30000, 34), _circle(3)[:1]
    assert 192 < len(rec[1]) <= 288
    if outlier:
        rec[0][20000, 150, 4] = 1e25
    out, ref = _gpu(rec, obs)[0], _oracle(rec, obs[0])
    m = np.abs(ref) < 1e12
    assert m.sum() > 29900 and np.max(np.abs(out - ref)[m]) <= 1e-12 * np.max(np.abs(ref[m]))
