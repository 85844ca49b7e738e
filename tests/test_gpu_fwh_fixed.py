"""FW-H sums in fixed point against the FP64 oracle where the kernel's tiles end: the shortest records, one sample
more or less than a warp's 124 and a block's 992, more panel copies than one set-up pass (96), sources of very
different size, silent panels, and records with NaN or infinities (summed in double)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

M, C0, RHO0, DT = [0.3, 0.05, 0.1], 340.75, 1.234, 0.004


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_05709_gb300 import build as B
    B.build()


def _record(nt, polar=6, seed=0):
    from paper_2501_05709_gb300 import workloads as W
    y, n, dS = W.sphere_surface(1.0, polar, 2 * np.pi / 9)
    fld = W.monopole_field(y[None], DT * np.arange(nt)[:, None], M)
    hist = np.concatenate([fld["rho"][..., None], fld["vel"], fld["p"][..., None]], axis=-1)
    rng = np.random.default_rng(seed)
    hist[..., 4] += 5.0 * rng.standard_normal(hist.shape[:2])      # every sample its own
    return hist, y, n, dS, fld["p0"]


def _both(hist, y, n, dS, p0, obs, Lspan=0.0, copies=1):
    from oracle import fwh as O
    from paper_2501_05709_gb300 import fr as F
    dev = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    obs = np.atleast_2d(obs)
    p, nt, t0 = F.fwh_integrate(dev(hist), dev(y), dev(n), dev(dS), DT, 0.0, obs, M, C0, RHO0, p0, Lspan=Lspan,
                                ncopies=copies)
    ref = [O.fwh_integrate(hist, y, n, dS, DT, o, M, C0, RHO0, p0, Lspan=Lspan, ncopies=copies)[1] for o in obs]
    got = p.cpu().numpy()
    assert [len(r) for r in ref] == list(nt)
    return [got[k, :nt[k]] for k in range(len(obs))], ref


# sample counts: the record's window is a few samples shorter than the record (delays differ by 2 m / c0 = 1.5 dt)
@pytest.mark.parametrize("nt", [7, 8, 9, 12, 125, 126, 127, 128, 994, 995, 996, 997])
def test_window_lengths_at_the_tile_edges(nt):
    out, ref = _both(*_record(nt, seed=nt), [[20.0, 3.0, 1.0], [0.0, -15.0, 2.0]])
    for a, b in zip(out, ref):
        assert np.max(np.abs(a - b)) <= 1e-12 * np.max(np.abs(b))


@pytest.mark.parametrize("copies", [3, 33, 97, 101])
def test_more_copies_than_one_setup_pass(copies):
    out, ref = _both(*_record(300, polar=4), [[0.0, 30.0, 1.0]], Lspan=0.05, copies=copies)
    assert np.max(np.abs(out[0] - ref[0])) <= 1e-12 * np.max(np.abs(ref[0]))


def test_panels_of_very_different_size_and_silent_ones():
    hist, y, n, dS, p0 = _record(200)
    U = C0 * np.array(M)
    k = np.arange(len(y))
    quiet = np.concatenate([[RHO0], U, [p0]])
    hist = quiet + (hist - quiet) * (10.0 ** -(k % 12))[None, :, None]
    hist[:, k % 5 == 0] = quiet
    out, ref = _both(hist, y, n, dS, p0, [[20.0, 3.0, 1.0]])
    assert np.max(np.abs(out[0] - ref[0])) <= 1e-12 * np.max(np.abs(ref[0]))
    out, _ = _both(np.broadcast_to(quiet, hist.shape).copy(), y, n, dS, p0, [[20.0, 3.0, 1.0]])
    assert np.max(np.abs(out[0])) <= 1e-9        # p0 is about 1e5


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_records_that_do_not_fit_fixed_point(bad):
    # one panel's one sample: only the observer samples whose stencils reach it change
    hist, y, n, dS, p0 = _record(200)
    hist[90, 7, 4] = bad
    with np.errstate(all="ignore"):
        out, ref = _both(hist, y, n, dS, p0, [[20.0, 3.0, 1.0]])
    a, b = out[0], ref[0]
    m = np.isfinite(b)
    assert np.array_equal(np.isfinite(a), m)
    assert m.sum() > 150 and np.max(np.abs(a[m] - b[m])) <= 1e-12 * np.max(np.abs(b[m]))
