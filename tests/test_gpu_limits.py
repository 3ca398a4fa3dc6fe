"""Sizes at the edge of an SM's shared memory."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_1408_7069_gb300 import synth  # noqa: E402
from paper_1408_7069_gb300.letkf import Letkf, LetkfError  # noqa: E402

pytestmark = pytest.mark.gpu

SIGMA2, RHO = 0.01, 1.03


def inputs(f, seed=1, scale=0.06):
    """An ensemble of loop-sized anomalies and slopes of a handle."""
    rng = np.random.default_rng(seed)
    dt = np.float64 if f.precision else np.float32
    X = 3 * rng.standard_normal((*f.state_shape[:-1], 1)) + scale * rng.standard_normal(f.state_shape)
    return X.astype(dt), rng.standard_normal(f.p).astype(dt)


def analysis(f, X, y):
    f.set_state(torch.from_numpy(X).cuda())
    mean, spread = f.analyze(torch.from_numpy(y).cuda())
    f.sync()
    return mean.cpu().numpy(), spread.cpu().numpy(), f.get_state().cpu().numpy()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("m", [17, 24, 25, 32])
def test_the_largest_window_of_17_to_32_members(m, precision):
    """A window of 25 is the largest whose 4 x 4 node tile fits an SM; the analysis to the
    tolerances of its precision."""
    mask = synth.pupil_subap_mask(6, 0.0)
    kw = dict(m=m, taper=1, rho=RHO, sigma2=SIGMA2, precision=precision)
    f = Letkf(mask, window=25, **kw)
    if precision == 0:
        f.set_tile_shape(1, 1)                          # 4 x 4
    X, y = inputs(f)
    mean, spread, _ = analysis(f, X, y)
    f.close()
    geom = oracle.build_geometry(mask, 25, 1, 0.0)
    ref = oracle.analysis(geom, X.astype(np.float64), y.astype(np.float64), SIGMA2, RHO)
    for got, want, tol in ((mean, ref[1], (1e-4, 1e-9)), (spread, ref[2], (1e-3, 1e-8))):
        assert np.linalg.norm(got - want) <= tol[precision] * np.linalg.norm(want)
    with pytest.raises(LetkfError):
        Letkf(mask, window=26, **kw)


def handle(nsub, window, bank=False, **kw):
    if bank:
        kw.update(bank=np.random.default_rng(3).standard_normal((2, 16, 16)).astype(np.float32),
                  a_ar1=0.99, noise_std=0.01)
    return Letkf(synth.pupil_subap_mask(nsub, 0.0), window=window, rho=RHO, sigma2=SIGMA2, **kw)


@pytest.mark.parametrize("big,small",
                         [(dict(window=9, m=24, precision=1, bank=True), dict(window=3, m=10, precision=1)),
                          (dict(window=9, m=24, precision=1, bank=True), dict(window=3, m=24, precision=1)),
                          (dict(window=11, m=32, precision=1, bank=True),
                           dict(window=1, m=32, precision=1, max_sweeps=20)),
                          (dict(window=15, m=24, bank=True), dict(window=3, m=24)),
                          (dict(window=15, m=64), dict(window=3, m=64)),
                          (dict(window=15, m=16, bank=True, max_sweeps=20), dict(window=1, m=8)),
                          (dict(window=5, m=64, partition=3), dict(window=3, m=64, partition=4)),
                          (dict(window=5, m=64, partition=3, max_sweeps=20), dict(window=3, m=64, partition=4)),
                          (dict(window=3, m=64, taper=0, partition=1), dict(window=3, m=34, taper=0, partition=1))],
                         ids=["fp64-widths", "fp64", "fp64-beside-sweeps", "fp32", "wide", "sweeps",
                              "domains", "domain-sweeps", "global"])
def test_a_handle_keeps_its_limits_when_smaller_ones_are_made(big, small):
    """Two handles in one process, the second with smaller windows, domains or ensembles: the
    first goes on as before, in analyses, loops and gradients, the second too."""
    f = handle(12, **big)
    X, y = inputs(f)
    before = analysis(f, X, y)
    frames = torch.from_numpy(np.stack([y, y])).cuda()
    truth = torch.zeros((2, f.n_pts), dtype=f.dtype, device="cuda")

    def loops():
        if not big.get("bank"):
            return []
        f.set_state(torch.from_numpy(X).cuda())
        f.set_frame(0)
        f.run(2, frames, use_graph=False)
        f.sync()
        out = [f.get_state().cpu().numpy()]
        if f.m <= 32:
            f.set_state(torch.from_numpy(X).cuda())
            f.set_frame(0)
            J, g = f.grad(2, frames, truth)
            out += [np.array(J), np.asarray(g)]
        return out
    loop = loops()
    g = handle(6, **small)
    Xs, ys = inputs(g)
    analysis(g, Xs, ys)
    after = analysis(f, X, y)
    assert all(np.array_equal(a, b) for a, b in zip(before, after))
    assert all(np.array_equal(a, b) for a, b in zip(loop, loops()))
    g.close()
    f.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_a_refused_handle_leaves_no_error_behind(precision):
    """A window too wide for an SM is refused by a runtime call; the calls of other handles
    that follow in the thread do not find that call's error."""
    def grad():
        f = handle(6, 3, bank=True, m=10, precision=precision)
        X, y = inputs(f)
        f.set_state(torch.from_numpy(X).cuda())
        out = f.grad(2, torch.from_numpy(np.stack([y, y])).cuda(),
                     torch.zeros((2, f.n_pts), dtype=f.dtype, device="cuda"))
        f.close()
        return out
    want = grad()
    with pytest.raises(LetkfError):
        handle(6, 31, m=32, precision=precision)
    got = grad()
    assert got[0] == want[0] and np.array_equal(got[1], want[1])
