"""FP64 handles hold what the pairs of floats of letkf_series64.cu promise (48 bits), at every
column width and over the ratios |G|_F / alpha that the series serves, those whose later terms
run in floats and those just below its end among them.

Tolerance of an analysis: a pair rounds to 2^-48 of its value, A^-1/2 and A^-1 change by at most
kappa times the relative change of A, and the sums of slopes and terms (up to 130) add up some of
these roundings: 8 kappa_hat 2^-47 of the size of the anomalies and increments, and 4 units of
2^-53 of the members themselves for the slopes' and the results' storage. An analysis to 40
bits, or one whose products lost a cross term or a sum's rounding (2^-24), misses it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_1408_7069_gb300 import synth  # noqa: E402
from paper_1408_7069_gb300.letkf import Letkf  # noqa: E402

pytestmark = pytest.mark.gpu

SIGMA2, RHO = 0.01, 1.03


def rms(v):
    return float(np.sqrt(np.mean(np.square(v))))


def anoms(X):
    return X - X.mean(-1, keepdims=True)


def problem(nsub, m, window, taper, ratio, square=False):
    """An ensemble whose largest |G|_F / alpha over the nodes is `ratio`, slopes, geometry and
    the largest kappa_hat."""
    mask = synth.pupil_subap_mask(nsub, 0.0, square)
    geom = oracle.build_geometry(mask, window, taper, 0.0)
    rng = np.random.default_rng(1000 * nsub + 10 * m + window)
    mean = 3 * rng.standard_normal((geom.n_pts, 2, 1))
    P = anoms(rng.standard_normal((geom.n_pts, 2, m)))
    y = rng.standard_normal(geom.p)
    _, _, Yb, _ = oracle.observe(geom, P)
    alpha, top, tr = (m - 1) / RHO, 0.0, 0.0
    for i, t in zip(geom.win_idx, geom.win_tau):
        G = (Yb[i] * (t / SIGMA2)[:, None]).T @ Yb[i] / alpha
        top, tr = max(top, np.linalg.norm(G)), max(tr, np.trace(G))
    s = (ratio / top) ** 0.5
    return mask, geom, mean + s * P, y, 1 + s * s * tr


def analyse(mask, X, y, m, window, taper, **kw):
    f = Letkf(mask, m=m, window=window, taper=taper, rho=RHO, sigma2=SIGMA2, precision=1, **kw)
    f.set_state(torch.from_numpy(X).cuda())
    mean, spread = f.analyze(torch.from_numpy(y).cuda())
    f.sync()
    out = f.get_state().cpu().numpy(), mean.cpu().numpy(), spread.cpu().numpy(), f.stats()
    f.close()
    return out


SIZES = [(3, 5, 3, 1), (4, 8, 3, 1), (4, 9, 4, 0), (5, 16, 5, 1), (5, 17, 3, 1), (5, 24, 9, 1),
         (5, 25, 5, 0), (5, 32, 7, 1)]


@pytest.mark.parametrize("ratio", [0.2, 2.9, 11.0, 24.0, 41.7])
@pytest.mark.parametrize("nsub,m,window,taper", SIZES)
def test_series_to_the_rounding_of_pairs(nsub, m, window, taper, ratio):
    mask, geom, X, y, khat = problem(nsub, m, window, taper, ratio)
    ref = oracle.analysis(geom, X, y, SIGMA2, RHO)
    Xa, mean, spread, st = analyse(mask, X, y, m, window, taper)
    assert st[1:] == (1, geom.n_pts)                    # every node by the series
    tol = 8 * khat * 2.0 ** -47 * (rms(anoms(X)) + rms(ref[1] - X.mean(-1))) \
        + 4 * 2.0 ** -53 * rms(X)
    assert rms(Xa - ref[0]) <= tol
    assert rms(mean - ref[1]) <= tol and rms(spread - ref[2]) <= tol
    # the eigensolve on the same handle's type, FP64 throughout
    Xj, mj, sj, st = analyse(mask, X, y, m, window, taper, max_sweeps=30)
    assert st[1] > 1 or m == 2
    assert rms(Xa - Xj) <= 2 * tol and rms(mean - mj) <= 2 * tol and rms(spread - sj) <= 2 * tol


def gradients(nsub, m, window, taper, X, y, truth, bank, noise, mask, geom, **kw):
    J, g, _ = oracle.closed_loop_grad(geom, truth, y, bank, m, SIGMA2, RHO, 0.999, noise, 9,
                                      len(y), X)
    f = Letkf(mask, m=m, window=window, taper=taper, rho=RHO, sigma2=SIGMA2, a_ar1=0.999,
              noise_std=noise, precision=1, seed=9, bank=bank, **kw)
    f.set_state(torch.from_numpy(X).cuda())
    Jg, gg = f.grad(len(y), torch.from_numpy(y).cuda(), torch.from_numpy(truth).cuda(), 2)
    f.close()
    return J, g, Jg, gg


@pytest.mark.parametrize("ratio", [2.9, 11.0, 41.7, 120.0])
@pytest.mark.parametrize("nsub,m,window,taper", [(3, 6, 3, 1), (4, 12, 3, 1), (4, 20, 5, 1),
                                                 (4, 24, 5, 0), (4, 32, 7, 1)])
def test_gradients_to_the_rounding_of_pairs(nsub, m, window, taper, ratio):
    """Two frames: degrees that keep their terms, that run them backwards, and (120) frames
    whose nodes are divided between series and eigensolve. Tolerance 1e-11: the analysis's
    bound at kappa 40, 2e-12, once more through the second frame and the adjoint."""
    mask, geom, X, y0, _ = problem(nsub, m, window, taper, ratio, square=True)
    geom = oracle.build_geometry(mask, window, taper, window / 4.0)
    rng = np.random.default_rng(nsub + m)
    y = 0.3 * rng.standard_normal((2, geom.p))
    truth = rng.standard_normal((2, geom.n_pts))
    bank = rng.standard_normal((2, 16, 16)).astype(np.float32)
    J, g, Jg, gg = gradients(nsub, m, window, taper, X, y, truth, bank, rms(anoms(X)) / 10, mask, geom)
    assert abs(Jg - J) <= 1e-12 * J
    assert np.all(np.abs(gg - g) <= 1e-11 * np.maximum(np.abs(g), 1e-2 * np.abs(g).max())), (gg, g)
