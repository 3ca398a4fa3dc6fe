"""The root, the mean and the status of the global ETKF of more than 64 members
(letkf_global.cu) against the FP64 oracle, where they can go wrong."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from oracle import letkf_domains as LD  # noqa: E402
from paper_1408_7069_gb300 import synth  # noqa: E402
from paper_1408_7069_gb300.letkf import Letkf, LetkfError  # noqa: E402

pytestmark = pytest.mark.gpu

SIGMA2, RHO = 0.01, 1.03
UNIT = 2.0 ** -24


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


def problem(nsub, m, seed=0):
    """Geometry, means and unit anomalies [n, 2, m] of an ensemble, slopes, and the Gram of
    its unit anomalies' slopes over sigma^2."""
    mask = synth.pupil_subap_mask(nsub, 0.0)
    dg = LD.build_domains(mask, 1, 3, 0, 0.0)
    rng = np.random.default_rng(seed + nsub + m)
    n = dg.geom.n_pts
    mean = 3 * rng.standard_normal((n, 2, 1))
    P = rng.standard_normal((n, 2, m))
    P -= P.mean(-1, keepdims=True)
    _, _, Yb, _ = oracle.observe(dg.geom, P)
    y = rng.standard_normal(dg.geom.p).astype(np.float32)
    return mask, dg, mean, P, y, Yb.T @ Yb / SIGMA2


def analyse(mask, m, X, y):
    f = Letkf(mask, m=m, window=3, taper=0, rho=RHO, sigma2=SIGMA2, partition=1)
    f.set_state(torch.from_numpy(X).cuda())
    mean, spread = f.analyze(torch.from_numpy(y).cuda())
    try:
        f.sync()
        return mean.cpu().numpy(), spread.cpu().numpy(), f.get_state().cpu().numpy()
    finally:
        f.close()


@pytest.mark.parametrize("kappa", [12.5, 14.0, 50.0, 100.0, 530.0, 3500.0])
def test_the_root_converges_in_the_directions_without_slopes(kappa):
    """Most of the eigenvalues of A sit at their lower bound (128 members, at most 32 slopes),
    the last to converge: what is left when the iteration stops is an error of the spread. At
    |A|_F / alpha of 14, 530 and 3500 a step ends just short of the others. Tolerance: the
    rounding of the products, 16 units of 2^-24, and sqrt(kappa) of them that Z's own
    condition adds."""
    m, alpha = 128, 127 / RHO
    mask, dg, mean, P, y, G = problem(4, m)
    lo, hi = 1e-6, 1e3
    for _ in range(60):                                 # the scale of the anomalies for kappa
        s = (lo * hi) ** 0.5
        big = np.linalg.norm(alpha * np.eye(m) + s * s * G) > kappa * alpha
        lo, hi = (lo, s) if big else (s, hi)
    X = (mean + s * P).astype(np.float32)
    _, rmean, rspread = LD.analysis_domains(dg, X.astype(np.float64), y.astype(np.float64), SIGMA2,
                                            RHO)
    gm, gs, _ = analyse(mask, m, X, y)
    assert rel(gs, rspread) <= (16 + kappa ** 0.5) * UNIT


@pytest.mark.parametrize("nsub,m", [(9, 192), (10, 128), (16, 320)])
@pytest.mark.parametrize("scale", [0.05, 3.0, 10.0, 30.0])
def test_the_mean_is_that_of_the_refined_solve(nsub, m, scale):
    """|A|_F / alpha from 16 to 4e6: the mean's increment X' wbar is as accurate as the FP64
    refinement leaves wbar and the FP32 slopes allow, whatever the FP32 root's rounding, 2^-23
    |A|_F / alpha in the anomalies, does. Tolerance, relative to the increment: the slopes'
    rounding, 2^-24 of each, amplified by sqrt(kappa) in the root mean square, a few times."""
    mask, dg, mean, P, y, G = problem(nsub, m)
    alpha = (m - 1) / RHO
    X = (mean + scale * P).astype(np.float32)
    _, rmean, _ = LD.analysis_domains(dg, X.astype(np.float64), y.astype(np.float64), SIGMA2, RHO)
    kappa = np.linalg.norm(alpha * np.eye(m) + scale ** 2 * G) / alpha
    _, _, Xa = analyse(mask, m, X, y)
    got = Xa.astype(np.float64).mean(-1)
    step = rmean - X.astype(np.float64).mean(-1)
    assert np.linalg.norm(got - rmean) <= 6 * kappa ** 0.5 * UNIT * np.linalg.norm(step) \
        + 2 * UNIT * np.linalg.norm(rmean)


@pytest.mark.parametrize("nsub,m", [(9, 192), (10, 128), (16, 320), (8, 480), (16, 70)])
def test_a_mean_that_did_not_converge_is_reported(nsub, m):
    """Conditions from 6e6 past the end of FP32's range, where the corrections of the mean stop
    converging before the root's own check fails: an error status, or a mean as accurate as
    the slopes' rounding, amplified by sqrt(kappa), allows (16 units)."""
    refused = 0
    for scale in (60.0, 95.0, 130.0, 151.0, 176.0, 205.0, 240.0, 325.0):
        mask, dg, mean, P, y, G = problem(nsub, m, seed=int(scale))
        alpha = (m - 1) / RHO
        X = (mean + scale * P).astype(np.float32)
        _, rmean, _ = LD.analysis_domains(dg, X.astype(np.float64), y.astype(np.float64), SIGMA2, RHO)
        kappa = np.linalg.norm(alpha * np.eye(m) + scale ** 2 * G) / alpha
        try:
            got = analyse(mask, m, X, y)[2].astype(np.float64).mean(-1)
        except LetkfError as e:
            assert "NOCONVERGE" in str(e) or "NONFINITE" in str(e)
            refused += 1
            continue
        step = rmean - X.astype(np.float64).mean(-1)
        assert np.linalg.norm(got - rmean) <= 16 * kappa ** 0.5 * UNIT * np.linalg.norm(step), scale
        assert scale != 60.0 or kappa > 5e6
    assert refused < 8                                   # not every one: the smallest is solved


@pytest.mark.parametrize("value", [float("inf"), -float("inf"), float("nan")])
@pytest.mark.parametrize("m", [48, 80])
def test_a_nonfinite_ensemble_is_reported_by_both_forms(m, value):
    """A member's infinite phase makes infinite slopes, whose exponent is no number to add to:
    the Gram's anchor is infinite then, and the analysis NaN and reported."""
    mask, dg, mean, P, y, _ = problem(6, m)
    X = (mean + 0.06 * P).astype(np.float32)
    X[20, 1, 5] = value
    with pytest.raises(LetkfError, match="NONFINITE"):
        analyse(mask, m, X, y)
