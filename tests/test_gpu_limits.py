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
