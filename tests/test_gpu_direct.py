"""The Chebyshev form of the per-node analysis (letkf_pair.cu: direct_apply) at the
sizes and spectra where it can go wrong, against the FP64 oracle and against the
eigensolve (a handle with an explicit sweep limit).

Tolerance of the ensemble, for the root mean square of its error over the nodes: A^-1/2
changes by at most kappa / 2 times the relative change of A, whose FP32 rounding is a
few units (the Gram's sums), and the series' own rounding is of the order of its degree,
about 10 sqrt(kappa) units: 32 kappa units of 2^-24 of the anomalies' size cover both.
The mean moves by X' A^-1 C d, kappa units of the increment's size. Storing the members
(background and analysis) in FP32 adds two units of their own size."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_1408_7069_gb300 import synth  # noqa: E402
from paper_1408_7069_gb300.letkf import Letkf, tile_shapes  # noqa: E402

pytestmark = pytest.mark.gpu

SIGMA2, RHO = 0.01, 1.03


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(b))


def anoms(X):
    X = np.asarray(X, np.float64)
    return X - X.mean(-1, keepdims=True)


def problem(nsub, m, window, taper, scale, square=False, ramp=None):
    """An ensemble of white member anomalies of size `scale` (times a factor growing from
    ramp[0] to ramp[1] along the grid), slopes, geometry and the nodes' kappa_hat."""
    mask = synth.pupil_subap_mask(nsub, 0.0, square)
    geom = oracle.build_geometry(mask, window, taper, 0.0)
    rng = np.random.default_rng(1000 * nsub + 10 * m + window)
    s = np.full(geom.n_pts, scale)
    if ramp:
        s = scale * np.geomspace(ramp[0], ramp[1], geom.n_pts)
    X = 3 * rng.standard_normal((geom.n_pts, 2, 1)) \
        + s[:, None, None] * rng.standard_normal((geom.n_pts, 2, m))
    X = X.astype(np.float32)
    y = rng.standard_normal(geom.p).astype(np.float32)
    _, _, Yb, _ = oracle.observe(geom, X.astype(np.float64))
    khat = np.array([1 + RHO / (m - 1) * np.sum((t / SIGMA2)[:, None] * Yb[i] ** 2)
                     for i, t in zip(geom.win_idx, geom.win_tau)])
    return mask, geom, X, y, khat


def analyse(mask, X, y, m, window, taper, shape=None, cls=None, **kw):
    f = Letkf(mask, m=m, window=window, taper=taper, rho=RHO, sigma2=SIGMA2, **kw)
    if shape is not None:
        f.set_tile_shape(cls, shape)
    f.set_state(torch.from_numpy(X).cuda())
    mean, spread = f.analyze(torch.from_numpy(y).cuda())
    f.sync()
    out = f.get_state().cpu().numpy(), mean.cpu().numpy(), spread.cpu().numpy(), f.stats()
    f.close()
    return out


SIZES = [(1, 2, 1, 0), (4, 3, 3, 1), (5, 15, 3, 1), (5, 16, 4, 0), (6, 17, 5, 1), (6, 23, 5, 1),
         (6, 24, 5, 0), (7, 25, 7, 1), (7, 31, 6, 1), (9, 32, 7, 1), (5, 33, 3, 1), (6, 47, 5, 1),
         (6, 48, 5, 1), (6, 49, 5, 0), (6, 63, 7, 1), (7, 64, 7, 1)]


@pytest.mark.parametrize("scale", [1e-3, 0.06, 0.4], ids=["tiny", "loop", "wide"])
@pytest.mark.parametrize("nsub,m,window,taper", SIZES)
def test_series_matches_oracle_and_eigensolve(nsub, m, window, taper, scale):
    mask, geom, X, y, khat = problem(nsub, m, window, taper, scale)
    ref = oracle.analysis(geom, X.astype(np.float64), y.astype(np.float64), SIGMA2, RHO)
    Xa, mean, spread, st = analyse(mask, X, y, m, window, taper)
    if khat.max() < 299:
        assert st == (0, 1, geom.n_pts)             # every node by the series
    assert rel(mean, ref[1]) <= 1e-4 and rel(spread, ref[2]) <= 1e-3
    if khat.max() < 299:
        def rms(v):
            return float(np.sqrt(np.mean(np.square(v))))
        Xb = X.astype(np.float64)
        step = ref[1] - Xb.mean(-1)
        unit = 2.0 ** -24
        assert rms(Xa - ref[0]) <= 32 * unit * khat.max() * (rms(anoms(Xb)) + rms(step)) \
            + 2 * unit * rms(Xb)
    Xj, mj, sj, st = analyse(mask, X, y, m, window, taper, max_sweeps=20)
    assert st[2] > geom.n_pts or m == 2 or scale == 1e-3
    assert rel(mean, mj) <= 1e-4 and rel(spread, sj) <= 1e-3


@pytest.mark.parametrize("kappa", [0.0, 300.0, 3.0], ids=["no-fp64", "default", "low"])
@pytest.mark.parametrize("m,cls", [(12, 0), (24, 1), (32, 1), (40, 2)])
def test_nodes_of_both_kinds_share_warps(m, cls, kappa):
    """kappa_hat from about 1 to 1e4 along the grid: nodes of the series, of the Jacobi
    sweeps (fp64_kappa = 0) and of the FP64 queue in one warp, each with its own degree;
    the outputs meet the FP32 tolerances and do not depend on the tile shape."""
    mask, geom, X, y, khat = problem(10, m, 5, 1, 0.3, ramp=(0.02, 10.0))
    assert khat.min() < 2 and khat.max() > 1500
    ref = oracle.analysis(geom, X.astype(np.float64), y.astype(np.float64), SIGMA2, RHO)
    Xa, mean, spread, st = analyse(mask, X, y, m, 5, 1, fp64_kappa=kappa)
    if kappa > 0:
        assert abs(st[0] - int((khat > kappa).sum())) <= 2
    assert rel(spread, ref[2]) <= 1e-3
    # without FP64 the mean of the ill-conditioned nodes is not held to 1e-4
    assert rel(mean, ref[1]) <= (1e-4 if kappa > 0 else 1e-2)
    assert rel(anoms(Xa), anoms(ref[0])) <= 1e-3
    for shape, (a, b) in enumerate(tile_shapes()):
        if (a * b) % (4 if cls == 0 else 2 if cls == 1 else 1) or (cls == 2 and a * b > 8):
            continue
        Xs, *_ = analyse(mask, X, y, m, 5, 1, shape=shape, cls=cls, fp64_kappa=kappa)
        assert np.array_equal(Xs, Xa), shape


def test_nonfinite_node_problem_takes_the_eigensolve_and_is_reported():
    from paper_1408_7069_gb300.letkf import LetkfError
    mask, geom, X, y, _ = problem(6, 24, 5, 1, 0.06)
    X[10, 1, 3] = np.inf
    with pytest.raises(LetkfError, match="LETKF_ERR_NONFINITE"):
        analyse(mask, X, y, 24, 5, 1)


# ---------------------------------------------------------------------------
# FP64 handles (letkf_series64.cu): the FP64 tolerances of the analysis tests, 1e-9 on
# the mean and 1e-8 on the spread and the anomalies; gradients as in the reverse mode's
# tests, 1e-8.
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("scale", [1e-3, 0.06, 0.3], ids=["tiny", "loop", "wide"])
@pytest.mark.parametrize("nsub,m,window,taper",
                         [(1, 2, 1, 0), (4, 7, 3, 1), (4, 8, 3, 1), (4, 9, 4, 0), (5, 16, 5, 1),
                          (5, 17, 3, 1), (6, 24, 9, 1), (6, 25, 5, 0), (5, 32, 7, 1)])
def test_fp64_series_matches_oracle(nsub, m, window, taper, scale):
    mask, geom, X, y, khat = problem(nsub, m, window, taper, scale)
    X, y = X.astype(np.float64), y.astype(np.float64)
    ref = oracle.analysis(geom, X, y, SIGMA2, RHO)
    Xa, mean, spread, st = analyse(mask, X, y, m, window, taper, precision=1)
    if khat.max() < 42:
        assert st[1:] == (1, geom.n_pts)
    assert rel(mean, ref[1]) <= 1e-9 and rel(spread, ref[2]) <= 1e-8
    assert rel(anoms(Xa), anoms(ref[0])) <= 1e-8


@pytest.mark.parametrize("m", [7, 24])
def test_fp64_series_keeps_the_range_of_fp64(m):
    """The node's values are scaled by powers of two before anything is rounded: an
    analysis in other units, by 2^+-200, has the same digits. And rows and innovations
    of nothing but zeros."""
    mask, geom, X, y, _ = problem(4, m, 3, 1, 0.06)
    X, y = X.astype(np.float64), y.astype(np.float64)

    def run(X, y, s):
        f = Letkf(mask, m=m, window=3, taper=1, rho=RHO, sigma2=SIGMA2 * s * s, precision=1)
        f.set_state(torch.from_numpy(X * s).cuda())
        mean, spread = f.analyze(torch.from_numpy(y * s).cuda())
        out = f.get_state().cpu().numpy(), mean.cpu().numpy(), spread.cpu().numpy()
        f.sync()
        assert f.stats()[1] == 1
        f.close()
        return [v / s for v in out]
    a = run(X, y, 1.0)
    for s in (2.0 ** 200, 2.0 ** -200):
        assert all(np.array_equal(u, v) for u, v in zip(a, run(X, y, s)))
    flat = np.repeat(X.mean(-1, keepdims=True), m, -1)
    Xz = X.copy()
    Xz[:, 1] = flat[:, 1]                        # no anomalies in the second row
    for Xb, yb in ((Xz, y), (flat, y), (X, np.zeros_like(y)), (flat, np.zeros_like(y))):
        ref = oracle.analysis(geom, Xb, yb, SIGMA2, RHO)
        got = run(Xb, yb, 1.0)
        for u, v in zip(got, ref):
            assert np.abs(u - v).max() <= 1e-9 * np.abs(X).max()


def test_fp64_series_and_eigensolve_nodes_in_one_frame():
    mask, geom, X, y, khat = problem(8, 20, 5, 1, 0.3, ramp=(0.02, 10.0))
    X, y = X.astype(np.float64), y.astype(np.float64)
    assert khat.min() < 2 and khat.max() > 1000
    ref = oracle.analysis(geom, X, y, SIGMA2, RHO)
    Xa, mean, spread, st = analyse(mask, X, y, 20, 5, 1, precision=1)
    assert 1 < st[1] <= 20
    assert rel(mean, ref[1]) <= 1e-9 and rel(spread, ref[2]) <= 1e-8
    assert rel(anoms(Xa), anoms(ref[0])) <= 1e-8


@pytest.mark.parametrize("nsub,m,window,taper,scale",
                         [(3, 6, 3, 1, 0.06), (4, 12, 3, 1, 0.06), (4, 20, 5, 1, 0.1),
                          (5, 24, 9, 0, 0.08), (4, 32, 7, 1, 0.1), (4, 24, 5, 0, 0.12)])
def test_fp64_series_adjoint_matches_oracle(nsub, m, window, taper, scale):
    """Gradients through the series: every column width, more slopes than one staged
    chunk, degrees below and above what the kernel keeps of the terms."""
    mask, geom, X, y0, khat = problem(nsub, m, window, taper, scale, square=True)
    assert khat.max() < 60
    frames, rng = 3, np.random.default_rng(nsub + m)
    geom = oracle.build_geometry(mask, window, taper, window / 4.0)
    X = X.astype(np.float64)
    y = 0.3 * rng.standard_normal((frames, geom.p))
    truth = rng.standard_normal((frames, geom.n_pts))
    bank = rng.standard_normal((2, 16, 16)).astype(np.float32)
    J, g, _ = oracle.closed_loop_grad(geom, truth, y, bank, m, SIGMA2, RHO, 0.999, scale, 9,
                                      frames, X)
    f = Letkf(mask, m=m, window=window, taper=taper, rho=RHO, sigma2=SIGMA2, a_ar1=0.999,
              noise_std=scale, precision=1, seed=9, bank=bank)
    f.set_state(torch.from_numpy(X).cuda())
    Jg, gg = f.grad(frames, torch.from_numpy(y).cuda(), torch.from_numpy(truth).cuda(), 2)
    Xg = f.get_state()
    f.set_state(torch.from_numpy(X).cuda())
    f.set_frame(0)
    f.run(frames, torch.from_numpy(y).cuda())
    f.sync()
    assert torch.equal(Xg, f.get_state())               # the state letkf_run leaves
    f.close()
    assert Jg == pytest.approx(J, rel=1e-10)
    assert np.all(np.abs(gg - g) <= 1e-8 * np.maximum(np.abs(g), 1e-6 * np.abs(g).max())), (gg, g)


# ---------------------------------------------------------------------------
# Multi-actuator domains (domain_series_kernel)
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("scale", [0.02, 0.08], ids=["small", "loop"])
@pytest.mark.parametrize("nsub,m,window,parts,piston",
                         [(8, 2, 3, 3, 1), (9, 16, 3, 3, 1), (9, 17, 3, 4, 0), (12, 32, 5, 3, 1),
                          (12, 33, 3, 2, 1), (14, 64, 5, 4, 0), (14, 65, 3, 2, 1),
                          (16, 101, 5, 4, 1), (20, 104, 5, 7, 1), (12, 105, 3, 3, 1),
                          (12, 128, 5, 3, 1)])
def test_domain_series_matches_oracle(nsub, m, window, parts, piston, scale):
    """Every column width, one to four CTAs per domain, domains of more than one pass of
    63 rows; the FP32 tolerances of the domain tests, and the anomalies to the series'
    own bound (see the module docstring; the domains' kappa_hat in place of the nodes')."""
    from oracle import letkf_domains as LD
    mask = synth.pupil_subap_mask(nsub, 0.0)
    dg = LD.build_domains(mask, parts, window, 1, 0.0)
    rng = np.random.default_rng(100 * nsub + m)
    n = dg.geom.n_pts
    X = (3 * rng.standard_normal((n, 2, 1)) + scale * rng.standard_normal((n, 2, m)))
    X = X.astype(np.float32)
    y = rng.standard_normal(dg.geom.p).astype(np.float32)
    Xb = X.astype(np.float64)
    rXa, rmean, rspread, parts_, _ = LD.analysis_domains(dg, Xb, y.astype(np.float64), SIGMA2, RHO,
                                                         piston=bool(piston), return_parts=True)
    khat = max(np.trace(A) / ((m - 1) / RHO) - m + 1 for A, _, _ in parts_)
    ratio = max(np.linalg.norm(A - (m - 1) / RHO * np.eye(m)) / ((m - 1) / RHO)
                for A, _, _ in parts_)
    f = Letkf(mask, m=m, window=window, taper=1, rho=RHO, sigma2=SIGMA2, partition=parts,
              piston=piston)
    f.set_state(torch.from_numpy(X).cuda())
    mean, spread = f.analyze(torch.from_numpy(y).cuda())
    f.sync()
    st = f.stats()
    Xa = f.get_state().cpu().numpy()
    f.close()
    if ratio < 99:
        assert st[1:] == (1, dg.n_dom)
    mean, spread = mean.cpu().numpy(), spread.cpu().numpy()
    assert rel(mean, rmean) <= 1e-4 and rel(spread, rspread) <= 1e-3
    step = rmean - Xb.mean(-1)
    unit, rms = 2.0 ** -24, lambda v: float(np.sqrt(np.mean(np.square(v))))
    if ratio < 99:
        assert rms(Xa - rXa) <= 32 * unit * khat * (rms(anoms(Xb)) + rms(step)) \
            + 2 * unit * rms(Xb)


def test_domains_of_both_kinds_in_one_frame():
    """Anomalies growing along the grid: well-conditioned domains by the series, the
    others by the sweeps, in one frame; every domain counted once."""
    from oracle import letkf_domains as LD
    nsub, m, window, parts = 16, 48, 5, 5
    mask = synth.pupil_subap_mask(nsub, 0.0)
    dg = LD.build_domains(mask, parts, window, 1, 0.0)
    n = dg.geom.n_pts
    rng = np.random.default_rng(77)
    s = 0.05 * np.geomspace(0.2, 100.0, n)
    X = (3 * rng.standard_normal((n, 2, 1))
         + s[:, None, None] * rng.standard_normal((n, 2, m))).astype(np.float32)
    y = rng.standard_normal(dg.geom.p).astype(np.float32)
    rXa, rmean, rspread = LD.analysis_domains(dg, X.astype(np.float64), y.astype(np.float64),
                                              SIGMA2, RHO, piston=False)
    f = Letkf(mask, m=m, window=window, taper=1, rho=RHO, sigma2=SIGMA2, partition=parts)
    f.set_state(torch.from_numpy(X).cuda())
    mean, spread = f.analyze(torch.from_numpy(y).cuda())
    f.sync()
    st = f.stats()
    Xa = f.get_state().cpu().numpy()
    f.close()
    assert 1 < st[1] <= 20 and st[2] > dg.n_dom and 0 < st[0] < dg.n_dom
    assert rel(spread.cpu().numpy(), rspread) <= 1e-3
    assert rel(anoms(Xa), anoms(rXa)) <= 1e-3


# ---------------------------------------------------------------------------
# Global ETKF of more than 64 members (ns_root_kernel, global_gram_kernel)
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("scale", [0.05, 3.0], ids=["loop", "ill"])
@pytest.mark.parametrize("nsub,m", [(3, 65), (10, 128), (12, 129), (9, 192), (16, 320), (12, 1000)])
def test_global_root_matches_oracle(nsub, m, scale):
    """Padding edges, fewer and more slopes than members, kappa from about 2 to 1e5, two
    analyses in a row (the grid barrier's counters): the tolerances of the global tests."""
    from oracle import letkf_domains as LD
    mask = synth.pupil_subap_mask(nsub, 0.0)
    dg = LD.build_domains(mask, 1, 3, 0, 0.0)
    rng = np.random.default_rng(nsub + m)
    n = dg.geom.n_pts
    X = (3 * rng.standard_normal((n, 2, 1)) + scale * rng.standard_normal((n, 2, m)))
    X = X.astype(np.float32)
    f = Letkf(mask, m=m, window=3, taper=0, rho=RHO, sigma2=SIGMA2, partition=1)
    f.set_state(torch.from_numpy(X).cuda())
    for _ in range(2):
        Xb = f.get_state().cpu().numpy().astype(np.float64)
        y = rng.standard_normal(dg.geom.p).astype(np.float32)
        rXa, rmean, rspread = LD.analysis_domains(dg, Xb, y.astype(np.float64), SIGMA2, RHO)
        mean, spread = f.analyze(torch.from_numpy(y).cuda())
        f.sync()
        Xa = f.get_state().cpu().numpy()
        assert rel(mean.cpu().numpy(), rmean) <= 1e-4
        assert rel(spread.cpu().numpy(), rspread) <= 1e-3
        assert rel(anoms(Xa), anoms(rXa)) <= 1e-3
    f.close()


def test_global_root_in_graphs_and_nonfinite_slopes():
    from paper_1408_7069_gb300.letkf import LetkfError
    mask = synth.pupil_subap_mask(8, 0.0)
    rng = np.random.default_rng(5)
    m, frames = 80, 3
    bank = rng.standard_normal((2, 32, 32)).astype(np.float32)
    f = Letkf(mask, m=m, window=3, taper=0, rho=RHO, sigma2=SIGMA2, partition=1, a_ar1=0.999,
              noise_std=0.05, seed=3, bank=bank)
    X = torch.from_numpy(rng.standard_normal((f.n_pts, 2, m)).astype(np.float32) * 0.1).cuda()
    y = torch.from_numpy(rng.standard_normal((frames, f.p)).astype(np.float32)).cuda()
    out = []
    for mode in ("plain", "graph", "one"):
        f.set_state(X)
        f.set_frame(0)
        if mode == "one":
            f.run_graph(frames, y)
        else:
            f.run(frames, y, use_graph=mode == "graph")
        f.sync()
        out.append(f.get_state().cpu().numpy())
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])
    bad = y[0].clone()
    bad[7] = float("nan")
    f.analyze(bad)
    with pytest.raises(LetkfError, match="LETKF_ERR_NONFINITE"):
        f.sync()
    f.set_state(X)
    f.set_frame(0)
    f.run(frames, y)
    f.sync()
    assert np.array_equal(f.get_state().cpu().numpy(), out[0])
    f.close()


# ---------------------------------------------------------------------------
# Ill-conditioned node problems of FP32 handles (letkf_tri.cuh)
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("scale", [2.0, 12.0, 60.0], ids=["3e2", "1e4", "3e5"])
@pytest.mark.parametrize("nsub,m,window,taper",
                         [(3, 2, 3, 1), (4, 3, 3, 1), (5, 15, 3, 1), (5, 16, 5, 0), (6, 17, 5, 1),
                          (6, 24, 9, 0), (6, 25, 5, 1), (6, 31, 4, 1), (7, 32, 7, 1),
                          (12, 32, 13, 0)])
def test_ill_conditioned_nodes_match_oracle(nsub, m, window, taper, scale):
    """Every queued node by the float-pair tridiagonal form, or by the FP64 sweeps beyond its
    range: more slopes than one staged chunk, windows with fewer slopes than members, both
    column widths. kappa_hat above 1 sends every node there. Tolerances: the FP32 ones on
    the mean; the storage's rounding, 4 units of 2^-24 of the background's size, plus 1e-6
    of the analysis anomalies (kappa to 1e5 times 2^-42 and the poles' 4e-9) on the members."""
    mask, geom, X, y, khat = problem(nsub, m, window, taper, scale)
    ref = oracle.analysis(geom, X.astype(np.float64), y.astype(np.float64), SIGMA2, RHO)
    Xa, mean, spread, st = analyse(mask, X, y, m, window, taper, fp64_kappa=1.0000001)
    assert st[0] == geom.n_pts
    if khat.max() < 9.9e4:
        assert st[1:] == (1, geom.n_pts)

    def rms(v):
        return float(np.sqrt(np.mean(np.square(v))))
    if khat.max() < 9.9e4:
        assert rel(mean, ref[1]) <= 1e-4
        assert rel(spread, ref[2]) <= 1e-3
        assert rel(anoms(Xa), anoms(ref[0])) <= 1e-3
    Xj, mj, sj, _ = analyse(mask, X, y, m, window, taper, fp64_kappa=1.0000001, max_sweeps=30)
    assert rms(Xa - Xj) <= 4 * 2.0 ** -24 * rms(X) + 1e-6 * rms(anoms(ref[0]))


# ---------------------------------------------------------------------------
# The forecast inside the analysis (lk_launch_cycle): letkf_run against the same frames
# by letkf_analyze and letkf_forecast, whose kernels are separate. The same bits.
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("use_graph", [True, False], ids=["graph", "stream"])
@pytest.mark.parametrize("m,precision,scale,kw",
                         [(10, 0, 0.1, {}), (20, 0, 0.1, {}), (32, 0, 3.0, {}),
                          (17, 0, 30.0, {}), (20, 0, 3.0, dict(max_sweeps=20)), (40, 0, 3.0, {}),
                          (64, 0, 0.1, {}), (24, 0, 0.1, dict(fp64_kappa=-1.0)),
                          (10, 1, 0.1, {}), (24, 1, 3.0, {})])
def test_run_equals_analyses_and_forecasts(m, precision, scale, kw, use_graph):
    mask, geom, X, y, _ = problem(6, m, 3, 1, scale)
    dt = np.float64 if precision else np.float32
    frames, rng = 3, np.random.default_rng(m)
    ys = torch.from_numpy(rng.standard_normal((frames, geom.p)).astype(dt)).cuda()
    bank = rng.standard_normal((2, 16, 16)).astype(np.float32)
    f = Letkf(mask, m=m, window=3, taper=1, rho=RHO, sigma2=SIGMA2, a_ar1=0.99, noise_std=0.1,
              precision=precision, seed=3, bank=bank, **kw)
    X = torch.from_numpy(X.astype(dt)).cuda()
    f.set_state(X)
    f.run(frames, ys, use_graph=use_graph)
    f.sync()
    a = f.get_state()
    f.set_state(X)
    f.set_frame(0)
    for k in range(frames):
        f.analyze(ys[k], outputs=False)
        f.forecast()
    f.sync()
    assert torch.equal(a, f.get_state())
    f.close()


def test_calls_are_ordered_against_the_current_stream():
    """Inputs still being written on one torch stream, outputs read on another, from two
    threads in turn: the events that order the handle's stream are kept between calls."""
    import threading
    mask, geom, X, _, _ = problem(6, 8, 3, 1, 0.1)
    f = Letkf(mask, m=8, window=3, taper=1, rho=RHO, sigma2=SIGMA2)
    X = torch.from_numpy(X).cuda()
    big = torch.randn(4096, 4096, device="cuda")
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()

    def turn(k):
        with torch.cuda.stream(a):
            z = big
            for _ in range(4):
                z = z @ big * 1e-2
            f.set_state(X * k + 0 * z[0, 0].nan_to_num(0.0, 0.0, 0.0))
        with torch.cuda.stream(b):
            out.append((k, f.get_state()))
    out = []
    for k in range(1, 5):
        t = threading.Thread(target=turn, args=(float(k),))
        if k % 2:
            t.start()
            t.join()
        else:
            turn(float(k))
    torch.cuda.synchronize()
    assert len(out) == 4 and all(torch.equal(v, X * k) for k, v in out)
    f.close()


# ---------------------------------------------------------------------------
# Two members (the closed form beside direct_apply). Tolerance: the members' storage and
# the means that the innovations take (two units of 2^-24 of the members), and the roundings
# of slopes, Gram, trace, root and products, eight units of the anomalies and increments:
# no factor of the condition, since the trace's relative error is that of A.
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("ratio", [3.0, 20.0, 80.0, 290.0])
@pytest.mark.parametrize("window,taper", [(3, 0), (5, 1)])
def test_two_members_to_the_rounding_of_fp32(window, taper, ratio):
    mask = synth.pupil_subap_mask(8, 0.0)
    geom = oracle.build_geometry(mask, window, taper, 0.0)

    def rms(v):
        return float(np.sqrt(np.mean(np.square(v))))
    for seed in range(6):
        rng = np.random.default_rng(seed)
        P = anoms(rng.standard_normal((geom.n_pts, 2, 2)))
        _, _, Yb, _ = oracle.observe(geom, P)
        g = [RHO * np.linalg.norm((Yb[i] * (t / SIGMA2)[:, None]).T @ Yb[i])
             for i, t in zip(geom.win_idx, geom.win_tau)]
        X = 3 * rng.standard_normal((geom.n_pts, 2, 1)) + (ratio / np.max(g)) ** 0.5 * P
        X = X.astype(np.float32)
        y = rng.standard_normal(geom.p).astype(np.float32)
        ref = oracle.analysis(geom, X.astype(np.float64), y.astype(np.float64), SIGMA2, RHO)
        Xa, mean, spread, st = analyse(mask, X, y, 2, window, taper, fp64_kappa=-1.0)
        assert st[1:] == (1, geom.n_pts)
        step = ref[1] - X.astype(np.float64).mean(-1)
        tol = 2.0 ** -24 * (2 * rms(X) + 8 * (rms(anoms(X)) + rms(step)))
        assert rms(Xa - ref[0]) <= tol and rms(mean - ref[1]) <= tol and rms(spread - ref[2]) <= tol
