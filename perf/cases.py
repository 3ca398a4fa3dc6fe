"""The workloads the framework's speed is measured on, each through its public entry points.

A case is one use of a ``Letkf`` handle: single analyses (``analyze``), closed loops
(``run``), the real-time call from host memory (``step``), the loop with a deformable
mirror, batches of many systems, multi-actuator domains with differential pistons, the
global ETKF and the reverse mode (``grad``). ``state`` says what the ensemble looks like
when the call comes:

* ``loop``: the statistics of a running loop. Measured on the FP64 oracle's loops of the
  8x8, 16 m and 80x80 systems: slope anomalies of about 0.65 sigma, smooth member
  anomalies, forecast noise of q times a von Karman screen.
* ``prior``: the first frame, members drawn from the turbulence's stationary law (slope
  anomalies of tens of sigma, so the node problems are ill conditioned).

Sizes come from ``workloads.py``, the tests and ``bench.py``; ``draw`` covers the ranges
between and around them. ``exact`` computes the same results in plain FP64 torch.
"""
import math
import random

import numpy as np
import torch

from paper_1408_7069_gb300.letkf import Letkf
from paper_1408_7069_gb300.workloads import Workload

SIGMA = 0.1           # slope noise (rad)
LOOP_SLOPE = 0.065    # standard deviation of a running loop's slope anomalies (rad)
PITCH, R0, L0 = 0.5, 0.15, 25.0
BANK = 16


def _case(kind, nsub, m, window, **kw):
    c = dict(kind=kind, nsub=nsub, m=m, window=window, obscuration=0.14, square=False, taper=1,
             rho=1.03, q=0.006, precision=0, frames=1, partition=0, piston=False, state="loop",
             ckpt=0, count=1)
    c.update(kw)
    return c


def listed():
    def named(name, *a, **kw):
        return dict(_case(*a, **kw), name=name)

    return [
        # the smallest system, FP64: a bench-top loop of 16 frames in one call
        named("toy-8x8-fp64-loop", "run", 8, 10, 3, obscuration=0.0, square=True, rho=1.05,
              q=0.003, precision=1, frames=16),
        # a 16 m telescope's real-time controller: four frames, each from host memory and back
        named("16m-step", "step", 32, 24, 5, frames=4),
        # the same telescope's loop fed from device memory (simulation, replay)
        named("16m-loop", "run", 32, 24, 5, frames=4),
        # the same with its deformable mirror: pseudo-open-loop slopes in, commands out
        named("16m-dm-loop", "dm", 32, 24, 5, frames=4),
        # ELT scale, the headline system: the running loop
        named("elt-loop", "run", 80, 32, 7, rho=1.02, q=0.005, frames=4),
        # ... and its first frame, when the loop is closed on the prior draw
        named("elt-first-frame", "analyze", 80, 32, 7, rho=1.02, q=0.005, state="prior"),
        # 48 systems of 16..96 subapertures and 16..48 members, one handle (survey, tuning)
        named("batch-48-loop", "run", 96, 48, 7, rho=1.02, q=0.005, frames=2, count=48),
        # the paper's multi-actuator domains with differential pistons, 16 m and 40 m
        named("16m-domains", "analyze", 32, 101, 5, obscuration=0.0, rho=1.02, partition=9,
              piston=True),
        named("40m-domains", "analyze", 80, 101, 5, obscuration=0.0, rho=1.02, q=0.005,
              partition=21, piston=True),
        # the global ETKF of the 16 m pupil: the running loop, and the first frame of the
        # paper's largest ensemble
        named("16m-global-m101", "analyze", 32, 101, 5, obscuration=0.0, rho=1.02, taper=0,
              partition=1),
        named("16m-global-m626-first", "analyze", 32, 626, 5, obscuration=0.0, rho=1.02, taper=0,
              partition=1, state="prior"),
        # tuning: gradient of the loop criterion in rho, sigma^2 and L, FP64, 16 m
        named("16m-grad-fp64", "grad", 32, 24, 5, precision=1, frames=10, ckpt=5),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    win, taper = rng.choice([3, 4, 5, 6, 7, 9]), rng.choice([0, 1, 1, 1])
    common = dict(obscuration=rng.choice([0.0, 0.14, 0.3]), square=rng.random() < 0.2,
                  rho=round(rng.uniform(1.0, 1.08), 3), q=round(rng.uniform(0.003, 0.008), 4))
    kind = rng.choice(["run", "run", "run64", "step", "dm", "analyze", "first", "batch",
                       "domains", "global", "grad"])
    if kind == "run":
        return _case("run", logint(6, 96), rng.randint(4, 64), win, taper=taper,
                     frames=rng.randint(1, 4), **common)
    if kind == "run64":
        return _case("run", logint(4, 32), rng.randint(4, 32), win, taper=taper, precision=1,
                     frames=rng.randint(1, 8), **common)
    if kind == "step":
        return _case("step", logint(6, 80), rng.randint(6, 48), win, frames=rng.randint(1, 4),
                     **common)
    if kind == "dm":
        return _case("dm", logint(6, 32), rng.randint(6, 48), rng.choice([3, 5, 7]),
                     frames=rng.randint(1, 4), **common)
    if kind == "analyze":
        return _case("analyze", logint(6, 96), rng.randint(2, 64), win, taper=taper, **common)
    if kind == "first":
        return _case("analyze", logint(8, 56), rng.randint(8, 64), rng.choice([3, 5, 7]),
                     state="prior", **common)
    if kind == "batch":
        return _case("run", rng.randint(24, 64), rng.choice([32, 48]), rng.choice([5, 7]),
                     frames=rng.randint(1, 2), count=rng.randint(2, 16), **common)
    if kind == "domains":
        nsub = logint(16, 80)
        return _case("analyze", nsub, rng.randint(24, 128), rng.choice([3, 5]),
                     partition=-(-(nsub + 1) // rng.choice([3, 4])), piston=rng.random() < 0.7,
                     **common)
    if kind == "global":
        return _case("analyze", logint(8, 40), logint(24, 640), 5, taper=0, partition=1,
                     state=rng.choice(["loop", "prior"]), **common)
    return _case("grad", logint(6, 24), rng.randint(6, 32), rng.choice([3, 5]), precision=1,
                 frames=rng.randint(2, 10), ckpt=rng.choice([0, 3, 5]), **common)


# ---------------------------------------------------------------------------
# Geometry (Fried grid, pupil, windows, domains)
# ---------------------------------------------------------------------------
def _pupil(nsub, obscuration, square):
    if square:
        return np.ones((nsub, nsub), bool)
    x = (np.arange(nsub * 16) + 0.5) / 16 - nsub / 2.0
    r = np.sqrt(x[:, None] ** 2 + x[None, :] ** 2)
    lit = (r <= nsub / 2.0) & (r >= obscuration * (nsub / 2.0))
    return lit.reshape(nsub, 16, nsub, 16).mean(axis=(1, 3)) > 0.5


class _Geometry:
    """Nodes, slopes and update groups (one node, one domain, or the whole pupil each) as
    index arrays: ``rows`` [G, R] nodes (padded with n), ``obs`` [G, L] subapertures (padded
    with the number of subapertures), ``dist`` [G, L] distance for the taper (pitches)."""

    def __init__(self, nsub, window, obscuration, square, partition):
        sm = _pupil(nsub, obscuration, square)
        nn = nsub + 1
        nodes = np.zeros((nn, nn), bool)
        for di in (0, 1):
            for dj in (0, 1):
                nodes[di:nsub + di, dj:nsub + dj] |= sm
        self.mask, self.nsub = sm.astype(np.uint8), nsub
        self.pts, saps = np.argwhere(nodes), np.argwhere(sm)
        self.n, self.ns = len(self.pts), len(saps)
        pid = -np.ones((nn, nn), np.int64)
        pid[nodes] = np.arange(self.n)
        s, t = saps[:, 0], saps[:, 1]
        self.corner = np.stack([pid[s, t], pid[s + 1, t], pid[s, t + 1], pid[s + 1, t + 1]])
        h = window // 2
        sid = np.full((nsub + 2 * window, nsub + 2 * window), self.ns, np.int64)
        sid[window:window + nsub, window:window + nsub][sm] = np.arange(self.ns)
        off = np.arange(window)
        self.edges = None
        if partition == 0:
            i, j = self.pts[:, 0], self.pts[:, 1]
            grid = (i[:, None, None] - h + window + off[:, None],
                    j[:, None, None] - h + window + off[None, :])
            self.rows = np.arange(self.n)[:, None]
            self.obs = sid[grid].reshape(self.n, -1)
            d = np.hypot(*np.meshgrid(off - h + 0.5, off - h + 0.5, indexing="ij")).reshape(-1)
            self.dist = np.broadcast_to(d, self.obs.shape)
            return
        bb = [(b * nn) // partition for b in range(partition + 1)]
        blk = np.searchsorted(bb, np.arange(nn), side="right") - 1
        key = blk[self.pts[:, 0]] * partition + blk[self.pts[:, 1]]
        _, self.dom = np.unique(key, return_inverse=True)
        rows, obs, dist = [], [], []
        for d in range(self.dom.max() + 1):
            ids = np.flatnonzero(self.dom == d)
            p = self.pts[ids]
            cells = np.unique((p[:, 0][:, None, None] - h + window + off[:, None]) * sid.shape[1]
                              + p[:, 1][:, None, None] - h + window + off[None, :])
            o = sid.reshape(-1)[cells]
            cells, o = cells[o < self.ns], o[o < self.ns]
            cs, ct = cells // sid.shape[1] - window + 0.5, cells % sid.shape[1] - window + 0.5
            dx = np.maximum(np.maximum(p[:, 0].min() - cs, cs - p[:, 0].max()), 0.0)
            dy = np.maximum(np.maximum(p[:, 1].min() - ct, ct - p[:, 1].max()), 0.0)
            rows.append(ids)
            obs.append(o)
            dist.append(np.hypot(dx, dy))

        def pad(v, fill):
            out = np.full((len(v), max(map(len, v))), fill, np.asarray(v[0]).dtype)
            for k, x in enumerate(v):
                out[k, :len(x)] = x
            return out

        self.rows, self.obs, self.dist = pad(rows, self.n), pad(obs, self.ns), pad(dist, 0.0)
        e = []
        for a, b in ((pid[:-1], pid[1:]), (pid[:, :-1], pid[:, 1:])):
            a, b = a.reshape(-1), b.reshape(-1)
            both = (a >= 0) & (b >= 0)
            a, b = a[both], b[both]
            cross = self.dom[a] != self.dom[b]
            e.append(np.stack([a[cross], b[cross]]))
        self.edges = np.concatenate(e, 1)

    def slopes(self, phi, dim=0):
        """Fried slopes (sx of every subaperture, then sy) of a phase over the nodes."""
        a, b, c, d = (phi.index_select(dim, _idx(q)) for q in self.corner)
        return torch.cat([0.5 * (b + d - a - c), 0.5 * (c + d - a - b)], dim)


def _idx(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def _instances(case):
    """(nsub, m) of every system of a case."""
    if case["count"] == 1:
        return [(case["nsub"], case["m"])]
    r = random.Random(1000 * case["count"] + case["nsub"])
    sizes = [m for m in (16, 24, 32, 48) if m <= case["m"]]
    return [(r.randint(16, case["nsub"]), r.choice(sizes)) for _ in range(case["count"])]


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _screens(gen, count, g, r0, l0):
    """von Karman phase screens [count, g, g] at the node pitch (periodic), rad."""
    f = torch.fft.fftfreq(g, PITCH, dtype=torch.float64, device="cuda")
    f2 = f[:, None] ** 2 + f[None, :] ** 2
    amp = (0.023 * r0 ** (-5 / 3) * (f2 + 1 / (l0 * l0)) ** (-11 / 6)).sqrt() / (g * PITCH)
    amp[0, 0] = 0.0
    out = []
    for k in range(0, count, 64):
        z = torch.randn((min(64, count - k), g, g, 2), generator=gen, dtype=torch.float64,
                        device="cuda")
        out.append((torch.fft.ifft2(torch.view_as_complex(z) * amp) * (g * g)).real)
    return torch.cat(out)


def _inputs(case, seed, k, nsub, m):
    """One system's inputs, FP64 values that the handle's real type holds exactly."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed * 1009 + k)
    geo = _Geometry(nsub, case["window"], case["obscuration"], case["square"], case["partition"])
    g = 32
    while g < 2 * (nsub + 1):
        g *= 2
    at = (_idx(geo.pts[:, 0]), _idx(geo.pts[:, 1]))
    q, a = case["q"], math.sqrt(1 - case["q"] ** 2)
    rt = torch.float64 if case["precision"] else torch.float32

    def at_nodes(count, l0=L0):
        return _screens(gen, count, g, R0, l0)[:, at[0], at[1]]

    def scaled(x, slope):
        return x * (slope / geo.slopes(x, 1).std())

    frames = case["frames"]
    bank = _screens(gen, BANK, g, R0, L0).float()
    phi = at_nodes(1)[0]                                     # the turbulence, and its evolution
    truth = []
    for x in at_nodes(frames):
        truth.append(phi)
        phi = a * phi + q * x
    truth = torch.stack(truth)
    if case["state"] == "prior":
        prev = at_nodes(m)
    else:
        mean = truth[0] + scaled(at_nodes(1, 16 * PITCH), 3 * SIGMA)[0]
        prev = mean + scaled(at_nodes(m, 16 * PITCH), LOOP_SLOPE)
    X = torch.stack([a * prev + q * at_nodes(m), prev], 1)   # [m, 2, n]
    noise = SIGMA * torch.randn((frames, 2 * geo.ns), generator=gen, dtype=torch.float64,
                                device="cuda")
    seen = truth                                             # what the sensor sees per frame
    if case["kind"] == "dm":                                 # residual phase: the error left
        seen = scaled(at_nodes(frames, 16 * PITCH), 3 * SIGMA)
    y = geo.slopes(seen, 1) + noise
    return dict(geo=geo, m=m, a=a, seed=seed * 64 + k,
                X0=X.permute(2, 1, 0).contiguous().to(rt), y=y.to(rt),
                truth=truth.to(rt), bank=bank,
                v=(q * at_nodes(2 * m)).reshape(2, m, -1).transpose(1, 2).contiguous().to(rt)
                if case["kind"] == "dm" else None)


class _Csr:
    """The CSR arrays ``Letkf.set_dm`` reads of a dense matrix."""

    def __init__(self, dense):
        nz = dense != 0
        self.indptr = np.concatenate([[0], np.cumsum(nz.sum(1))])
        self.indices, self.data = np.nonzero(nz)[1], dense[nz]

    def tocsr(self):
        return self


def _mirror(geo):
    """Influence matrix N (coupling 0.3, 5 x 5 support) and command matrix P = N^-1 with its
    smallest entries dropped, as a controller calibrates them."""
    d = np.abs(geo.pts[:, None, :] - geo.pts[None, :, :])
    N = np.where(d.max(-1) <= 2, 0.3 ** (d ** 2).sum(-1), 0.0)
    P = np.linalg.inv(N)
    return N, np.where(np.abs(P) >= 1e-6 * np.abs(P).max(), P, 0.0)


def prepare(case, seed):
    ins = [_inputs(case, seed, k, nsub, m) for k, (nsub, m) in enumerate(_instances(case))]
    dev = dict(rho=case["rho"], precision=case["precision"])
    work = [Workload(f"perf-{k}", nsub=i["geo"].nsub, pitch=PITCH, obscuration=case["obscuration"],
                     square=case["square"], m=i["m"], window=case["window"], taper=case["taper"],
                     loc_len=0.0, sigma=SIGMA, q_model=case["q"], r0=R0, L0=L0,
                     frames=case["frames"], truth="frozen", seeds=(0, 0, i["seed"]),
                     bank_count=BANK, partition=case["partition"], piston=int(case["piston"]),
                     **dev) for k, i in enumerate(ins)]
    banks = [i["bank"].cpu().numpy() for i in ins]
    f = Letkf.batch(work, banks) if len(ins) > 1 else Letkf.from_workload(work[0], banks[0])
    s = dict(case=case, f=f, X0=ins[0]["X0"], y=torch.cat([i["y"] for i in ins], 1),
             truth=ins[0]["truth"], v=ins[0]["v"])
    if len(ins) > 1:
        s["X0"] = torch.cat([i["X0"].reshape(-1) for i in ins])
    if case["kind"] == "dm":
        N, P = _mirror(ins[0]["geo"])
        f.set_dm(_Csr(N), _Csr(P))
    if case["kind"] == "step":
        s["y"] = [np.ascontiguousarray(v) for v in s["y"].cpu().numpy()]
    return s


def run(s):
    case, f, y = s["case"], s["f"], s["y"]
    f.set_state(s["X0"])
    if case["kind"] == "analyze":
        mean, spread = f.analyze(y[0])
        return dict(mean=mean, spread=spread, X=f.get_state())
    f.set_frame(0)
    if case["kind"] == "run":
        f.run(case["frames"], y)
        return dict(X=f.get_state())
    if case["kind"] == "step":
        means = [f.step(v)[0] for v in y]
        return dict(means=means, X=f.get_state())
    if case["kind"] == "dm":
        # two predictions drive the mirror before the sensor's first frame arrives
        f.forecast(s["v"][0])
        f.forecast(s["v"][1])
        f.run(case["frames"], y)
        return dict(X=f.get_state(), u=f.command())
    J, g = f.grad(case["frames"], y, s["truth"], case["ckpt"])
    return dict(J=J, grad=g, X=f.get_state())


def work(case):
    size, total = 8 if case["precision"] else 4, dict(bytes=0.0, flops=0.0)
    for nsub, m in _instances(case):
        geo = _Geometry(nsub, case["window"], case["obscuration"], case["square"],
                        case["partition"])
        tau = _taper(case, torch.as_tensor(np.array(geo.dist)), None).numpy()
        slopes = 2.0 * float(((geo.obs < geo.ns) & (tau != 0)).sum())
        # the slope anomalies, the symmetric Gram matrices, and the ensemble's rows times the
        # transform; a gradient does as much again twice
        frame = 8.0 * geo.ns * m + slopes * m * (m + 1) + 4.0 * geo.n * m * m
        io = 2.0 * 2 * geo.n * m + 2.0 * geo.ns + 4.0 * geo.n
        n = case["frames"] if case["kind"] != "analyze" else 1
        total["flops"] += n * frame * (3 if case["kind"] == "grad" else 1)
        total["bytes"] += n * io * size * (2 if case["kind"] == "grad" else 1)
    return total


# ---------------------------------------------------------------------------
# The same results in FP64 torch
# ---------------------------------------------------------------------------
def _gaspari_cohn(z):
    a = (((-0.25 * z + 0.5) * z + 0.625) * z - 5.0 / 3.0) * z * z + 1.0
    b = ((((z / 12.0 - 0.5) * z + 0.625) * z + 5.0 / 3.0) * z - 5.0) * z + 4.0 \
        - (2.0 / 3.0) / z.clamp(min=0.5)
    return torch.where(z <= 1, a, torch.where(z < 2, b, torch.zeros_like(z)))


def _taper(case, dist, c):
    if case["taper"] == 0:
        return torch.ones_like(dist)
    return _gaspari_cohn(dist / (case["window"] / 4.0 if c is None else c))


def _newton_root(A):
    """A^-1/2 of SPD matrices [.., m, m] by coupled Newton-Schulz iterations."""
    s = A.flatten(-2).norm(dim=-1)[..., None, None]
    eye = torch.eye(A.shape[-1], dtype=A.dtype, device=A.device)
    Y, Z = A / s, eye.expand_as(A)
    left = math.inf
    for _ in range(80):
        T = 0.5 * (3 * eye - Z @ Y)
        Y, Z = Y @ T, T @ Z
        now = float((T - eye).abs().max())
        if now < 1e-14 or (now < 1e-9 and now >= left):
            break
        left = now
    return Z / s.sqrt()


class _EigRoot(torch.autograd.Function):
    """A^-1/2 of a symmetric A with its derivative (divided differences)."""

    @staticmethod
    def forward(ctx, A):
        lam, Q = (x.to(A.device) for x in torch.linalg.eigh(A.cpu()))
        ctx.save_for_backward(lam, Q)
        return (Q / lam.sqrt()[..., None, :]) @ Q.mT

    @staticmethod
    def backward(ctx, g):
        lam, Q = ctx.saved_tensors
        r = lam.sqrt()
        F = -1.0 / (r[..., :, None] * r[..., None, :] * (r[..., :, None] + r[..., None, :]))
        return Q @ (F * (Q.mT @ (0.5 * (g + g.mT)) @ Q)) @ Q.mT


def _analysis(geo, tau, X, y, sigma2, rho, root):
    """Analysis ensemble: per group A = (m-1)/rho I + Yb^T R^-1 Yb, wbar = A^-1 Yb^T R^-1 d,
    W = sqrt(m-1) A^-1/2, Xa = xbar + X' (wbar 1^T + W)."""
    n, m = X.shape[0], X.shape[-1]
    mean = X.mean(-1, keepdim=True)
    P = X - mean
    zero = X.new_zeros((1, 2, m))
    Yb = geo.slopes(P[:, 1]).reshape(2, geo.ns, m).transpose(0, 1)
    d = (y - geo.slopes(mean[:, 1, 0])).reshape(2, geo.ns).T
    Yb, d = torch.cat([Yb, zero]), torch.cat([d, zero[..., 0]])
    Pz = torch.cat([P, zero])
    eye = torch.eye(m, dtype=X.dtype, device=X.device)
    out, at = [], []
    step = max(1, int(2e8 // (m * (2 * geo.obs.shape[1] + 6 * m) * 8)))
    for k in range(0, len(geo.obs), step):
        ob, ro = _idx(geo.obs[k:k + step]), _idx(geo.rows[k:k + step])
        Yl = Yb[ob].flatten(1, 2)                               # [G, 2L, m]
        w = (tau[k:k + step] / sigma2).repeat_interleave(2, 1)
        A = Yl.mT @ (w[..., None] * Yl) + (m - 1) / rho * eye
        c = (Yl.mT @ (w * d[ob].flatten(1))[..., None])
        S = root(A)
        wbar = S @ (S @ c)
        wbar = wbar + S @ (S @ (c - A @ wbar))
        rows = Pz[ro].flatten(1, 2)                             # [G, 2R, m]
        upd = rows @ (wbar + math.sqrt(m - 1) * S)
        keep = (ro < n).flatten()
        out.append(upd.reshape(-1, 2, m)[keep])
        at.append(ro.flatten()[keep])
    order = torch.argsort(torch.cat(at))
    return mean + torch.cat(out)[order]


def _pistons(geo, delta):
    """Per domain and state row the constant that best removes the jumps of the increment
    ``delta`` [n, 2] across domain borders, with zero node-weighted mean."""
    D = int(geo.dom.max()) + 1
    i, j = geo.dom[geo.edges[0]], geo.dom[geo.edges[1]]
    E = torch.zeros((len(i), D), dtype=torch.float64, device="cuda")
    r = torch.arange(len(i), device="cuda")
    E[r, _idx(i)] = 1.0
    E[r, _idx(j)] = -1.0
    jump = delta[_idx(geo.edges[0])] - delta[_idx(geo.edges[1])]
    c = -torch.linalg.pinv(E.T @ E, hermitian=True) @ (E.T @ jump)
    w = torch.bincount(_idx(geo.dom), minlength=D).double()
    return c - (w[:, None] * c).sum(0) / w.sum()


def _bank_noise(inp, q, frame):
    bank, m, mask64 = inp["bank"].double(), inp["m"], (1 << 64) - 1
    g = bank.shape[-1]
    i, j = _idx(inp["geo"].pts[:, 0]), _idx(inp["geo"].pts[:, 1])
    out = []
    for k in range(m):
        z = (inp["seed"] + (((frame << 16) | k) + 1) * 0x9E3779B97F4A7C15) & mask64
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask64
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask64
        z ^= z >> 31
        out.append(bank[z % bank.shape[0], (i + (z >> 16) % g) % g, (j + (z >> 40) % g) % g])
    return q * torch.stack(out, -1)


def _exact_one(case, inp):
    geo, a, q, sigma2, rho = inp["geo"], inp["a"], case["q"], SIGMA ** 2, case["rho"]
    X, y, kind = inp["X0"].double(), inp["y"].double(), case["kind"]
    tau = _taper(case, _idx(np.array(geo.dist)), None) * (_idx(geo.obs) < geo.ns)

    def forecast(Xa, v):
        return torch.stack([a * Xa[:, 0] + v, Xa[:, 0]], 1)

    if kind == "analyze":
        Xa = _analysis(geo, tau, X, y[0], sigma2, rho, _newton_root)
        if case["piston"]:
            Xa = Xa + _pistons(geo, (Xa - X).mean(-1))[_idx(geo.dom)][..., None]
        return dict(mean=Xa.mean(-1), spread=Xa.std(-1), X=Xa)
    if kind == "grad":
        par = [torch.tensor(v, dtype=torch.float64, device="cuda", requires_grad=True)
               for v in (rho, sigma2, case["window"] / 4.0)]
        tau = _taper(case, _idx(np.array(geo.dist)), par[2]) * (_idx(geo.obs) < geo.ns)
        J = 0.0
        for k in range(case["frames"]):
            r = inp["truth"][k].double() - X[:, 0].mean(-1)
            J = J + r.var(unbiased=False) / case["frames"]
            X = _analysis(geo, tau, X, y[k], par[1], par[0], _EigRoot.apply)
            X = forecast(X, _bank_noise(inp, q, k))
        J.backward()
        return dict(J=float(J.detach()), grad=np.array([float(p.grad) for p in par]),
                    X=X.detach())
    u, first = [], 0
    if kind == "dm":
        N, P = (torch.as_tensor(v, device="cuda") for v in _mirror(geo))
        for k in range(2):
            X = forecast(X, inp["v"][k].double())
            u.append(P @ X[:, 0].mean(-1))
        first = 2
    means = []
    for k in range(case["frames"]):
        yk = y[k] + geo.slopes(N @ u[-2]) if kind == "dm" else y[k]
        X = _analysis(geo, tau, X, yk, sigma2, rho, _newton_root)
        means.append(X.mean(-1))
        X = forecast(X, _bank_noise(inp, q, first + k))
        if kind == "dm":
            u.append(P @ X[:, 0].mean(-1))
    if kind == "dm":
        return dict(X=X, u=u[-1])
    return dict(means=means, X=X) if kind == "step" else dict(X=X)


def exact(case, seed):
    ins = _instances(case)
    if len(ins) == 1:
        return _exact_one(case, _inputs(case, seed, 0, *ins[0]))
    out = [_exact_one(case, _inputs(case, seed, k, *s))["X"].reshape(-1)
           for k, s in enumerate(ins)]
    return dict(X=torch.cat(out))
