"""The work that is timed and compared from one version of this package to the next.

A case is one call (or one whole solve) as a user's program makes it, through the
public entry points of ``paper_1807_10151_gb300``.  ``listed()`` names the fixed
cases, ``draw(rng)`` gives more of the same ranges, ``prepare`` makes what the program
has in hand before the call, ``run`` is the call, ``work`` what it cannot do without,
and ``exact`` the same result from plain torch in FP64.

Inputs are seeded: sums of random ellipses (their images at pixel centres, their line
integrals in closed form), Gaussian or Poisson noise, and for the network random
parameters of the initialiser's scale.
"""
import math
import random

import numpy as np
import torch

import paper_1807_10151_gb300 as S

DEV = "cuda"


def listed():
    return [
        # one projection of a small slice: launch and call latency decide
        dict(name="project_64", op="project", nx=64, ny=64, views=90, bins=95, batch=1, storage="f32", shift=0.0),
        # one projection of the benchmark's slice
        dict(name="project_512", op="project", nx=512, ny=512, views=720, bins=725, batch=1, storage="f32", shift=0.0),
        # two large slices in BF16 storage
        dict(name="project_2048_bf16_x2", op="project", nx=2048, ny=2048, views=2880, bins=2900, batch=2,
             storage="bf16", shift=0.0),
        # a stack of odd-sized slices (the paper's 243-pixel image), backprojected together
        dict(name="backproject_243_x8", op="backproject", nx=243, ny=243, views=360, bins=345, batch=8,
             storage="f32", shift=0.0),
        # the preconditioner alone, on the benchmark's image size
        dict(name="precondition_512", op="precondition", nx=512, ny=512, batch=1, mu=1e-5, rho=0.8),
        # Algorithm 1 with Table 1's parameters: forty nonascending steps, as for the training pairs
        dict(name="superiorize_512_k40", op="superiorize", nx=512, ny=512, K=40, a=1 - 1e-5, gamma=1e-2),
        # the network's proposals for eight iterates at once (the batched learned solve)
        dict(name="network_512_x8", op="network", nx=512, ny=512, count=8),
        # the gradients of one training minibatch
        dict(name="gradients_128_x32", op="gradients", nx=128, ny=128, count=32),
        # a whole solve of the small configuration
        dict(name="solve_64", op="solve", problems="64:90", K=1, a=0.995, gamma=0.5, iters=8, photons=0.0),
        # a whole solve of the benchmark's problem
        dict(name="solve_512", op="solve", problems="512:720", K=1, a=0.995, gamma=0.5, iters=8, photons=1e5),
        # uneven problems in one batched schedule
        dict(name="batch_uneven", op="batch", problems="256:180,320:500,375:240,432:360,512:720,640:300", K=1,
             a=0.995, gamma=0.5, iters=5, photons=0.0),
        # one cycle of the row-action method the paper compares with
        dict(name="art_512", op="art", problems="512:720", r=5.0, lam=1e-2, cycles=1, photons=1e5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _smooth(lo, hi):
    """Sides of the form 2^a 3^b 5^c."""
    out = []
    for n in range(lo, hi + 1):
        m = n
        for p in (2, 3, 5):
            while m % p == 0:
                m //= p
        if m == 1:
            out.append(n)
    return out


def draw(rng):
    op = rng.choice(["project", "backproject", "precondition", "superiorize", "network", "gradients", "solve", "solve",
                     "batch", "art"])
    if op in ("project", "backproject"):
        nx = _log_int(rng, 40, 1100)
        ny = nx if rng.random() < 0.5 else max(33, int(nx * rng.uniform(0.6, 1.2)))
        n = max(nx, ny)
        batch = rng.choice([1, 1, 1, 2, 5]) if n < 600 else 1
        return dict(op=op, nx=nx, ny=ny, views=_log_int(rng, 45, 1440), bins=int(math.ceil(1.42 * n)) + rng.randrange(8),
                    batch=batch, storage=rng.choice(["f32", "f32", "bf16"]), shift=rng.choice([0.0, 0.3]))
    if op == "precondition":
        side, want = _smooth(32, 1536), _log_int(rng, 32, 1536)
        nx = min(side, key=lambda n: abs(n - want))
        ny = nx if rng.random() < 0.5 else min(side, key=lambda n: abs(n - int(nx * rng.uniform(0.7, 1.3))))
        return dict(op=op, nx=nx, ny=ny, batch=rng.choice([1, 1, 2, 3]), mu=rng.choice([1e-5, 1e-4, 1e-3]),
                    rho=rng.choice([0.6, 0.8]))
    if op == "superiorize":
        nx = _log_int(rng, 96, 1400)
        ny = nx if rng.random() < 0.5 else max(96, int(nx * rng.uniform(0.6, 1.2)))
        K, gamma = rng.choice([(1, 0.5), (1, 5e-2), (5, 1e-2), (10, 1e-2), (20, 1e-2), (40, 1e-2)])
        return dict(op=op, nx=nx, ny=ny, K=K, a=rng.choice([1 - 1e-5, 1 - 1e-3]), gamma=gamma)
    if op == "network":
        nx = _log_int(rng, 64, 800)
        ny = nx if rng.random() < 0.5 else max(64, int(nx * rng.uniform(0.6, 1.0)))
        return dict(op=op, nx=nx, ny=ny, count=rng.randrange(1, max(1, min(8, 2097152 // (nx * ny))) + 1))
    if op == "gradients":
        nx = _log_int(rng, 32, 256)
        ny = nx if rng.random() < 0.5 else max(32, int(nx * rng.uniform(0.6, 1.0)))
        return dict(op=op, nx=nx, ny=ny, count=rng.randrange(4, max(4, min(32, 524288 // (nx * ny))) + 1))
    side = _smooth(40, 640)
    pick = lambda lo, hi: min(side, key=lambda n, t=_log_int(rng, lo, hi): abs(n - t))  # noqa: E731
    # the benchmark's perturbation (one step of length 0.5 a^l) or Table 1's short steps
    K, a, gamma = rng.choice([(1, 0.995, 0.5), (1, 0.995, 0.5), (10, 1 - 1e-5, 1e-2), (40, 1 - 1e-5, 1e-2)])
    if op == "solve":
        return dict(op=op, problems="%d:%d" % (pick(64, 640), _log_int(rng, 60, 720)), K=K, a=a, gamma=gamma,
                    iters=rng.randrange(3, 9), photons=rng.choice([0.0, 1e5]))
    if op == "batch":
        some = ["%d:%d" % (pick(64, 480), _log_int(rng, 60, 500)) for _ in range(rng.randrange(2, 7))]
        return dict(op=op, problems=",".join(some), K=min(K, 10), a=a, gamma=gamma, iters=rng.randrange(3, 7), photons=0.0)
    return dict(op=op, problems="%d:%d" % (_log_int(rng, 40, 512), _log_int(rng, 60, 500)), r=5.0,
                lam=rng.choice([1e-2, 5e-2]), cycles=1, photons=rng.choice([0.0, 1e5]))


# ---------------------------------------------------------------- inputs
def _problems(case):
    """[(N, views, bins)] of a case that solves problems."""
    out = []
    for p in case["problems"].split(","):
        n, v = (int(t) for t in p.split(":"))
        out.append((n, v, 725 if (n, v) == (512, 720) else 95 if (n, v) == (64, 90) else int(math.ceil(1.42 * n))))
    return out


def _ellipses(seed, count=15):
    r = random.Random(seed)
    out = []
    for _ in range(count):
        rad, phi = 0.35 * math.sqrt(r.random()), 2 * math.pi * r.random()
        out.append((rad * math.cos(phi), rad * math.sin(phi), r.uniform(0.03, 0.2), r.uniform(0.03, 0.2),
                    math.pi * r.random(), 0.4 * r.random()))
    return out


def _centres(nx, ny, d):
    x = (torch.arange(nx, device=DEV, dtype=torch.float64) - 0.5 * (nx - 1)) * d
    y = (0.5 * (ny - 1) - torch.arange(ny, device=DEV, dtype=torch.float64)) * d
    return x[None, :], y[:, None]


def _image(nx, ny, seed, noise=0.0):
    """Sum of ellipses at pixel centres on the unit square, with the noise of an iterate."""
    x, y = _centres(nx, ny, 1.0 / max(nx, ny))
    img = torch.zeros(ny, nx, device=DEV)
    for cx, cy, ax, ay, ang, rho in _ellipses(seed):
        u = (x - cx) * math.cos(ang) + (y - cy) * math.sin(ang)
        v = -(x - cx) * math.sin(ang) + (y - cy) * math.cos(ang)
        img += rho * ((u / ax) ** 2 + (v / ay) ** 2 <= 1.0).float()
    if noise:
        g = torch.Generator(device=DEV).manual_seed(seed)
        img += noise * torch.randn(ny, nx, device=DEV, generator=g)
    return img


def _cos_sin(views):
    """cos and sin of v pi / V, exact on the axes."""
    c, s = [], []
    for v in range(views):
        q = 2.0 * v / views
        on_axis = q == int(q)
        c.append((1.0, 0.0)[int(q)] if on_axis else math.cos(v * math.pi / views))
        s.append((0.0, 1.0)[int(q)] if on_axis else math.sin(v * math.pi / views))
    return (torch.tensor(t, device=DEV, dtype=torch.float64) for t in (c, s))


def _data(N, views, bins, seed, photons):
    """Line integrals of the ellipses with Poisson counts (photons > 0) or 1 % Gaussian noise."""
    c, s = (t[:, None] for t in _cos_sin(views))
    pos = ((torch.arange(bins, device=DEV, dtype=torch.float64) - 0.5 * (bins - 1)) / N)[None, :]
    b = torch.zeros(views, bins, device=DEV, dtype=torch.float64)
    for cx, cy, ax, ay, ang, rho in _ellipses(seed):
        ca, sa = c * math.cos(ang) + s * math.sin(ang), s * math.cos(ang) - c * math.sin(ang)
        w = ax * ax * ca * ca + ay * ay * sa * sa
        b += 2.0 * rho * ax * ay * torch.sqrt((w - (pos - cx * c - cy * s) ** 2).clamp_min(0.0)) / w
    g = torch.Generator(device=DEV).manual_seed(seed)
    if photons:
        counts = torch.poisson(photons * torch.exp(-b), generator=g)
        b = -torch.log(counts.clamp_min(1.0) / photons)
    else:
        b = b + 0.01 * b.square().mean().sqrt() * torch.randn(b.shape, device=DEV, dtype=torch.float64, generator=g)
    return b.float()


def _net_params(seed):
    r = np.random.RandomState(seed % (1 << 31))
    flat = []
    for k, (co, ci) in enumerate(S.CNN_SHAPES):
        flat.append(r.standard_normal(co * ci * 9) * math.sqrt(2.0 / (9 * ci)) * (0.3 if k == len(S.CNN_SHAPES) - 1 else 1.0))
        flat.append(0.05 * r.standard_normal(co))
    return np.concatenate(flat).astype(np.float32)


def _inputs(case, seed):
    """The arrays a case starts from (the same for run and exact)."""
    op = case["op"]
    if op == "project":
        dt = torch.bfloat16 if case["storage"] == "bf16" else torch.float32
        return torch.stack([_image(case["nx"], case["ny"], seed + 100 * k, 0.01) for k in range(case["batch"])]).to(dt)
    if op == "backproject":
        dt = torch.bfloat16 if case["storage"] == "bf16" else torch.float32
        n = max(case["nx"], case["ny"])
        return torch.stack([_data(n, case["views"], case["bins"], seed + 100 * k, 0.0) for k in range(case["batch"])]).to(dt)
    if op == "precondition":
        # a gradient: smooth and large at low frequencies, noisy at the others
        out = []
        for k in range(case["batch"]):
            img = _image(case["nx"], case["ny"], seed + 100 * k, 0.01)
            x, y = _centres(case["nx"], case["ny"], 1.0 / max(case["nx"], case["ny"]))
            out.append(img + (20.0 * torch.exp(-4.0 * (x * x + y * y))).float())
        return torch.stack(out)
    if op == "superiorize":
        return _image(case["nx"], case["ny"], seed, 0.02)
    if op in ("network", "gradients"):
        xs = torch.stack([_image(case["nx"], case["ny"], seed + 100 * k, 0.02) for k in range(case["count"])])
        ts = torch.stack([_tv_tbar(x.double())[1] for x in xs]).float()
        if op == "network":
            return xs, ts, _net_params(seed)
        # the target: the direction of a longer path, near tbar and smoother
        return xs, ts, (0.8 * ts + 0.1 * (ts.roll(1, -1) + ts.roll(1, -2))).contiguous(), _net_params(seed)
    return [_data(N, v, u, seed + 100 * k, case["photons"]) for k, (N, v, u) in enumerate(_problems(case))]


def _geometry(case):
    return S.Geometry(case["nx"], case["ny"], n_views=case["views"], n_bins=case["bins"],
                      offset=case["shift"] / max(case["nx"], case["ny"]), storage=case["storage"])


def prepare(case, seed):
    op = case["op"]
    st = {"case": case, "in": _inputs(case, seed)}
    if op in ("project", "backproject"):
        st["G"] = _geometry(case)
    elif op in ("precondition", "superiorize"):
        st["G"] = S.Geometry(case["nx"], case["ny"], n_views=4)
    elif op in ("network", "gradients"):
        st["net"] = S.CNN(case["ny"], case["nx"], max_batch=case["count"], seed=1)
        st["net"].set_params(st["in"][-1])
    else:
        st["Gs"] = [S.Geometry(N, n_views=v, n_bins=u) for N, v, u in _problems(case)]
    return st


def run(st):
    case, a = st["case"], st["in"]
    op = case["op"]
    if op == "project":
        return st["G"].project(a)
    if op == "backproject":
        return st["G"].backproject(a)
    if op == "precondition":
        return st["G"].precondition(a, mu=case["mu"], rho=case["rho"])
    if op == "superiorize":
        x = a.clone()
        rc, ell, trials = st["G"].superiorize(x, 0, case["a"], case["gamma"], case["K"])
        return {"x": x, "ell": ell, "trials": np.array(trials), "status": rc}
    if op == "network":
        return st["net"].forward(a[0], a[1])
    if op == "gradients":
        g, loss = st["net"].gradients(a[0], a[1], a[2])
        return {"gradients": g, "loss": loss}
    if op == "art":
        x, rep = st["Gs"][0].art(a[0], r=case["r"], lam=case["lam"], cycles=case["cycles"])
        return {"x": x, "mu": rep["mu"]}
    kw = dict(K=case["K"], a=case["a"], gamma=case["gamma"], max_iter=case["iters"])
    if op == "solve":
        x, rep, _ = st["Gs"][0].solve(a[0], **kw)
        xs, reps = [x], [rep]
    else:
        xs = [torch.zeros(G.ny, G.nx, device=DEV) for G in st["Gs"]]
        reps = S.solve_batched(st["Gs"], a, xs, **kw)
    return {"x": xs, "ell": [r["ell"] for r in reps], "f": [r["f_last"] for r in reps], "tv": [r["tv_last"] for r in reps]}


# ---------------------------------------------------------------- what a pass cannot do without
def _nnz(nx, ny, views):
    """Ray-pixel intersections of one projection (4/pi of them per pixel and view on average)."""
    return nx * ny * views * 4.0 / math.pi


def work(case):
    op = case["op"]
    if op in ("project", "backproject"):
        es = 2 if case["storage"] == "bf16" else 4
        n, m = case["nx"] * case["ny"], case["views"] * case["bins"]
        return {"bytes": es * case["batch"] * (n + m), "flops": 2.0 * case["batch"] * _nnz(case["nx"], case["ny"], case["views"])}
    if op in ("art", "solve", "batch"):
        nbytes = flops = 0.0
        for N, v, u in _problems(case):
            n, nnz = N * N, _nnz(N, N, v)
            if op == "art":
                nbytes += 4.0 * (n + v * u)
                flops += case["cycles"] * 4.0 * nnz
            else:   # per iteration two projections, two backprojections, the filter, the nonascending steps
                nbytes += 4.0 * (n + v * u)
                flops += (case["iters"] + 1) * (8.0 * nnz + 5.0 * n * math.log2(n)) + case["iters"] * case["K"] * 40.0 * n
        return {"bytes": nbytes, "flops": flops}
    n = case["nx"] * case["ny"]
    if op == "precondition":
        return {"bytes": 8.0 * n * case["batch"], "flops": 5.0 * n * math.log2(n) * case["batch"]}
    if op == "superiorize":
        return {"bytes": 8.0 * n, "flops": 40.0 * n * case["K"]}
    macs = sum(co * ci * 9 for co, ci in S.CNN_SHAPES)
    if op == "network":
        return {"bytes": 12.0 * n * case["count"], "flops": 2.0 * macs * n * case["count"]}
    return {"bytes": 12.0 * n * case["count"], "flops": 6.0 * macs * n * case["count"]}


# ---------------------------------------------------------------- the same in FP64
class _R64:
    """Ray sums and their transpose from exact intersection lengths in FP64, in bin units."""

    def __init__(self, nx, ny, views, bins, d, off=0.0):
        self.nx, self.ny, self.V, self.U, self.d = nx, ny, views, bins, d
        self.c, self.s = _cos_sin(views)
        self.uc = 0.5 * (bins - 1) - off / d
        big, small = torch.maximum(self.c.abs(), self.s.abs()), torch.minimum(self.c.abs(), self.s.abs())
        self.E, self.P, self.hw = 0.5 * (big + small), d / big, 0.5 * (big + small) / big
        self.slope = torch.where(small > 0, 1.0 / small.clamp_min(1e-300), torch.zeros_like(small))   # of length / P per bin
        self.axis = small == 0
        self.X = torch.arange(nx, device=DEV, dtype=torch.float64) - 0.5 * (nx - 1)
        self.Y = 0.5 * (ny - 1) - torch.arange(ny, device=DEV, dtype=torch.float64)

    def _w(self, v, delta):
        """Lengths at distance `delta` of rays of the views v (first dimension)."""
        at = lambda t: t[v].reshape([-1] + [1] * (delta.dim() - 1))  # noqa: E731
        ad, E = delta.abs(), at(self.E)
        w = ((E - ad) * at(self.slope)).clamp(0.0, 1.0)
        if bool(self.axis[v].any()):
            box = (ad < E).double() + 0.5 * (ad == E).double()
            w = torch.where(at(self.axis), box, w)
        return w * at(self.P)

    def _groups(self, per_view):
        """(walks rows?, views) in runs that keep the temporaries small."""
        rows = self.c.abs() >= self.s.abs()
        step = max(1, int(1.2e7 // per_view))
        for flag in (True, False):
            v = torch.nonzero(rows == flag).flatten()
            for k in range(0, v.numel(), step):
                yield flag, v[k:k + step]

    def entries(self, flag, v):
        """For each candidate k: lengths [v][outer][u] and inner indices of the rays of the views v."""
        co, ci = (self.s, self.c) if flag else (self.c, self.s)
        O = (self.Y if flag else self.X)[None, :, None]
        tau = (torch.arange(self.U, device=DEV, dtype=torch.float64) - self.uc)[None, None, :]
        rest = tau - co[v][:, None, None] * O
        cin = ci[v][:, None, None]
        centre = rest / cin
        q = centre + 0.5 * (self.nx - 1) if flag else 0.5 * (self.ny - 1) - centre
        q0 = torch.ceil(q - self.hw[v][:, None, None])
        for k in range(3):
            qk = q0 + k
            inner = qk - 0.5 * (self.nx - 1) if flag else 0.5 * (self.ny - 1) - qk
            yield self._w(v, rest - cin * inner), qk.clamp(-1, (self.nx if flag else self.ny)).long()

    def forward(self, x):
        """x [B][ny][nx] -> [B][V][U]."""
        y = torch.zeros(x.shape[0], self.V, self.U, device=DEV, dtype=torch.float64)
        pads = {f: torch.nn.functional.pad(x if f else x.transpose(1, 2), (1, 1)).contiguous() for f in (True, False)}
        for flag, v in self._groups(max(self.nx, self.ny) * self.U):
            img = pads[flag]
            row = torch.arange(img.shape[1], device=DEV)[None, :, None] * img.shape[2] + 1
            for w, q in self.entries(flag, v):
                at = (row + q).reshape(-1)
                for b in range(x.shape[0]):
                    y[b, v] += (w * img[b].reshape(-1)[at].reshape(w.shape)).sum(1)
        return y

    def backward(self, y):
        """y [B][V][U] -> [B][ny][nx]."""
        x = torch.zeros(y.shape[0], self.ny, self.nx, device=DEV, dtype=torch.float64)
        yp = torch.nn.functional.pad(y, (1, 1)).contiguous()
        for v in torch.arange(self.V, device=DEV).split(max(1, int(1.2e7 // (self.nx * self.ny)))):
            t = self.c[v][:, None, None] * self.X[None, None, :] + self.s[v][:, None, None] * self.Y[None, :, None] + self.uc
            u0 = torch.ceil(t - self.E[v][:, None, None])
            base = v[:, None, None] * (self.U + 2) + 1
            for k in range(2 if float(self.E.max()) < 1.0 else 3):
                u = u0 + k
                w = self._w(v, u - t)
                at = (base + u.clamp(-1, self.U).long()).reshape(-1)
                for b in range(y.shape[0]):
                    x[b] += (w * yp[b].reshape(-1)[at].reshape(w.shape)).sum(0)
        return x


def _tv_terms(y):
    a, b = y[:-1, :-1] - y[1:, :-1], y[:-1, :-1] - y[:-1, 1:]
    return a, b, torch.sqrt(a * a + b * b)


def _tv_tbar(y):
    """(TV, tbar): tbar = -dTV/dy where it exists, else 0."""
    a, b, t = _tv_terms(y)
    flat = t == 0
    ti = torch.where(flat, torch.zeros_like(t), 1.0 / torch.where(flat, torch.ones_like(t), t))
    g = torch.zeros_like(y)
    g[:-1, :-1] += (a + b) * ti
    g[1:, :-1] -= a * ti
    g[:-1, 1:] -= b * ti
    bad = torch.zeros_like(y, dtype=torch.bool)
    bad[:-1, :-1] |= flat
    bad[1:, :-1] |= flat
    bad[:-1, 1:] |= flat
    return t.sum(), torch.where(bad, torch.zeros_like(g), -g)


def _stv(y, ell, a, gamma, K):
    """Algorithm 1: (image, l, trials of each step)."""
    trials = []
    for _ in range(K):
        tv, t = _tv_tbar(y)
        nrm = float(t.square().sum().sqrt())
        t = t / nrm if nrm > 0 else t
        for n in range(1, 10001):
            z = y + gamma * a ** ell * t
            ell += 1
            if bool(_tv_terms(z)[2].sum() <= tv):
                break
        y = z
        trials.append(n)
    return y, ell, trials


def _filter(g, mu, rho):
    ny, nx = g.shape[-2:]
    w = [2 * math.pi * torch.minimum(torch.arange(n, device=DEV), n - torch.arange(n, device=DEV)).double() / n for n in (ny, nx)]
    wr = torch.sqrt(w[0][:, None] ** 2 + w[1][None, :] ** 2).clamp_max(math.pi)
    return torch.fft.ifft2((wr + mu) * (rho + (1 - rho) * torch.cos(wr)) * torch.fft.fft2(g)).real


def _solve64(R, b, K, a, gamma, iters, mu=1e-5, rho=0.8):
    """Algorithm 3 from x_0 = 0."""
    fwd, bwd = (lambda x: R.forward(x[None])[0]), (lambda y: R.backward(y[None])[0])
    x = torch.zeros(R.ny, R.nx, device=DEV, dtype=torch.float64)
    ell, p, h, tv, f = 0, None, None, 0.0, 0.0
    for k in range(iters + 1):
        if k:
            x = x + alpha * p  # noqa: F821
            x, ell, _ = _stv(x, ell, a, gamma, K)
            tv = float(_tv_terms(x)[2].sum())
        r = fwd(x) - b
        f = float(r.square().sum())
        if k == iters:
            break
        g = bwd(r)
        z = _filter(g, mu, rho)
        p = -z if p is None else -z + ((z * h).sum() / (p * h).sum()) * p
        h = bwd(fwd(p))
        alpha = -(g * p).sum() / (p * h).sum()
    return x, ell, f, tv


def _art64(R, b, r, lam, cycles):
    """Row action on r R (x - mu) + u = r (b - R mu), views in order, residue classes within a view."""
    mu = float(b.sum(1).mean()) * R.d / (R.nx * R.ny * R.d * R.d)
    classes = int(math.floor(2.0 * float(R.E.max()))) + 1
    x = torch.full((R.ny * R.nx + 1,), mu, device=DEV, dtype=torch.float64)   # the last entry: off the image
    u = torch.zeros_like(b)
    for _ in range(cycles):
        for v in range(R.V):
            flag = bool(R.c[v].abs() >= R.s[v].abs())
            ws, at = [], []
            for w, q in R.entries(flag, torch.tensor([v], device=DEV)):
                n_in = R.nx if flag else R.ny
                o = torch.arange(q.shape[1], device=DEV)[:, None]
                inside = (q[0] >= 0) & (q[0] < n_in)
                ws.append(torch.where(inside, w[0], torch.zeros_like(w[0])))
                at.append(torch.where(inside & (w[0] > 0), o * R.nx + q[0] if flag else q[0] * R.nx + o, R.ny * R.nx))
            w, pix = torch.stack(ws), torch.stack(at)
            x[-1] = 0.0
            for c in range(classes):
                wc, pc = w[:, :, c::classes], pix[:, :, c::classes]
                old = x[pc]
                cc = lam * (r * (b[v, c::classes] - (wc * old).sum((0, 1))) - u[v, c::classes]) / (1.0 + r * r * wc.square().sum((0, 1)))
                u[v, c::classes] += cc
                x[pc] = old + r * cc * wc
                x[-1] = 0.0
    return x[:-1].reshape(R.ny, R.nx), mu


def _net64(params, xs, ts):
    """The network without BF16 roundings: (output, parameters as FP64 leaves)."""
    unit = lambda t: t / t.square().mean((1, 2), keepdim=True).sqrt()  # noqa: E731
    leaves, off = [], 0
    flat = torch.tensor(params, device=DEV, dtype=torch.float64)
    for co, ci in S.CNN_SHAPES:
        for shape in ((co, ci, 3, 3), (co,)):
            n = math.prod(shape)
            leaves.append(flat[off:off + n].reshape(shape).clone().requires_grad_(True))
            off += n
    outs = []
    for x, t in zip(unit(xs.double()), unit(ts.double())):
        a = torch.stack([x, t])[None]
        for k in range(0, len(leaves), 2):
            a = torch.nn.functional.conv2d(a, leaves[k], leaves[k + 1], padding=1)
            a = torch.relu(a) if k + 2 < len(leaves) else a
        outs.append(a[0, 0] + t)
    return torch.stack(outs), leaves


def exact(case, seed):
    op = case["op"]
    a = _inputs(case, seed)
    if op in ("project", "backproject"):
        n = max(case["nx"], case["ny"])
        R = _R64(case["nx"], case["ny"], case["views"], case["bins"], 1.0 / n, case["shift"] / n)
        return R.forward(a.double()) if op == "project" else R.backward(a.double())
    if op == "precondition":
        return _filter(a.double(), case["mu"], case["rho"])
    if op == "superiorize":
        x, ell, trials = _stv(a.double(), 0, case["a"], case["gamma"], case["K"])
        return {"x": x, "ell": ell, "trials": np.array(trials), "status": 0}
    if op == "network":
        with torch.no_grad():
            return _net64(a[2], a[0], a[1])[0]
    if op == "gradients":
        out, leaves = _net64(a[3], a[0], a[1])
        t = a[2].double()
        loss = (out - t / t.square().mean((1, 2), keepdim=True).sqrt()).square().mean()
        loss.backward()
        return {"gradients": torch.cat([p.grad.reshape(-1) for p in leaves]), "loss": float(loss.detach())}
    Rs = [_R64(N, N, v, u, 1.0 / N) for N, v, u in _problems(case)]
    if op == "art":
        x, mu = _art64(Rs[0], a[0].double(), case["r"], case["lam"], case["cycles"])
        return {"x": x, "mu": mu}
    got = [_solve64(R, b.double(), case["K"], case["a"], case["gamma"], case["iters"]) for R, b in zip(Rs, a)]
    return {"x": [g[0] for g in got], "ell": [g[1] for g in got], "f": [g[2] for g in got], "tv": [g[3] for g in got]}
