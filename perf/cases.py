"""Performance cases of the library: what its users have it do, at the sizes they do it.

A case is a dict of plain values; `prepare` makes the inputs on the GPU and the context (and plan) that a
program keeps, `run` is one pass through the public entry points, `exact` the same results in 64 bits from
plain torch and numpy.  The kinds:

  pieces      S(h), dS/dh and one theta sweep of a given state, the calls a program with its own sampler makes
  chain       rsv_hmc_chain: a segment of a chain, in either precision, with or without theta, a mass, leverage
  trajectory  rsv_hmc_trajectory with the caller's momenta and Metropolis uniform
  batched     rsv_hmc_batched on a plan of many series
  mass        the learned mass from a segment of snapshots: moments, features, training, inference
  ess         effective sample sizes of a block of snapshots
"""
import math

import numpy as np
import torch

THETA = (0.95, -0.5, -0.2, 0.05, 0.1)         # phi, mu, xi, sigma_eta^2, sigma_u^2
THETA_LARGE = (0.97, -0.5, -0.2, 0.03, 0.1)
SCHEMES = {  # drifts a, kicks b per step
    "leapfrog": ((0.5, 0.5), (1.0,)),
    "omelyan2": ((0.19318332750378357, 1.0 - 2 * 0.19318332750378357, 0.19318332750378357), (0.5, 0.5)),
}


def listed():
    return [
        # ten years of daily data: the smallest calls, all launch latency and short reductions
        dict(name="pieces daily", kind="pieces", T=2000),
        # the same calls on the longest series of the benchmark
        dict(name="pieces 2^22", kind="pieces", T=1 << 22),
        # the FP64 reference sampler on a daily series, theta fixed
        dict(name="fp64 chain daily", kind="chain", prec="fp64", T=2000, n_md=50, dtau=0.02, n_traj=100,
             theta=False, mass=False, rho=0.0, integrator="leapfrog", snaps=False),
        # the FP64 sampler on a long series, theta sampled (the benchmark's FP64 arm)
        dict(name="fp64 chain 2^20", kind="chain", prec="fp64", T=1 << 20, n_md=100, dtau=0.005, n_traj=4,
             theta=True, mass=False, rho=0.0, integrator="leapfrog", snaps=False),
        # everyday use: a daily series, mixed precision, theta sampled, every state recorded
        dict(name="mixed chain daily", kind="chain", prec="mixed", T=2000, n_md=50, dtau=0.02, n_traj=200,
             theta=True, mass=False, rho=0.0, integrator="leapfrog", snaps=True),
        # the benchmark's headline: the learned-mass sampler on a long series, one window of trajectories
        dict(name="mixed chain 2^20 mass", kind="chain", prec="mixed", T=1 << 20, n_md=78, dtau=0.035, n_traj=50,
             theta=True, mass=True, rho=0.0, integrator="leapfrog", snaps=True),
        # the cheapest sampler per effective sample: minimum-norm integrator, few steps
        dict(name="mixed chain 2^20 2MN", kind="chain", prec="mixed", T=1 << 20, n_md=6, dtau=0.5 / 6, n_traj=50,
             theta=True, mass=False, rho=0.0, integrator="omelyan2", snaps=True),
        # the leverage model, theta fixed
        dict(name="mixed leverage 2^20", kind="chain", prec="mixed", T=1 << 20, n_md=100, dtau=0.005, n_traj=20,
             theta=False, mass=False, rho=-0.4, integrator="leapfrog", snaps=False),
        # one trajectory with the caller's momenta on the longest series
        dict(name="trajectory 2^22", kind="trajectory", prec="mixed", T=1 << 22, n_md=80, dtau=0.006),
        # many series at once, each with its own theta
        dict(name="batched 4096", kind="batched", prec="mixed", n=4096, T_lo=500, T_hi=8192, n_md=50, dtau=0.02,
             n_traj=4, mass=False),
        # one segment of snapshots folded in, then the mass trained and inferred
        dict(name="mass 2^20", kind="mass", T=1 << 20, rows=100, steps=500, batch=4096),
        # effective sample sizes of a recorded chain
        dict(name="ess 1000 x 2^17", kind="ess", n=1000, T=1 << 17),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pieces", "chain", "chain", "chain", "chain", "trajectory", "batched", "mass", "ess"])
    if kind == "pieces":
        return dict(kind=kind, T=_log_int(rng, 500, 1 << 22))
    if kind == "chain":
        prec = rng.choice(["fp64", "mixed", "mixed"])
        rho = rng.choice([0.0, 0.0, 0.0, -0.4])
        integ = rng.choice(["leapfrog", "leapfrog", "omelyan2"])
        T = _log_int(rng, 500, 1 << (20 if prec == "fp64" else 21))
        dtau = (0.02 if integ == "leapfrog" else 0.2) * (2000.0 / T) ** 0.25
        mass = rng.random() < 0.35
        if mass:
            dtau *= math.sqrt(30.0)  # time in units of the root of the mass
        n_md = max(1, round(0.5 * (math.sqrt(30.0) if mass else 1.0) / dtau))
        forces = n_md * (2 if integ == "omelyan2" else 1)
        cap = 4e8 if prec == "fp64" else 2.5e9  # site-steps of a pass
        n_traj = max(1, min(_log_int(rng, 4, 40 if prec == "fp64" else 200), int(cap / (T * forces))))
        return dict(kind=kind, prec=prec, T=T, n_md=n_md, dtau=dtau, n_traj=n_traj, theta=rho == 0.0 and rng.random() < 0.7,
                    mass=mass, rho=rho, integrator=integ, snaps=T * n_traj <= 1 << 26 and rng.random() < 0.6)
    if kind == "trajectory":
        prec = rng.choice(["fp64", "mixed"])
        T = _log_int(rng, 500, 1 << (20 if prec == "fp64" else 22))
        dtau = 0.04 * (2000.0 / T) ** 0.25
        return dict(kind=kind, prec=prec, T=T, n_md=rng.randint(20, 100), dtau=dtau)
    if kind == "batched":
        prec = rng.choice(["mixed", "mixed", "fp64"])
        T_hi = _log_int(rng, 600, 8192)
        n = _log_int(rng, 8, 4096 if prec == "mixed" else 256)
        return dict(kind=kind, prec=prec, n=n, T_lo=rng.randint(100, 500), T_hi=T_hi, n_md=rng.randint(20, 50), dtau=0.02,
                    n_traj=rng.randint(1, 4), mass=rng.random() < 0.3)
    if kind == "mass":
        return dict(kind=kind, T=_log_int(rng, 2000, 1 << 20), rows=rng.randint(2, 100), steps=_log_int(rng, 20, 500),
                    batch=64 * rng.randint(1, 64))
    return dict(kind="ess", n=_log_int(rng, 50, 1000), T=_log_int(rng, 500, 1 << 17))


# ---- inputs --------------------------------------------------------------------------------------------------------


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def _series(g, T, theta, rho=0.0):
    """Packed series of lengths T drawn from the model (theta [n, 5]): latent path h, returns y, lnRV, and the site's
    position in its series."""
    T = torch.as_tensor(T, device="cuda")
    N = int(T.sum())
    start = torch.cumsum(T, 0) - T
    pos = torch.arange(N, device="cuda") - torch.repeat_interleave(start, T)
    phi, mu, xi, se2, su2 = (torch.repeat_interleave(theta[:, k].contiguous(), T) for k in range(5))
    eps, z = _normal(g, N), _normal(g, N)
    prev = torch.cat([eps[:1], eps[:-1]])
    x = se2.sqrt() * (rho * prev + math.sqrt(1.0 - rho * rho) * z)
    x = torch.where(pos == 0, z * (se2 / (1.0 - phi * phi)).sqrt(), x)
    s, w = 1, phi.clone()  # x_t = sum_k phi^k eta_{t-k}, the window doubled each time
    longest, slow = int(T.max()), float(theta[:, 0].max())
    while s < longest and slow ** s > 1e-18:
        x[s:] += torch.where(pos[s:] >= s, w[s:] * x[:-s], torch.zeros((), dtype=x.dtype, device="cuda"))
        s, w = 2 * s, w * w
    h = x + mu
    y = torch.exp(0.5 * h) * eps
    lnrv = xi + h + su2.sqrt() * _normal(g, N)
    return h, y, lnrv, pos


def _mass(g, N):
    """1/m with the spread that a trained mass has: a few per cent around 1/30."""
    return (torch.exp(-0.03 * _normal(g, N).abs()) / 29.5).float()


def _inputs(c, seed):
    g, k = _gen(seed), c["kind"]
    d = {"seed": int(seed) & 0xFFFFFFFF}
    if k == "ess":
        rho = torch.rand(c["T"], generator=g, device="cuda") * 0.9
        x = torch.empty(c["n"], c["T"], device="cuda")
        x[0] = torch.randn(c["T"], generator=g, device="cuda")
        e = (1.0 - rho * rho).sqrt()
        for i in range(1, c["n"]):
            x[i] = rho * x[i - 1] + e * torch.randn(c["T"], generator=g, device="cuda")
        d["x"] = 0.2 * x - 0.5
        return d
    if k == "batched":
        r = np.random.default_rng(int(seed))
        T = np.random.default_rng(2).integers(c["T_lo"], c["T_hi"] + 1, c["n"])
        th = np.stack([r.uniform(0.85, 0.99, c["n"]), r.normal(-0.5, 0.3, c["n"]), r.normal(-0.2, 0.1, c["n"]),
                       r.uniform(0.02, 0.1, c["n"]), r.uniform(0.05, 0.2, c["n"])], axis=1)
    else:
        T = np.array([c["T"]])
        th = np.array([THETA_LARGE if k == "trajectory" else THETA])
    d["T"], d["theta"] = T, torch.tensor(th, device="cuda")
    d["h"], d["y"], d["lnrv"], d["pos"] = _series(g, T, d["theta"], c.get("rho", 0.0))
    if c.get("mass"):
        d["minv"] = _mass(g, d["h"].numel())
    if k == "trajectory":
        d["p"] = _normal(g, c["T"])
        d["log_u"] = torch.rand(1, generator=g, device="cuda", dtype=torch.float64).log()
    if k == "mass":
        sd = 0.18 + 0.02 * torch.rand(c["T"], generator=g, device="cuda")
        d["snaps"] = (d["h"].float() + sd * torch.randn(c["rows"], c["T"], generator=g, device="cuda")).contiguous()
    return d


def prepare(case, seed):
    from paper_1603_08114_gb300 import rsv

    s = _inputs(case, seed)
    s["case"], s["traj"] = case, 0
    ctx = s["ctx"] = rsv.Context(0)
    k = case["kind"]
    s.pop("pos", None)
    if k == "ess":
        return s
    rsv.rsv_reserve(ctx, s["h"].numel(), len(s["T"]))
    if k == "chain":
        rsv.rsv_set_leverage(ctx, case["rho"])
        rsv.rsv_set_integrator(ctx, case["integrator"])
        n = case["n_traj"]
        s["accept"] = torch.empty(n, dtype=torch.int32, device="cuda")
        s["dH"] = torch.empty(n, dtype=torch.float64, device="cuda") if case["prec"] == "fp64" else None
        s["theta_out"] = torch.empty(n, 5, dtype=torch.float64, device="cuda") if case["theta"] else None
        s["snaps"] = torch.empty(n, case["T"], device="cuda") if case["snaps"] else None
    if k == "batched":
        off = np.concatenate([[0], np.cumsum(s["T"])])
        s["plan"] = rsv.Plan(ctx, off, case["n_md"], prec=case["prec"], with_mass=case["mass"])
        s["accept"] = torch.empty(case["n_traj"], case["n"], dtype=torch.int32, device="cuda")
        s["dH"] = torch.empty(case["n_traj"], case["n"], dtype=torch.float64, device="cuda")
    return s


# ---- one pass ------------------------------------------------------------------------------------------------------


def run(s):
    from paper_1603_08114_gb300 import learned, rsv

    c, ctx, k = s["case"], s["ctx"], s["case"]["kind"]
    traj = s["traj"]
    if k == "pieces":
        S = rsv.rsv_action(ctx, s["h"], s["y"], s["lnrv"], THETA)
        F = rsv.rsv_force(ctx, s["h"], s["y"], s["lnrv"], THETA)
        th = s["theta"].clone()
        rsv.rsv_gibbs_theta(ctx, s["h"], s["lnrv"], th[0], seed=s["seed"], traj=traj)
        s["traj"] += 1
        return {"S": S, "F": F, "theta": th}
    if k == "chain":
        n = c["n_traj"]
        rsv.rsv_hmc_chain(ctx, s["h"], s["y"], s["lnrv"], s["theta"][0], c["n_md"], c["dtau"], n, prec=c["prec"],
                          minv=s.get("minv"), seed=s["seed"], traj0=traj, update_theta=c["theta"], dH_out=s["dH"],
                          accept_out=s["accept"], theta_out=s["theta_out"], snaps=s["snaps"])
        s["traj"] += n
        return {"h": s["h"], "theta": s["theta"], "accept": s["accept"], "dH": s["dH"], "theta_out": s["theta_out"],
                "snaps": s["snaps"]}
    if k == "trajectory":
        h, p = s["h"].clone(), s["p"].clone()
        dH, acc = rsv.rsv_hmc_trajectory(ctx, h, p, s["y"], s["lnrv"], THETA_LARGE, c["n_md"], c["dtau"], prec=c["prec"],
                                         log_u=s["log_u"])
        return {"h": h, "p": p, "dH": dH, "accept": acc}
    if k == "batched":
        n = c["n_traj"]
        rsv.rsv_hmc_batched(ctx, s["plan"], s["h"], s["y"], s["lnrv"], s["theta"], c["dtau"], minv=s.get("minv"),
                            seed=s["seed"], traj0=traj, n_traj=n, dH_out=s["dH"], accept_out=s["accept"])
        s["traj"] += n
        return {"h": s["h"], "dH": s["dH"], "accept": s["accept"]}
    if k == "mass":
        mean, m2 = torch.zeros_like(s["h"]), torch.zeros_like(s["h"])
        count = rsv.rsv_welford_update(ctx, s["snaps"], 0, mean, m2)
        tm = learned.train_mass(ctx, s["y"], s["lnrv"], THETA, mean, m2, count, steps=c["steps"], batch=c["batch"],
                                seed=s["seed"])
        return {"mean": mean, "m2": m2, "hbar": tm.hbar, "target": tm.target, "log_scale": tm.log_scale,
                "features": tm.features, "params": tm.params, "losses": tm.losses, "minv": tm.minv}
    return {"ess": rsv.rsv_ess(ctx, s["x"])}


def work(c):
    """Bytes: every input array once, every output once.  Flops: per site and force evaluation 11 (the force of eq. (7) 7
    with its exponential as one, the kick 2, the drift 2); per site of S 14, dS/dh 13, the theta sums 14."""
    k = c["kind"]
    if k == "pieces":
        return {"bytes": (24 + 32 + 16) * c["T"], "flops": 41 * c["T"]}
    if k == "chain":
        f = c["n_md"] * len(SCHEMES[c["integrator"]][1])
        b = 24 + 8 + (4 if c["mass"] else 0) + (4 * c["n_traj"] if c["snaps"] else 0)
        return {"bytes": b * c["T"] + 60 * c["n_traj"], "flops": 11 * c["T"] * f * c["n_traj"]}
    if k == "trajectory":
        return {"bytes": (24 + 8 + 16) * c["T"], "flops": 11 * c["T"] * c["n_md"]}
    if k == "batched":
        N = c["n"] * (c["T_lo"] + c["T_hi"]) // 2
        return {"bytes": (32 + (4 if c["mass"] else 0)) * N, "flops": 11 * N * c["n_md"] * c["n_traj"]}
    if k == "mass":
        net = 2 * (20 * 32 + 32 * 32 + 32)
        return {"bytes": (4 * c["rows"] + 16 + 8 + 4 + 16 + 80 + 4) * c["T"],
                "flops": (4 * c["rows"] + 60 + net) * c["T"] + 3 * net * c["batch"] * c["steps"]}
    # the lags a chain of this kind needs: about 16 pairs of the mean site
    return {"bytes": 4 * (c["n"] + 1) * c["T"], "flops": 2 * 32 * c["n"] * c["T"]}


# ---- the same in 64 bits -------------------------------------------------------------------------------------------


def _words(seed, series, traj, stream, blocks):
    """Philox4x64-10 words of counters {0 .. blocks-1, traj, stream, series}, key {seed, 0}.  numpy's generator
    advances its counter before each block."""
    c = (traj << 64) | (stream << 128) | (series << 192)
    c = (c - 1) % (1 << 256)
    ctr = [(c >> (64 * i)) & 0xFFFFFFFFFFFFFFFF for i in range(4)]
    return np.random.Philox(counter=np.array(ctr, dtype=np.uint64), key=np.array([seed, 0], dtype=np.uint64)).random_raw(4 * blocks)


def _uniform(w, bits):
    return ((w >> np.uint64(64 - bits)).astype(np.float64) + 0.5) * 2.0 ** -bits


def _normals(seed, series, traj, T, bits):
    u = torch.from_numpy(_uniform(_words(seed, series, traj, 0, (T + 3) // 4), bits)).cuda().view(-1, 2)
    r, a = (-2.0 * u[:, 0].log()).sqrt(), 2.0 * math.pi * u[:, 1]
    return torch.stack([r * a.cos(), r * a.sin()], 1).reshape(-1)[:T]


def _sweep(h, lnrv, th, seed, traj, bits):
    """One Gibbs sweep of theta (list of five floats) given one series' h."""
    u = _uniform(_words(seed, 0, traj, 2, 64), bits)
    at = [0]

    def uni():
        at[0] += 1
        return float(u[at[0] - 1])

    def normal():
        a, b = uni(), uni()
        return math.sqrt(-2.0 * math.log(a)) * math.cos(2.0 * math.pi * b)

    def gamma(alpha):
        if alpha < 1.0:
            return gamma(alpha + 1.0) * uni() ** (1.0 / alpha)
        d = alpha - 1.0 / 3.0
        c = 1.0 / math.sqrt(9.0 * d)
        while True:
            z = normal()
            v = 1.0 + c * z
            if v <= 0.0:
                continue
            x = c * z
            r = (3.0 * d * sum((-1) ** (k + 1) * x ** k / k for k in range(4, 40)) if abs(x) < 0.25  # the same, without cancellation
                 else 0.5 * z * z + d - d * v ** 3 + 3.0 * d * math.log(v))
            if math.log(uni()) < r:
                return d * v ** 3

    phi, mu, xi, se2, su2 = th
    T = h.numel()
    q = lnrv - xi - h
    x = h - mu
    e = x[1:] - phi * x[:-1]
    x0 = float(x[0])
    dxi = float(q.mean()) + math.sqrt(su2 / T) * normal()
    xi2 = xi + dxi
    su2 = 0.5 * float(((q - dxi) ** 2).sum()) / gamma(0.5 * T)
    den = (1.0 - phi * phi) + (T - 1) * (1.0 - phi) ** 2
    dmu = ((1.0 - phi * phi) * x0 + (1.0 - phi) * float(e.sum())) / den + normal() / math.sqrt(den / se2)
    x = x - dmu
    Q = (1.0 - phi * phi) * float(x[0]) ** 2 + float(((x[1:] - phi * x[:-1]) ** 2).sum())
    se2 = 0.5 * Q / gamma(0.5 * T)
    if T >= 3:
        D = float((x[1:-1] ** 2).sum())
        m, sd = float((x[1:] * x[:-1]).sum()) / D, math.sqrt(se2 / D)
        while True:
            prop = m + sd * normal()
            if -1.0 < prop < 1.0:
                break
        if math.log(uni()) < 0.5 * math.log1p(-prop * prop) - 0.5 * math.log1p(-phi * phi):
            phi = prop
    th = [phi, mu + dmu, xi2, se2, su2]
    return [float(np.float32(v)) for v in th] if bits == 23 else th


class _Model:
    """S and dS/dh of packed series in 64 bits (theta per site)."""

    def __init__(self, T, pos, y, lnrv, theta, rho):
        T = torch.as_tensor(T, device="cuda")
        self.T, self.y, self.lnrv, self.rho = T, y, lnrv, rho
        self.first, self.last = pos == 0, pos == torch.repeat_interleave(T, T) - 1
        self.sid = torch.repeat_interleave(torch.arange(len(T), device="cuda"), T)
        self.set_theta(theta)

    def set_theta(self, theta):
        one = len(self.T) == 1
        get = (lambda k: theta[0, k]) if one else (lambda k: torch.repeat_interleave(theta[:, k].contiguous(), self.T))
        self.phi, self.mu, self.xi, self.se2, self.su2 = (get(k) for k in range(5))
        self.B = 1.0 / (self.se2 * (1.0 - self.rho ** 2))

    def _parts(self, h):
        x = h - self.mu
        eps = self.y * torch.exp(-0.5 * h)
        rs = self.rho * torch.as_tensor(self.se2, device="cuda").sqrt()
        nxt = torch.cat([x[1:], x[:1]])
        d = torch.where(self.last, torch.zeros_like(x), nxt - self.phi * x - rs * eps)
        return x, eps, rs, d

    def sites(self, h):
        x, eps, _, d = self._parts(h)
        s = 0.5 * h + 0.5 * eps * eps + (self.lnrv - self.xi - h) ** 2 / (2.0 * self.su2) + 0.5 * self.B * d * d
        return s + torch.where(self.first, (1.0 - self.phi ** 2) * x * x / (2.0 * self.se2), torch.zeros_like(x))

    def force(self, h):
        x, eps, rs, d = self._parts(h)
        prev = torch.cat([d[-1:], d[:-1]])
        left = torch.where(self.first, (1.0 - self.phi ** 2) * x / self.se2, self.B * prev)
        return 0.5 - 0.5 * eps * eps - (self.lnrv - self.xi - h) / self.su2 + left + self.B * d * (0.5 * rs * eps - self.phi)

    def per_series(self, v):
        if len(self.T) == 1:
            return v.sum().reshape(1)
        return torch.zeros(len(self.T), dtype=torch.float64, device="cuda").index_add_(0, self.sid, v)

    def trajectory(self, h, p, minv, scheme, n_md, dtau):
        """(h', p', dH per series)"""
        a, b = SCHEMES[scheme]
        w = 1.0 if minv is None else minv
        h1, p1 = h.clone(), p.clone()
        for _ in range(n_md):
            h1 = h1 + a[0] * dtau * w * p1
            for i, kick in enumerate(b):
                p1 = p1 - kick * dtau * self.force(h1)
                h1 = h1 + a[i + 1] * dtau * w * p1
        dH = self.per_series(self.sites(h1) - self.sites(h) + 0.5 * w * (p1 - p) * (p1 + p))
        return h1, p1, dH


def exact(case, seed):
    c, k = case, case["kind"]
    s = _inputs(c, seed)
    if k == "ess":
        return {"ess": _exact_ess(s["x"].double())}
    if k == "mass":
        return _exact_mass(c, s)
    M = _Model(s["T"], s["pos"], s["y"], s["lnrv"], s["theta"], c.get("rho", 0.0))
    h = s["h"]
    if k == "pieces":
        th = _sweep(h, s["lnrv"], list(THETA), s["seed"], 0, 53)
        return {"S": M.sites(h).sum().reshape(1), "F": M.force(h), "theta": torch.tensor([th], dtype=torch.float64)}
    if k == "trajectory":
        h1, p1, dH = M.trajectory(h, s["p"], None, "leapfrog", c["n_md"], c["dtau"])
        take = bool(s["log_u"][0] < -dH[0])
        return {"h": h1 if take else h, "p": p1, "dH": dH, "accept": None}
    bits = 53 if c["prec"] == "fp64" else 23
    minv = s["minv"].double() if c.get("mass") else None
    theta, n = s["theta"], c["n_traj"]
    dHs, thetas = [], []
    snaps = torch.empty(n, c["T"], dtype=torch.float64, device="cuda") if c.get("snaps") else None
    for i in range(n):
        p = torch.cat([_normals(s["seed"], j, i, int(T), bits) for j, T in enumerate(s["T"])])
        if minv is not None:
            p = p / minv.sqrt()
        h1, _, dH = M.trajectory(h, p, minv, c.get("integrator", "leapfrog"), c["n_md"], c["dtau"])
        lu = np.log([_uniform(_words(s["seed"], j, i, 1, 1), 53)[0] for j in range(len(s["T"]))])
        take = torch.from_numpy(lu).cuda() < -dH
        h = torch.where(take[M.sid] if len(s["T"]) > 1 else take, h1, h)
        dHs.append(dH)
        if c.get("theta"):
            theta = torch.tensor([_sweep(h, s["lnrv"], theta[0].tolist(), s["seed"], i, bits)], dtype=torch.float64, device="cuda")
            M.set_theta(theta)
            thetas.append(theta[0])
        if snaps is not None:
            snaps[i] = h
    if k == "batched":
        return {"h": h, "dH": torch.stack(dHs), "accept": None}
    return {"h": h, "theta": theta, "accept": None, "dH": torch.cat(dHs) if c["prec"] == "fp64" else None,
            "theta_out": torch.stack(thetas) if thetas else None, "snaps": snaps}


def _exact_ess(x):
    """Geyer's initial monotone sequence estimator of every column."""
    n, T = x.shape
    x = x - x.mean(0)

    def gamma(lag):
        return (x[: n - lag] * x[lag:]).sum(0) / n

    g0 = gamma(0)
    go, prev = g0 > 0, torch.full((T,), math.inf, dtype=x.dtype, device=x.device)
    tau = torch.zeros(T, dtype=x.dtype, device=x.device)
    m = 0
    while 2 * m + 1 < n and bool(go.any()):
        G = ((gamma(2 * m) if m else g0) + gamma(2 * m + 1)) / g0
        go = go & (G > 0)
        prev = torch.where(go, torch.minimum(G, prev), prev)
        tau += torch.where(go, prev, torch.zeros_like(prev))
        m += 1
    tau = torch.clamp(-1.0 + 2.0 * tau, min=1.0 / math.log10(max(n, 10)))
    return torch.where(g0 > 0, n / tau, torch.zeros_like(tau))


def _exact_mass(c, s):
    """Moments, target and features; the network's own results depend on its BF16 arithmetic and have no such value."""
    x = s["snaps"].double()
    mean = x.mean(0)
    m2 = ((x - mean) ** 2).sum(0)
    target = -(m2 / (c["rows"] - 1)).log()
    phi, mu, xi, se2, su2 = THETA
    T, y = c["T"], s["y"]
    pad = torch.nn.functional.pad(mean, (4, 4))
    t = torch.arange(T, device="cuda")
    edge = torch.exp2(-torch.minimum(torch.minimum(t, T - 1 - t), torch.tensor(64, device="cuda")).double())
    const = [phi, mu, xi, se2, su2]
    cols = [y * y, s["lnrv"]] + [pad[i: i + T] for i in range(9)] + [torch.full_like(y, v) for v in const]
    cols += [edge, torch.full_like(y, (1.0 + phi * phi) / se2), torch.full_like(y, 1.0 / su2), 0.5 * y * y * torch.exp(-mean)]
    F = torch.stack(cols, 1)
    m = F.mean(0)
    sd = ((F - m) ** 2).mean(0).sqrt()
    inv = torch.where(sd > 1e-12 * torch.clamp(m.abs(), min=1.0), 1.0 / sd, torch.zeros_like(sd))
    m[16], inv[16] = 0.0, 1.0
    return {"mean": mean, "m2": m2, "hbar": mean, "target": target, "log_scale": target.mean().reshape(1),
            "features": torch.clamp((F - m) * inv, -8.0, 8.0), "params": None, "losses": None, "minv": None}
