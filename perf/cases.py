"""What is measured: the work a user of this library has it do, through its Python entry points.

One case is one call (or one short sequence of calls) of a host program: a hydro code that hands its zones to the
integrator and takes abundances back, an operator-split loop, the training of the step proposal.  Networks and zone
recipes are those of `kn_inputs` (the 16/48 chain, the 150/1604 and 365/4400 networks, the size sweep's networks between
them); zone conditions and records are drawn from the seed.
"""
import math

import numpy as np
import torch

from kn_inputs import (binding_energies, chain_network, mixed_assignment, net150, net365, profile_zones, sweep_network)
from paper_1409_5826_gb300 import kn, learned, opsplit

PREC = {"mixed": kn.PREC_MIXED, "fp64": kn.PREC_FP64, "mixed_fp64": kn.PREC_MIXED_FP64}
ZONE_ARRAYS = ("Y0", "T0", "rho0", "tau", "t_start", "t_end", "dt_trial")
_NETS = {}


def listed():
    return [
        # One cell of a hydro code, the smallest network, host arrays in and out: the call's latency counts.
        dict(name="cell_chain", path="cell", species=16, zones=1, precision="mixed", t_end=1e-11),
        # The single 150-species zone in the strict FP64 form (the paper's own setting).
        dict(name="cell_150_fp64", path="cell", species=150, zones=1, precision="fp64", t_end=1e-11),
        # An operator-split loop over a small patch: 100 cells (fewer than the SMs), four hydro intervals, energy release.
        dict(name="split_150", path="split", species=150, zones=100, intervals=4, precision="mixed", t_end=1e-11),
        # The headline batch: 4096 profiled zones of 150/1604, device arrays, one captured launch.
        dict(name="batch_150", path="batch", species=150, zones=4096, precision="mixed", t_end=1e-9),
        # The same network in the two forms with FP64 in the step: the strict one, and FP32 fluxes with an FP64 update.
        dict(name="batch_150_fp64", path="batch", species=150, zones=2048, precision="fp64", t_end=3e-11),
        dict(name="batch_150_mixed_fp64", path="batch", species=150, zones=1024, precision="mixed_fp64", t_end=1e-10),
        # The largest network, a ragged zone count.
        dict(name="batch_365", path="batch", species=365, zones=1000, precision="mixed", t_end=1e-10),
        # Many cells of the smallest network over its own long interval (rates refreshed along the profile).
        dict(name="batch_chain", path="batch", species=16, zones=8001, precision="mixed", t_end=1e-3),
        # The alpha-QSS update where it is the better one: the chain to the end of its interval.
        dict(name="qss_chain", path="qss", species=16, zones=4096, precision="mixed", t_end=1e-2),
        # Zones of three network sizes in one launch, 1:2:1 (a hydro grid with adaptive networks).
        dict(name="uneven", path="uneven", zones=2048, precision="mixed", t_end=1e-9),
        # The integrator with the learned step proposal.
        dict(name="learned_150", path="learned", species=150, zones=512, precision="mixed", t_end=3e-11),
        # Training that proposal: forward, backward and Adam over 16 batches of 4096 records.
        dict(name="train", path="train", batch=4096, steps=16),
    ]


def draw(rng):
    def logu(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    def zones(lo, hi):
        return int(round(logu(lo, hi)))

    path = rng.choice(["cell", "split", "batch", "batch", "batch", "batch", "qss", "uneven", "learned", "train"])
    if path == "cell":
        return dict(path=path, species=rng.choice([16, 32, 64, 100, 150]), zones=zones(1, 40),
                    precision=rng.choice(["mixed", "mixed", "fp64"]), t_end=logu(3e-12, 3e-11))
    if path == "split":
        return dict(path=path, species=rng.choice([16, 64, 150]), zones=zones(10, 600), intervals=rng.randint(2, 5),
                    precision="mixed", t_end=logu(3e-12, 3e-11))
    if path == "qss":
        return dict(path=path, species=16, zones=zones(500, 4096), precision=rng.choice(["mixed", "mixed", "fp64"]),
                    t_end=logu(1e-5, 1e-2))
    if path == "uneven":
        return dict(path=path, zones=zones(200, 2048), precision="mixed", t_end=logu(1e-11, 3e-10))
    if path == "learned":
        return dict(path=path, species=rng.choice([100, 150]), zones=zones(50, 1000), precision="mixed",
                    t_end=logu(3e-12, 3e-11))
    if path == "train":
        return dict(path=path, batch=zones(512, 8192), steps=rng.randint(4, 24))
    species = rng.choice([16, 32, 64, 100, 150, 150, 250, 365])
    precision = rng.choice(["mixed", "mixed", "mixed", "fp64", "mixed_fp64"])
    if species == 16:
        return dict(path="batch", species=16, zones=zones(500, 8000), precision=precision, t_end=logu(1e-6, 2e-3))
    if precision == "fp64":
        return dict(path="batch", species=species, zones=zones(100, 1000), precision=precision, t_end=logu(3e-12, 2e-11))
    return dict(path="batch", species=species, zones=zones(200, 2500), precision=precision, t_end=logu(1e-11, 1e-10))


def _net(species):
    if species not in _NETS:
        _NETS[species] = {16: chain_network, 150: net150, 365: net365}.get(species, lambda: sweep_network(species))()
    return _NETS[species]


def _opts(case, **more):
    return kn.Opts(precision=PREC[case["precision"]], **more)


def _zones(net, n, seed, t_end):
    return profile_zones(net, n, base_seed=1000 + 10007 * seed, t_end=t_end)


def _on_gpu(z):
    return {k: torch.from_numpy(np.ascontiguousarray(getattr(z, k))).cuda() for k in ZONE_ARRAYS}


def _results(n_zones, n_species):
    d = dict(device="cuda")
    return dict(Y=torch.empty((n_zones, n_species), dtype=torch.float64, **d),
                t=torch.empty(n_zones, dtype=torch.float64, **d), dt_next=torch.empty(n_zones, dtype=torch.float64, **d),
                steps=torch.empty(n_zones, dtype=torch.int64, **d), rejects=torch.empty(n_zones, dtype=torch.int64, **d),
                status=torch.empty(n_zones, dtype=torch.int32, **d))


def _split_schedule(case, z, seed):
    """Per hydro interval: T9 and rho held constant along each zone's profile, ends evenly spaced in log t."""
    n, ends = case["intervals"], []
    for k in range(n):
        ends.append(1e-12 * (case["t_end"] / 1e-12) ** ((k + 1) / n))
    rng = np.random.default_rng(seed)
    out = []
    for k, te in enumerate(ends):
        cool = 1.0 - 0.02 * k * rng.uniform(0.5, 1.5, z.n_zones)
        out.append((z.T0 * cool, z.rho0 * cool ** 3, np.full(z.n_zones, te)))
    return out


def _proposal(seed):
    """A step-proposal network and its feature normalisation: He-uniform weights, an output near the steps that the
    controller takes by itself (ln 1.5, plus the margin), so that some proposals exceed them and some do not."""
    p = learned.init_params(seed)
    d = kn.mlp_unpack(p)
    d["W3"], d["b3"] = 0.3 * d["W3"], d["b3"] + 0.9
    mu = np.concatenate([[1.4, 18.4, -32.0, 0.3], np.full(20, -9.0), np.full(20, 2.0), np.full(20, 2.0)])
    sd = np.concatenate([[0.4, 1.3, 4.0, 0.2], np.full(20, 6.0), np.full(20, 8.0), np.full(20, 8.0)])
    return kn.mlp_pack(d), mu.astype(np.float32), sd.astype(np.float32)


def _records(case, seed):
    """Training records: features around the ranges the integrator writes, labels ln(dt_best / dt_prev) in the grid's
    range with a smooth dependence on the features."""
    rng = np.random.default_rng(seed)
    n = case["batch"] * case["steps"]
    x = rng.standard_normal((n, kn.MLP_FEATURES)).astype(np.float32)
    y = np.clip(0.4 + 0.3 * x[:, 2] - 0.2 * x[:, 3] * x[:, 0] + 0.1 * rng.standard_normal(n), -1.386, 2.773)
    mu = rng.uniform(-5, 5, kn.MLP_FEATURES).astype(np.float32)
    sd = rng.uniform(0.5, 6, kn.MLP_FEATURES).astype(np.float32)
    return mu + sd * x, y.astype(np.float32), mu, sd, learned.init_params(seed + 1)


def prepare(case, seed):
    path = case["path"]
    s = {"path": path}
    if path == "train":
        x, y, mu, sd, p = _records(case, seed)
        s.update(mlp=kn.MLP(), params=p, mu=mu, sd=sd, x=torch.from_numpy(x).cuda().split(case["batch"]),
                 y=torch.from_numpy(y).cuda().split(case["batch"]),
                 loss=torch.zeros(case["steps"], dtype=torch.float32, device="cuda"))
        return s
    if path == "uneven":
        lab = mixed_assignment(case["zones"], seed=seed)
        s.update(opts=_opts(case, use_graph=1), nets=[], zones=[], out=[])
        for k, species in enumerate((16, 150, 365)):
            net = _net(species)
            z = _zones(net, case["zones"], seed, 1e-2 if species == 16 else case["t_end"]).subset(np.nonzero(lab == k)[0])
            s["nets"].append(kn.Network(net))
            s["zones"].append(_on_gpu(z))
            s["out"].append(_results(z.n_zones, net.n_species))
        return s
    net = _net(case["species"])
    z = _zones(net, case["zones"], seed, case["t_end"])
    s["net"] = kn.Network(net)
    if path == "cell":
        z.tau[:] = 0.0  # the conditions of one hydro step: constant
        s.update(zones=z, opts=_opts(case))
    elif path == "split":
        s.update(zones=z, opts=_opts(case), schedule=_split_schedule(case, z, seed))
        s["net"].set_binding_energies(binding_energies(net))
    else:
        more = dict(use_graph=1)
        if path == "qss":
            more.update(method=kn.METHOD_QSS)
        if path == "learned":
            s["mlp"] = kn.MLP()
            s["mlp"].set_params(*_proposal(seed))
            more.update(mlp=s["mlp"])
        s.update(zones=_on_gpu(z), out=_results(z.n_zones, net.n_species), opts=_opts(case, **more))
    return s


def run(s):
    path = s["path"]
    if path == "train":
        s["mlp"].set_params(s["params"], s["mu"], s["sd"])
        for i, (x, y) in enumerate(zip(s["x"], s["y"])):
            s["mlp"].backward(x, y, s["loss"][i:i + 1])
            s["mlp"].adam(1e-3)
        params, grads = s["mlp"].get_params()
        return {"params": params, "grads": grads, "loss": s["loss"]}
    if path == "cell":
        s["net"].set_zones(s["zones"])
        kn.integrate_batch([s["net"]], s["opts"])
        return s["net"].get()
    if path == "split":
        return opsplit.run(s["net"], s["zones"], s["schedule"], s["opts"])
    if path == "uneven":
        for net, z in zip(s["nets"], s["zones"]):
            net.set_zones(z)
        kn.integrate_batch(s["nets"], s["opts"])
        return [net.get_device(o) for net, o in zip(s["nets"], s["out"])]
    s["net"].set_zones(s["zones"])
    kn.integrate_batch([s["net"]], s["opts"])
    return s["net"].get_device(s["out"])


# Mean accepted steps per zone of the profiled recipe to t_end, from FP64 runs of the method: (t_end, steps) per network
# size; read off on log axes (the networks between take the 150-species curve).
_STEPS = {16: ((1e-12, 10), (1e-11, 700), (1e-9, 1510), (1e-7, 2080), (1e-5, 2350), (1e-4, 2750), (1e-3, 4610), (1e-2, 23100)),
          150: ((1e-12, 10), (1e-11, 1800), (3e-11, 2240), (1e-10, 4940), (3e-10, 22900), (1e-9, 42000)),
          365: ((1e-12, 10), (1e-11, 1530), (3e-11, 2270), (1e-10, 3200), (3e-10, 5310), (1e-9, 20000))}


def _steps(species, t_end, qss):
    curve = _STEPS.get(species, _STEPS[150])
    x = np.interp(math.log(t_end), [math.log(a) for a, _ in curve], [math.log(b) for _, b in curve])
    return math.exp(x) * (0.3 if qss and species == 16 and t_end > 1e-3 else 1.0)


def _zone_work(species, zones, t_end, qss=False):
    """Zone arrays in and out once; per step a rate factor (2 operations) per reaction, the fluxes and partials of r
    reactants (about r^2 products), the gathers' additions, and about 15 operations per species for the update and the
    accept test; the QSS update evaluates the right-hand side twice."""
    net = _net(species)
    r = net.n_reac.astype(int)
    s_r, s_p = net.slot_counts()
    rhs = 2 * len(r) + int((r * r).sum()) + s_r + s_p
    step = (2 if qss else 1) * rhs + (40 if qss else 15) * net.n_species
    return {"bytes": zones * (16 * net.n_species + 6 * 8 + 36), "flops": zones * _steps(species, t_end, qss) * step}


def work(case):
    path = case["path"]
    if path == "train":
        rows = case["batch"] * case["steps"]
        f, h = kn.MLP_FEATURES, kn.MLP_HIDDEN
        return {"bytes": 4 * rows * (f + 1) + 8 * kn.MLP_PARAMS, "flops": rows * 2 * (2 * f * h + 3 * h * h + 3 * h)}
    if path == "uneven":
        z = case["zones"]
        parts = [_zone_work(16, z // 4, 1e-2), _zone_work(150, z // 2, case["t_end"]), _zone_work(365, z // 4, case["t_end"])]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    return _zone_work(case["species"], case["zones"], case["t_end"], path == "qss")


# ---------------------------------------------------------------------------
# 64-bit values, from plain torch
# ---------------------------------------------------------------------------
def _integrate64(net, Y, T0, rho0, tau, t, t_end, dt, kappa=1.0, eps_r=0.05, eps_c=1e-6, y_min=1e-10):
    """Eq. 1 and Eq. 3 with the kappa switch and the adaptive step, every zone in step with the others; torch float64."""
    dev = Y.device
    N, R = net.n_species, net.n_reactions
    reac = np.where(net.reac < 0, N, net.reac)
    idx = [torch.from_numpy(reac[:, q].astype(np.int64)).to(dev) for q in range(3)]
    has = [torch.from_numpy((net.reac[:, q] >= 0).astype(np.float64)).to(dev) for q in range(3)]
    into = np.zeros((R, N))
    out = np.zeros((3, R, N))
    for q in range(3):
        ok = net.prod[:, q] >= 0
        np.add.at(into, (np.nonzero(ok)[0], net.prod[ok, q]), 1.0)
        ok = net.reac[:, q] >= 0
        out[q][np.nonzero(ok)[0], net.reac[ok, q]] = 1.0
    into = torch.from_numpy(into).to(dev)
    out = [torch.from_numpy(o).to(dev) for o in out]
    A = torch.from_numpy(net.A).to(dev)
    lnk = torch.from_numpy(net.ln_k0).to(dev)
    n = torch.from_numpy(net.t9_exp).to(dev)
    nr = torch.from_numpy((net.reac >= 0).sum(1).astype(np.float64)).to(dev)
    K = torch.exp(lnk + n * torch.log(T0)[:, None] + (nr - 1) * torch.log(rho0)[:, None])
    c = n + 3 * (nr - 1)
    inv_tau = torch.where(tau > 0, 1 / tau, torch.zeros_like(tau))
    one = torch.ones((Y.shape[0], 1), dtype=torch.float64, device=dev)
    left = 60000
    for _ in range(left):
        live = t < t_end
        if _ % 16 == 0 and not bool(live.any()):
            break
        k = K * torch.exp(-c * (t * inv_tau)[:, None])
        Yx = torch.cat([Y, one], 1)
        y = [Yx[:, i] for i in idx]
        Fp = (k * y[0] * y[1] * y[2]) @ into
        kk = (k * y[1] * y[2] * has[0]) @ out[0] + (k * y[0] * y[2] * has[1]) @ out[1] + (k * y[0] * y[1] * has[2]) @ out[2]
        clip = dt >= t_end - t
        h = torch.where(clip, t_end - t, dt)
        kh = kk * h[:, None]
        Yn = torch.where(kh >= kappa, (Y + h[:, None] * Fp) / (1 + kh), Y + h[:, None] * (Fp - kk * Y))
        cons = ((Yn - Y) @ A).abs()
        m = torch.maximum(Y, Yn)
        rel = torch.where(m > y_min, (Yn - Y).abs() / m, torch.zeros_like(m)).amax(1)
        ok = (cons <= eps_c) & (rel <= eps_r)
        go, no = live & ok, live & ~ok
        grow = torch.clamp(torch.minimum(0.9 * eps_r / rel.clamp_min(1e-300), 0.9 * eps_c / cons.clamp_min(1e-300)), max=1.5)
        Y = torch.where(go[:, None], Yn, Y)
        t = torch.where(go, torch.where(clip, t_end, t + h), t)
        dt = torch.where(go, h * grow, torch.where(no, 0.5 * h, dt))
    return Y, t, dt


def _exact_train(case, seed):
    x, y, mu, sd, p0 = _records(case, seed)
    x = torch.from_numpy(((x.astype(np.float64) - mu) / sd)).cuda()
    y = torch.from_numpy(y.astype(np.float64)).cuda()
    f, h = kn.MLP_FEATURES, kn.MLP_HIDDEN
    p = torch.from_numpy(p0.astype(np.float64)).cuda().requires_grad_(True)
    m, v, losses, g = torch.zeros_like(p), torch.zeros_like(p), [], None
    for i in range(case["steps"]):
        w1, b1, w2, b2, w3, b3 = p.split([f * h, h, h * h, h, h, 1])
        rows = slice(i * case["batch"], (i + 1) * case["batch"])
        a = torch.relu(x[rows] @ w1.view(f, h) + b1)
        a = torch.relu(a @ w2.view(h, h) + b2)
        loss = ((a @ w3 + b3 - y[rows]) ** 2).mean()
        g, = torch.autograd.grad(loss, p)
        losses.append(loss.detach())
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        q = p.detach() - 1e-3 * (m / (1 - 0.9 ** (i + 1))) / (torch.sqrt(v / (1 - 0.999 ** (i + 1))) + 1e-8)
        p = q.requires_grad_(True)
    return {"params": p.detach().cpu().numpy(), "grads": g.cpu().numpy(), "loss": torch.stack(losses)}


def exact(case, seed):
    """Abundances and times in 64 bits for the cells and the split intervals.  The long batches have none: their zones
    take up to 10^5 steps one after another, and two valid runs part at the first step that one accepts and the other
    rejects; the step counts, the next step, which is as sensitive, and the energy release, a difference that cancels,
    have none either."""
    path = case["path"]
    if path == "train":
        return _exact_train(case, seed)
    if path not in ("cell", "split"):
        return None
    net = _net(case["species"])
    z = _zones(net, case["zones"], seed, case["t_end"])
    d = _on_gpu(z)
    blank = dict(dt_next=None, steps=None, rejects=None, status=None)
    if path == "cell":
        Y, t, _ = _integrate64(net, d["Y0"], d["T0"], d["rho0"], 0 * d["tau"], d["t_start"], d["t_end"], d["dt_trial"])
        return dict(Y=Y.cpu().numpy(), t=t.cpu().numpy(), **blank)
    Y, t, dt, out = d["Y0"], d["t_start"], d["dt_trial"], []
    for T9, rho, te in _split_schedule(case, z, seed):
        T9, rho, te = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (T9, rho, te))
        Y, t, dt = _integrate64(net, Y, T9, rho, 0 * T9, t, te, dt)
        out.append(dict(Y=Y.cpu().numpy(), t=t.cpu().numpy(), energy=None, **blank))
    return out
