"""FP64 form: the rate factors formed in integers, and the accept test that forms the
exact largest ratio only where it matters, against the same values in FP64
arithmetic, bit for bit (tolerance zero)."""
from fractions import Fraction

import numpy as np
import pytest

from kn_inputs import (Zones, chain_network, custom_network, net150, pair_network, profile_zones,
                       sweep_network)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kn():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_5826_gb300 import build, kn as knmod
    build.build()
    return knmod


def _fma(a, b, c):
    return float(Fraction(float(a)) * Fraction(float(b)) + Fraction(float(c)))  # rounds to nearest even


def test_rate_factors_are_the_fp64_ones(kn):
    # one decay a species, so k_i is its rate: K_j at s = 0, K_j (1 - x + x^2/2) later.
    # Exponents in and around the integer form's range, zero and negative ones; s from
    # the smallest to both sides of the largest that it takes.
    rng = np.random.default_rng(3)
    c = np.concatenate([[0.0, -2.0, 2.0 ** -20, 2.0 ** -21, 0.3, 1.0, 1.5, 3.0, 31.75], rng.uniform(1e-3, 32, 54), [32.0]])
    n = len(c)
    net = custom_network([1.0] * (n + 1), [((i,), (n,)) for i in range(n)], rng.uniform(-3, 3, n), c)
    t = np.concatenate([[1e-25, 1e-18, 1e-12, 4.6e-7 / 32, 4.6999e-7 / 32, 4.7001e-7 / 32, 9e-7 / 32],
                        10.0 ** rng.uniform(-17, -7.84, 57)])
    Z = len(t)
    f = lambda v: np.broadcast_to(np.asarray(v, float), (Z,)).copy()
    Y = np.full((Z, n + 1), 1.0 / (n + 1))
    k = []
    for tau in (0.0, 1.0):
        g = kn.Network(net)
        g.set_zones(Zones(Y0=Y, T0=f(3.0), rho0=f(1e8), tau=f(tau), t_start=t, t_end=f(1.0), dt_trial=f(1e-9)))
        k.append(g.probe(kn.Opts(precision=kn.PREC_FP64))["k"][:, :n])
        g.close()
    for z in range(Z):
        for j in range(n):
            x = float(c[j]) * float(t[z])
            fac = _fma(x, _fma(x, 0.5, -1.0), 1.0)
            assert k[1][z, j] == k[0][z, j] * fac, (z, j, c[j], t[z])


def _twins(net):
    """Two copies of a network side by side: every largest ratio is shared by two species."""
    n = net.n_species
    two = []
    for o in (0, n):
        for r, p in zip(net.reac, net.prod):
            two.append((tuple(int(i) + o for i in r if i >= 0), tuple(int(i) + o for i in p if i >= 0)))
    return custom_network(np.concatenate([net.A, net.A]), two, np.concatenate([net.ln_k0] * 2),
                          np.concatenate([net.t9_exp] * 2))


@pytest.mark.parametrize("method", [0, 1])
@pytest.mark.parametrize("name", ["chain", "twins", "sweep", "150"])
def test_accept_test_bits(kn, name, method):
    # y_min on both sides of the limit below which the ratios are compared in FP64:
    # no abundance lies between the two, so the same decisions and steps
    base = {"chain": chain_network, "twins": chain_network, "sweep": lambda: sweep_network(64), "150": net150}[name]()
    z = profile_zones(base, 13, base_seed=5, t_end=3e-11)
    net = base
    if name == "twins":
        net = _twins(base)
        z = Zones(Y0=np.concatenate([z.Y0, z.Y0], 1) / 2, T0=z.T0, rho0=z.rho0, tau=z.tau, t_start=z.t_start,
                  t_end=z.t_end, dt_trial=z.dt_trial)
    out = []
    for y_min in (0.9e-250, 1.1e-250, 1e-10):
        g = kn.Network(net)
        g.set_zones(z)
        kn.integrate_batch([g], kn.Opts(precision=kn.PREC_FP64, y_min=y_min, max_steps=3000, method=method))
        out.append(g.get())
        g.close()
    for k in ("Y", "t", "dt_next", "steps", "rejects", "status"):
        assert np.array_equal(out[0][k], out[1][k]), k
    assert (out[2]["steps"] > 0).all()
    # and the ratios that end a step in the reject limit, with growth far beyond the safe step
    r = []
    for y_min in (0.9e-250, 1.1e-250):
        g = kn.Network(net)
        g.set_zones(z)
        kn.integrate_batch([g], kn.Opts(precision=kn.PREC_FP64, y_min=y_min, max_steps=300, max_reject=1, grow_max=1e6,
                                        safety=3.0, method=method))
        r.append(g.get())
        g.close()
    for k in ("Y", "t", "dt_next", "steps", "rejects", "status"):
        assert np.array_equal(r[0][k], r[1][k]), k


@pytest.mark.parametrize("zones", [1, 5, 153, 311])
@pytest.mark.parametrize("prec", [0, 2])
@pytest.mark.parametrize("species,G", [(40, 128), (130, 160), (150, 160), (300, 320)])
def test_few_zones_keep_their_bits(kn, species, G, prec, zones):
    # the chosen tiling spreads few zones over the SMs and widens the FP64 form's groups;
    # an explicit one of the same summation order does neither
    net = net150() if species == 150 else sweep_network(species)
    z = profile_zones(net, zones, base_seed=6, t_end=3e-12)
    out = []
    for tiling in ({}, {"threads_per_zone": G, "threads_per_cta": G}):
        g = kn.Network(net)
        g.set_zones(z)
        kn.integrate_batch([g], kn.Opts(precision=prec, max_steps=400, **tiling))
        out.append(g.get())
        g.close()
    for k in ("Y", "t", "dt_next", "steps", "rejects", "status"):
        assert np.array_equal(out[0][k], out[1][k]), k


@pytest.mark.parametrize("zones", [(1, 1), (2, 700), (310, 3), (0, 160)])
@pytest.mark.parametrize("prec", [0, 2])
def test_several_networks_keep_their_bits(kn, prec, zones):
    # the CTAs' first zones are dealt, the others come from the queues
    opts = kn.Opts(precision=prec, threads_per_zone=160, threads_per_cta=160, max_steps=300)
    nets = [n for n, Z in zip((chain_network(), net150()), zones) if Z]
    zs = [profile_zones(n, Z, base_seed=8, t_end=3e-12) for n, Z in zip(nets, [Z for Z in zones if Z])]
    gs = [kn.Network(n) for n in nets]
    for g, z in zip(gs, zs):
        g.set_zones(z)
    kn.integrate_batch(gs, opts)
    for net, g, z in zip(nets, gs, zs):
        one = kn.Network(net)
        one.set_zones(z)
        kn.integrate_batch([one], opts)
        a, b = g.get(), one.get()
        for k in ("Y", "t", "dt_next", "steps", "rejects", "status"):
            assert np.array_equal(a[k], b[k]), k
        assert (a["steps"] > 0).all()
        g.close()
        one.close()


@pytest.mark.parametrize("prec", [1, 2])
def test_rates_without_temperature_dependence(kn, prec):
    # every rate exponent 0: the cached rates never go stale, and the first pass still forms
    # them.  Another network's values are left in shared memory first.
    z = profile_zones(net150(), 300, base_seed=9, t_end=3e-12)
    g = kn.Network(net150())
    g.set_zones(z)
    kn.integrate_batch([g], kn.Opts(precision=prec, max_steps=50, threads_per_zone=160, threads_per_cta=160))
    g.close()
    net = pair_network(2.0, 1.0)
    f = lambda v: np.full(300, float(v))
    z = Zones(Y0=np.tile([0.9, 0.1], (300, 1)), T0=f(1), rho0=f(1), tau=f(2), t_start=f(0.1), t_end=f(1), dt_trial=f(1e-3))
    out = []
    for p in (0, prec):
        g = kn.Network(net)
        g.set_zones(z)
        kn.integrate_batch([g], kn.Opts(precision=p, max_steps=100000))
        out.append(g.get())
        g.close()
    assert np.array_equal(out[0]["steps"], out[1]["steps"])
    assert np.allclose(out[0]["Y"], out[1]["Y"], rtol=1e-4, atol=0)  # the forms' bar for equal steps
