"""The mixed form's kernel with several zones per thread group against the group
kernel, bit for bit: kn_integrate_batch runs the first, kn_integrate_noalloc the
second, on the same zones with the same summation order (threads_per_zone).  Both
take the same additions in the same order, so the tolerance is zero.

Sizes at the edges of the first one's choices: one zone, one and two zones an SM,
an odd zone left in a pair, more zones than slots; networks of one warp, of one
and of several species warps, with and without cached rates; constant and profiled
conditions; both updates; and networks that only the group kernel can take."""
import ctypes as C

import numpy as np
import pytest

from kn_inputs import (Zones, chain_network, constant_zones, custom_network, net150, net365, profile_zones,
                       random_tiny_network, sweep_network)

pytestmark = pytest.mark.gpu
IN = ("Y0", "T0", "rho0", "tau", "t_start", "t_end", "dt_trial")
OUT = ("Y", "t", "dt_next", "steps", "rejects", "status")


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_5826_gb300 import build, kn
    build.build()
    return torch, kn


def _both(env, net, z, G, **more):
    torch, kn = env
    opts = kn.Opts(precision=kn.PREC_MIXED, threads_per_zone=G, threads_per_cta=G, max_steps=20000, **more)
    g = kn.Network(net)
    dz = {k: torch.from_numpy(np.ascontiguousarray(getattr(z, k))).cuda() for k in IN}
    g.set_zones(dz)
    kn.integrate_batch([g], opts)
    a = g.get()
    Z, N = z.n_zones, net.n_species
    f64 = dict(dtype=torch.float64, device="cuda")
    out = {"Y": torch.empty((Z, N), **f64), "t": torch.empty(Z, **f64), "dt_next": torch.empty(Z, **f64),
           "steps": torch.empty(Z, dtype=torch.int64, device="cuda"),
           "rejects": torch.empty(Z, dtype=torch.int64, device="cuda"),
           "status": torch.empty(Z, dtype=torch.int32, device="cuda")}
    zc = kn._Zones(*[dz[k].data_ptr() for k in IN])
    rc = kn.lib().kn_integrate_noalloc(g.h, Z, C.byref(zc), C.byref(opts.c()), *[out[k].data_ptr() for k in OUT],
                                       C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == kn.KN_OK, kn.lib().kn_last_error()
    torch.cuda.synchronize()
    b = {k: v.cpu().numpy() for k, v in out.items()}
    g.close()
    for k in OUT:
        x, y = (v.view(np.int64) if v.dtype == np.float64 else v for v in (a[k], b[k]))  # an invalid zone's NaN too
        assert np.array_equal(x, y), (k, np.nonzero(x != y))
    return a


@pytest.mark.parametrize("net,G,zones,t_end", [
    (chain_network, 32, 1, 1e-9), (chain_network, 32, 5001, 1e-6),
    (lambda: sweep_network(32), 128, 153, 3e-12), (lambda: sweep_network(64), 192, 304, 3e-12),
    (lambda: sweep_network(100), 160, 457, 3e-12), (net150, 192, 1, 1e-11), (net150, 192, 611, 5e-12),
    (net150, 160, 1301, 3e-12), (lambda: sweep_network(250), 320, 305, 3e-12), (net365, 512, 307, 3e-12),
    (net150, 128, 7, 3e-12),  # fewer lanes than species: the group kernel on both sides
])
def test_same_bits_as_the_group_kernel(env, net, G, zones, t_end):
    r = _both(env, net(), profile_zones(net(), zones, base_seed=31, t_end=t_end), G)
    assert (r["status"] == 0).all()


@pytest.mark.parametrize("net,G,zones", [(chain_network, 32, 601), (net150, 192, 460), (net365, 512, 9)])
def test_same_bits_qss(env, net, G, zones):
    _both(env, net(), profile_zones(net(), zones, base_seed=32, t_end=3e-12), G, method=1)


def test_same_bits_long_profiles_and_limits(env):
    # rates refreshed on most steps; the step limit, the reject limit and invalid
    # zones end one zone of a pair while the other goes on
    net = chain_network()
    _both(env, net, profile_zones(net, 1500, base_seed=33, t_end=1e-3), 32)
    net = net150()
    z = profile_zones(net, 900, base_seed=34, t_end=4e-12)
    z.Y0[3, 7] = np.nan
    z.rho0[5] = -1.0
    z.t_end[::7] = 1e-11
    z.tau[::5] = 0.0
    r = _both(env, net, z, 192)
    assert r["status"][3] == 5 and r["status"][5] == 5
    _both(env, net, z, 192, max_reject=0)
    _both(env, net, z, 192, dt_min_frac=0.01)
    c = constant_zones(net, 500, t_end=4e-12)
    _both(env, net, c, 192)


def test_same_bits_small_odd_networks(env):
    # species that no reaction touches, repeated reactants, a single reaction
    net = custom_network([1, 1, 2, 3], [((0,), (0,)), ((0, 0), (2,)), ((2,), (0, 0)), ((0, 0, 0), (3,))],
                         np.log([5.0, 2.0, 1.0, 3.0]), [1.0, 0.0, 2.0, 0.5])
    z = Zones(Y0=np.tile([0.5, 0.2, 0.1, 0.0], (6, 1)), T0=np.linspace(1, 2, 6), rho0=np.ones(6), tau=np.full(6, 3.0),
              t_start=np.full(6, 1e-3), t_end=np.full(6, 1.0), dt_trial=np.full(6, 1e-3))
    for G in (32, 64):
        _both(env, net, z, G)
    for seed in range(6):
        net = random_tiny_network(4 + 3 * seed, 6 + 5 * seed, seed)
        z = Zones(Y0=np.tile(net.initial_Y(), (4, 1)), T0=np.ones(4), rho0=np.linspace(1, 2, 4), tau=np.zeros(4),
                  t_start=np.zeros(4), t_end=np.full(4, 0.2), dt_trial=np.full(4, 1e-6))
        _both(env, net, z, 32 if seed % 2 else 64)


@pytest.mark.parametrize("zones", [(1, 1, 1), (2, 40, 1), (900, 3, 160), (0, 310, 5), (7, 1, 2, 3), (60, 200, 33, 90)])
def test_same_bits_with_several_networks(env, zones):
    # networks of several sizes in one launch, some with fewer zones than CTAs of their own
    torch, kn = env
    G = 384
    nets = [chain_network(), net150(), net365(), sweep_network(64)][:len(zones)]
    opts = kn.Opts(precision=kn.PREC_MIXED, threads_per_zone=G, threads_per_cta=G, max_steps=20000)
    gs, dzs = [], []
    for net, Z in zip(nets, zones):
        if not Z:
            continue
        z = profile_zones(net, Z, base_seed=33, t_end=3e-12)
        gs.append((net, Z, kn.Network(net)))
        dzs.append({k: torch.from_numpy(np.ascontiguousarray(getattr(z, k))).cuda() for k in IN})
        gs[-1][2].set_zones(dzs[-1])
    kn.integrate_batch([g for _, _, g in gs], opts)
    for (net, Z, g), dz in zip(gs, dzs):
        a = g.get()
        one = kn.Network(net)
        one.set_zones(dz)
        kn.integrate_batch([one], opts)
        b = one.get()
        for k in OUT:
            assert np.array_equal(a[k], b[k]), (k, net.n_species)
        assert (a["status"] == 0).all()
        g.close()
        one.close()
