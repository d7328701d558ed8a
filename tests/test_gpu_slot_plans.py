"""The launches of the kernel with several zones per thread group: which networks it
takes (kn_get_launch_info); several networks in one launch, bit for bit against the
group kernel; and that a network's first launch prepares what its launches with any
number of zones need."""
import ctypes as C

import numpy as np
import pytest

from kn_inputs import chain_network, net150, net365, profile_zones, random_tiny_network, sweep_network

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


def _device(torch, z):
    return {k: torch.from_numpy(np.ascontiguousarray(getattr(z, k))).cuda() for k in IN}


@pytest.mark.parametrize("net,most,zones", [(chain_network, 5000, (1, 300, 1000)), (net150, 900, (1, 200, 400)),
                                            (net365, 500, (2, 152))])
def test_another_number_of_zones_under_capture(env, net, most, zones):
    """After one launch at the largest number of zones, a launch with fewer -- one zone a
    group instead of two, fewer and larger groups -- neither allocates nor copies from the
    host: it can be captured in a CUDA graph, whose replay gives the eager call's bits."""
    torch, kn = env
    net = net()
    opts = kn.Opts(precision=kn.PREC_MIXED)
    ref = {}
    for Z in zones:
        one = kn.Network(net)
        one.set_zones(_device(torch, profile_zones(net, Z, base_seed=41, t_end=3e-12)))
        kn.integrate_batch([one], opts)
        ref[Z] = one.get()
        one.close()
    g = kn.Network(net)
    g.set_zones(_device(torch, profile_zones(net, most, base_seed=42, t_end=3e-12)))
    kn.integrate_batch([g], opts)
    assert (g.get()["status"] == 0).all()
    for Z in zones:
        dz = _device(torch, profile_zones(net, Z, base_seed=41, t_end=3e-12))
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            s = torch.cuda.current_stream()
            g.set_zones(dz, s)
            kn.integrate_batch([g], opts, s)
        graph.replay()
        torch.cuda.synchronize()
        r = g.get()
        for k in OUT:
            assert np.array_equal(r[k], ref[Z][k]), (Z, k)
        assert (r["status"] == 0).all()
        del graph
    g.close()


@pytest.mark.parametrize("prec", [0, 1, 2])
def test_first_launch_on_a_stream_of_its_own(env, prec):
    """A network's tables are on the device before its first launch on a stream that does
    not follow the default stream: the same bits as a launch that finds them there."""
    torch, kn = env
    net = net150()
    dz = _device(torch, profile_zones(net, 40, base_seed=43, t_end=3e-12))
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    for rep in range(4):
        g = kn.Network(net)
        g.set_binding_energies(np.linspace(1.0, 2.0, net.n_species))
        runs = []
        for _ in range(2):
            g.set_zones(dz, s)
            kn.integrate_batch([g], kn.Opts(precision=prec), s)
            runs.append({**g.get(s), "E": g.energy(s)})
        for k in OUT + ("E",):
            assert np.array_equal(runs[0][k], runs[1][k]), k
        g.close()


# the networks and orders that test_gpu_slots compares, and the kernel that each is to run
@pytest.mark.parametrize("net,G,zones,kernel,per_group", [
    (chain_network, 32, 1, 1, 1), (chain_network, 32, 5001, 1, 2), (lambda: sweep_network(32), 128, 153, 1, 1),
    (lambda: sweep_network(64), 192, 304, 1, 1), (lambda: sweep_network(100), 160, 457, 1, 2),
    (net150, 192, 1, 1, 1), (net150, 192, 611, 1, 2), (net150, 160, 1301, 1, 2),
    (lambda: sweep_network(250), 320, 305, 1, 2), (net365, 512, 307, 1, 2), (net150, 128, 7, 0, 1),
    (lambda: random_tiny_network(7, 11, 1), 32, 4, 1, 1), (lambda: random_tiny_network(10, 16, 2), 64, 4, 1, 1),
])
def test_the_kernel_that_runs(env, net, G, zones, kernel, per_group):
    torch, kn = env
    net = net()
    opts = kn.Opts(precision=kn.PREC_MIXED, threads_per_zone=G, threads_per_cta=G, max_steps=20)
    g = kn.Network(net)
    with pytest.raises(kn.KnError) as e:
        g.launch_info()
    assert e.value.code == kn.KN_ERR_STATE
    g.set_zones(_device(torch, profile_zones(net, zones, base_seed=31, t_end=3e-12)))
    kn.integrate_batch([g], opts)
    i = g.launch_info()
    assert (i["kernel"], i["threads_per_zone"], i["zones_per_group"]) == (kernel, G, per_group)
    assert i["groups_per_cta"] * i["threads_per_group"] <= 1024 and i["ctas"] >= 1
    g.get()
    # replay and records run the group kernel
    if kernel:
        feat = torch.zeros((1, 64), dtype=torch.float32, device="cuda")
        lab = torch.zeros(1, dtype=torch.float32, device="cuda")
        cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
        g.set_zones(_device(torch, profile_zones(net, 1, base_seed=31, t_end=3e-12)))
        kn.integrate_batch([g], kn.Opts(precision=kn.PREC_MIXED, threads_per_zone=G, threads_per_cta=G, max_steps=2,
                                        record_features=feat.data_ptr(), record_labels=lab.data_ptr(),
                                        record_capacity=1, record_count=cnt.data_ptr()))
        assert g.launch_info()["kernel"] == 0
        g.get()
    g.close()


def _group_kernel(torch, kn, g, dz, opts):
    """kn_integrate_noalloc: the group kernel on the same zones."""
    Z = dz["T0"].shape[0]
    f64 = dict(dtype=torch.float64, device="cuda")
    out = {"Y": torch.empty((Z, g.N), **f64), "t": torch.empty(Z, **f64), "dt_next": torch.empty(Z, **f64),
           "steps": torch.empty(Z, dtype=torch.int64, device="cuda"),
           "rejects": torch.empty(Z, dtype=torch.int64, device="cuda"),
           "status": torch.empty(Z, dtype=torch.int32, device="cuda")}
    zc = kn._Zones(*[dz[k].data_ptr() for k in IN])
    rc = kn.lib().kn_integrate_noalloc(g.h, Z, C.byref(zc), C.byref(opts.c()), *[out[k].data_ptr() for k in OUT],
                                       C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == kn.KN_OK, kn.lib().kn_last_error()
    torch.cuda.synchronize()
    return {k: v.cpu().numpy() for k, v in out.items()}


# CTAs of 480 threads give the 16-species chain one-warp groups, 64 and 150 species
# groups of 160 threads and 365 species one of 480: a mix of all capacities.
# (1, 0, 900): the chain's share of the CTAs rounds to none.
@pytest.mark.parametrize("zones", [(1, 1, 1, 1), (2, 40, 1, 0), (1, 0, 900, 0), (700, 3, 160, 0), (0, 310, 5, 90),
                                   (5000, 200, 33, 0), (40, 500, 60, 300), (0, 700, 0, 2)])
@pytest.mark.parametrize("method", [0, 1])
def test_several_networks_against_the_group_kernel(env, zones, method):
    torch, kn = env
    cta, order = 480, {16: 32, 64: 160, 150: 160, 365: 480}
    gs, dzs = [], []
    for net, Z in zip((chain_network(), net150(), net365(), sweep_network(64)), zones):
        if Z:
            gs.append(kn.Network(net))
            dzs.append(_device(torch, profile_zones(net, Z, base_seed=44, t_end=3e-12)))
            gs[-1].set_zones(dzs[-1])
    opts = dict(precision=kn.PREC_MIXED, method=method, max_steps=20000)
    kn.integrate_batch(gs, kn.Opts(threads_per_cta=cta, **opts))
    for g, dz in zip(gs, dzs):
        i = g.launch_info()
        assert (i["kernel"], i["threads_per_zone"]) == (kn.KERNEL_SLOTS, order[g.N])
        a = g.get()
        G = order[g.N]
        b = _group_kernel(torch, kn, g, dz, kn.Opts(threads_per_zone=G, threads_per_cta=G, **opts))
        for k in OUT:
            assert np.array_equal(a[k], b[k]), (g.N, k)
        assert method or (a["status"] == 0).all()
    assert zones != (1, 0, 900, 0) or gs[0].launch_info()["ctas"] == 0
    for g in gs:
        g.close()


@pytest.mark.parametrize("net,zones,smallest", [(chain_network, 700, 32), (net150, 300, 160)])
def test_autotune_times_each_order_once(env, net, zones, smallest):
    """Trials of the several-zones kernel differ in the order of the sums alone: one each
    for the group sizes from the smallest to 512 threads, and the CTA size that comes back
    is the built-in rule's for the group kernel."""
    torch, kn = env
    net = net()
    z = profile_zones(net, zones, base_seed=45, t_end=3e-12)
    g = kn.Network(net)
    g.set_zones(z)
    t = kn.autotune([g], kn.Opts(precision=kn.PREC_MIXED), max_steps=20)
    G, M = t["threads_per_zone"], t["threads_per_cta"] // t["threads_per_zone"]
    assert t["candidates"] == (512 - smallest) // 32 + 1
    assert t["threads_per_cta"] == G * M and M == min(1024 // G, 15 if smallest == 32 else 5)
    g.set_zones(z)
    kn.integrate_batch([g], kn.Opts(precision=kn.PREC_MIXED))
    i = g.launch_info()
    assert i["kernel"] == kn.KERNEL_SLOTS and i["threads_per_zone"] == G
    # a form on the group kernel: as many candidates as before, two for most group sizes
    g.set_zones(z)
    t = kn.autotune([g], kn.Opts(precision=kn.PREC_MIXED_FP64), max_steps=20)
    assert t["candidates"] > (512 - smallest) // 32 + 1
    g.close()


# (species, zones per SM, QSS, kernel, zones per group, groups per CTA): above 160 species a
# CTA holds two groups at most, in the wide capacities from five zones an SM on; where one
# group fits alone, the QSS update goes back to the group kernel's five (188 species, from
# five zones an SM on) or four (200 species, from sixteen on)
@pytest.mark.parametrize("species,per_sm,method,kernel,nz,groups", [
    (165, 4, 0, 1, 2, 1), (165, 5, 0, 1, 2, 2), (180, 4, 1, 1, 2, 1), (180, 5, 1, 1, 2, 2), (180, 16, 0, 1, 2, 2),
    (188, 4, 1, 1, 2, 1), (188, 5, 1, 0, 1, 5), (188, 16, 0, 1, 2, 1), (200, 15, 1, 1, 2, 1), (200, 16, 1, 0, 1, 4),
    (200, 16, 0, 1, 2, 1), (150, 16, 1, 1, 2, 2), (250, 16, 1, 1, 2, 1),
])
def test_groups_per_cta_above_160_species(env, species, per_sm, method, kernel, nz, groups):
    torch, kn = env
    net = sweep_network(species)
    Z = per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    dz = _device(torch, profile_zones(net, Z, base_seed=46, t_end=2e-12))
    opts = dict(precision=kn.PREC_MIXED, method=method, max_steps=40)
    g = kn.Network(net)
    g.set_zones(dz)
    kn.integrate_batch([g], kn.Opts(**opts))
    i = g.launch_info()
    assert (i["kernel"], i["zones_per_group"], i["groups_per_cta"]) == (kernel, nz, groups)
    a = g.get()
    G = i["threads_per_zone"]
    b = _group_kernel(torch, kn, g, dz, kn.Opts(threads_per_zone=G, threads_per_cta=G, **opts))
    for k in OUT:
        assert np.array_equal(a[k], b[k]), k
    g.close()
