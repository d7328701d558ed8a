"""The launches of the kernel with several zones per thread group: a network's first
launch prepares what its launches with any number of zones need."""
import numpy as np
import pytest

from kn_inputs import chain_network, net150, net365, profile_zones

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
