"""The group kernel's queue: every zone is taken once, by a group's dealt first zone or
from the queue behind it, also where a group takes several and where nothing is written
back (kn_probe_step)."""
import numpy as np
import pytest

from kn_inputs import chain_network, net150, profile_zones

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_5826_gb300 import build, kn
    build.build()
    return torch, kn


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("net,tpz,tpc", [(chain_network, 32, 64), (net150, 192, 192)])
def test_probe_of_more_zones_than_groups(env, net, tpz, tpc, prec):
    """Every zone of a probe of several zones a group has the values of that zone alone."""
    torch, kn = env
    net = net()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    Z = 70 * sms + 3  # more than 32 groups an SM could hold, twice over
    z = profile_zones(net, Z, base_seed=51, t_end=1e-11)
    opts = kn.Opts(precision=prec, threads_per_zone=tpz, threads_per_cta=tpc)
    g = kn.Network(net)
    g.set_zones(z)
    a = g.probe(opts)
    for i in (0, 1, sms, 2 * sms + 1, Z // 2, Z - 2, Z - 1):
        g.set_zones(z.subset([i]))
        b = g.probe(opts)
        for k in a:
            assert np.array_equal(a[k][i:i + 1], b[k]), (k, i)
    g.close()


@pytest.mark.parametrize("prec", [0, 2])
def test_each_zone_is_integrated_once(env, prec):
    """A batch of several zones a group gives each zone the results of a batch of its own."""
    torch, kn = env
    net = chain_network()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    Z = 70 * sms + 3
    z = profile_zones(net, Z, base_seed=52, t_end=2e-12)
    opts = kn.Opts(precision=prec, threads_per_zone=32, threads_per_cta=64)
    g = kn.Network(net)
    g.set_zones(z)
    kn.integrate_batch([g], opts)
    assert g.launch_info()["kernel"] == kn.KERNEL_GROUP
    a = g.get()
    assert (a["status"] == 0).all() and np.array_equal(a["t"], z.t_end)
    pick = np.r_[0:40, Z // 2:Z // 2 + 40, Z - 40:Z]
    g.set_zones(z.subset(pick))
    kn.integrate_batch([g], opts)
    b = g.get()
    for k in a:
        assert np.array_equal(a[k][pick], b[k]), k
    g.close()
