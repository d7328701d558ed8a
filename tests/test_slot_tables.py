"""Host-only checks of the tables of the kernel with several zones per thread group
(no device needed): kn_check_gather_tables builds, in KN_PREC_MIXED, every one that
kn_integrate_batch may use for the summation order, and verifies each."""
import time

import pytest

from kn_inputs import net150, sweep_network


@pytest.fixture(scope="module")
def kn():
    from paper_1409_5826_gb300 import build, kn
    build.build()
    return kn


@pytest.mark.parametrize("net,G", [(sweep_network(100), 128), (net150(), 192)], ids=["100", "150"])
def test_check_searches_banks_once(kn, net, G):
    """The mixed form's check searches the banks of the values once for a summation
    order.  That search (400 trials a value) takes about five times the FP64 check of
    the same network; with one search for each of the up to 60 tables the check took
    157 to 229 times as long, so the bound lies between, a factor of four from each."""
    best = {}
    for prec in (kn.PREC_FP64, kn.PREC_MIXED):
        best[prec] = float("inf")
        for _ in range(3):
            t0 = time.perf_counter()
            kn.check_gather_tables(net, prec, G)
            best[prec] = min(best[prec], time.perf_counter() - t0)
    assert best[kn.PREC_MIXED] < 30 * best[kn.PREC_FP64]
