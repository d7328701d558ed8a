"""Host-only checks of the tables of the kernel with several zones per thread group
and of the FP64 form (no device needed): kn_check_gather_tables builds, in KN_PREC_MIXED, every one that
kn_integrate_batch may use for the summation order, and verifies each."""
import time

import pytest

from kn_inputs import chain_network, net150, net365, sweep_network


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


@pytest.mark.parametrize("net,G,size", [(chain_network, 32, 1376), (net150, 160, 31440), (net365, 384, 85040)])
def test_fp64_tables_stage_what_every_group_reads(kn, net, G, size):
    """The FP64 form's tables in shared memory decide how many groups fit a CTA.  The
    list of slices dealt to a wide group's warps (16, 48 and 80 bytes here) is staged for
    wide groups alone, so the others keep the sizes that the tables had without it."""
    assert kn.check_gather_tables(net(), kn.PREC_FP64, G)["table_bytes"] == size
