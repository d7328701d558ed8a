"""What bench.py reports beside the contract's figures (no GPU)."""
import bench


def test_occupancy_counts_the_launch_s_slots():
    """The slots are those of the launch, filled or not: 152 CTAs of three groups of two
    zones hold 912, of which a batch that keeps 600 busy all the time fills 600 / 912."""
    import numpy as np
    info = {"kernel": 1, "threads_per_zone": 192, "threads_per_group": 160, "zones_per_group": 2, "groups_per_cta": 3,
            "ctas": 152}
    slots = bench.zone_slots(info)
    assert slots == 912 and bench.KERNELS[info["kernel"]] == "slots_kernel"
    ns = np.zeros((600, 2), np.int64)
    ns[:, 1] = 7_000_000
    assert abs(bench.tail_stats(ns, np.ones(600), slots)["group_occupancy"] - 600 / 912) < 1e-12
