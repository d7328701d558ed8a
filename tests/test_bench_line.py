"""What bench.py reports beside the contract's figures (no GPU)."""
import json

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


def _record():
    """A line of the shape that main() collects, every form with its full record."""
    roof = {"bound": "alu", "resource": "shared-memory bandwidth (SM-local)", "unit": "GB/s", "kernel": "slots_kernel",
            "achieved": 12539.0123456789, "peak": 40273.92, "frac": 0.311344123456789, "peak_source": "p" * 60,
            "algorithmic_smem_bytes_per_launch": 7856008878480.0, "algorithmic_unit": "u" * 120,
            "full_count_smem_bytes_per_launch": 12879060661104.0, "full_count_frac": 0.510374123456789,
            "kernel_ms": 626.573123456789, "traffic": 1.5e9, "traffic_source": "s" * 100,
            "issue": {"active_frac": 0.43, "lsu_pipe_frac": 0.44, "source": "s" * 120}, "smem": {"unit": "u" * 500}}
    tail = {"span_ms": 626.603123, "queue_drained_ms": 620.5, "tail_ms": 6.144123, "finish_ms_p50_p90_p99_max": [1.0] * 4,
            "longest_zone": {"ms": 523.1}, "group_occupancy": 0.995127}
    clocks = {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "samples": 16, "power_w_max": 405.37, "reasons": []}
    launch = {"kernel": 1, "threads_per_zone": 160, "threads_per_group": 256, "zones_per_group": 2,
              "groups_per_cta": 2, "ctas": 152}
    form = {"zone_steps_per_s": 91436301.23456789, "zones_per_s": 2174.890123, "ms_per_batch": 1.5, "kernel_ms": 1883.31,
            "kernel_ms_all": [1883.3] * 3, "accepted_steps": 172203888, "rejects": 15646134, "zones": 4096,
            "zones_ok": 4096, "clocks": clocks, "roofline": roof, "launch": [launch],
            "median_rel_err_vs_tight_oracle": 0.009707123, "tiling": {"threads_per_cta": 960}, "tail": tail}
    forms = {k: dict(form) for k in ("mixed_fp64_update", "fp64", "qss_fp64", "qss_mixed", "mixed_learned",
                                     "uneven_sizes")}
    forms.update({"mixed": {"median_rel_err_vs_tight_oracle": 0.0098, "see": "the headline"}, "note": "n" * 300,
                  "qss_vs_asymptotic_fp64_zones_per_s": 0.297632123,
                  "qss_chain": {"workload": "w" * 80, "qss_vs_asymptotic_fp64_zones_per_s": 2.0,
                                **{k: dict(form) for k in ("asymptotic_fp64", "qss_fp64", "asymptotic_mixed",
                                                           "qss_mixed")}},
                  "mlp_training_kernels": {"us_per_training_step": 24.649123, "frac": 0.0111833, "peak_source": "p" * 80},
                  "perfect_proposal_ceiling": {"plain": {}, "perfect": {}, "steps_ratio": 0.99, "attempts_ratio": 1.0,
                                               "note": "n" * 300}})
    cpu = {"value": 109547.123, "unit": "zone-steps/s", "cores": 16, "kind": "oracle", "sample": "s" * 80}
    one = {k: 1.23456789e-6 for k in ("gpu_fp64_s_per_step", "gpu_mixed_s_per_step", "cpu_oracle_s_per_step",
                                      "cpu_backward_euler_s_per_step")}
    return {"metric": bench.METRIC, "value": 274801490.9071153, "unit": "zone-steps/s", "n_gpus": 1, "steps": 20,
            "warmup": 5, "ms_per_step": 626.6483032226563, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32 (float-float state)", "data": "synthetic", "zones_per_s": 6536.36175,
            "config": {"workload": bench.WORKLOAD, "zones_per_gpu": 4096, "launch": launch,
                       "l2": "flushed between timed steps (256 MB write)"},
            "clocks": clocks, "e2e": {"value": 274002343.39589196, "unit": "zone-steps/s",
                                      "h2d_bytes_per_step": 5111808, "d2h_bytes_per_step": 5062656},
            "gpu_launches": 60, "roofline": roof, "tail": tail, "paper_context": "c" * 160, "forms": forms,
            "single_zone": {"chain16_48": dict(one, cores=1), "net150_1604": dict(one, cores=1),
                            "conditions": "c" * 80},
            "cpu_baseline": cpu, "cpu_implicit_be": cpu}


def test_the_printed_line_is_short_and_keeps_the_contract():
    rec = _record()
    s = bench.short_line(rec)
    # a tail of a few thousand characters of the output has to hold the whole line
    assert len(json.dumps(s)) < 4500 < len(json.dumps(rec))
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "clocks", "e2e", "gpu_launches"):
        assert s[k] == rec[k], k
    assert s["cpu_baseline"]["cores"] == 16 and s["cpu_baseline"]["sample"] == rec["cpu_baseline"]["sample"]
    assert abs(s["roofline"]["frac"] - rec["roofline"]["frac"]) < 1e-6
    assert set(s["forms"]) >= {"fp64", "mixed_learned", "chain_qss_mixed", "mlp_training_kernels"}
    assert s["forms"]["fp64"] == {"zone_steps_per_s": 91436300.0, "zones_per_s": 2174.89, "ms": 1883.31,
                                  "rel_err": 0.00970712, "frac": 0.311344}
    # without the other forms
    for k in ("forms", "single_zone", "cpu_baseline", "cpu_implicit_be"):
        del rec[k]
    assert "forms" not in bench.short_line(rec)
