"""The benchmark's standard output is one line short enough for a log's tail to keep whole: a full
record (tuning tables, per-kernel tables of every leg, accuracies) reduced to its headline."""
import json

import bench


def _kernels():
    names = ["k_project", "k_scan_tiles", "k_emit", "k_sort_tiles", "k_track_tile", "k_bproject", "k_finalize"]
    return {k: 1234.56 for k in names}


def _record():
    sched = {"tile_w": 16, "tile_h": 16, "sub_buckets": 4, "fwd_batch": 256, "bwd_batch": 256, "flags": 1}
    tuned = {"schedule": sched, "tuned": True,
             "timings_ms": [{"stage": "backward", "schedule": sched, "ms": 0.1234}] * 17}
    leg = {"ms_per_step": 62.12168579101562, "mpix_per_s": 2915.1559184858897, "launch_schedule": tuned,
           "roofline_kernels": {k: {"bound": "hbm", "work": "x" * 100} for k in _kernels()}}
    err = {"inf": 1.234567890123456e-05, "l2": 1.234567890123456e-05}
    acc = {"max_err_unflagged": 3.798899781060072e-05, "loss_rel_err": 3.483330850052336e-07, "pose_grad_rel_err": err,
           "param_grad_rel_err": {k: err for k in "abcde"}}
    seq = {"ms_per_frame": 88.816, "launch_schedule": sched, "ate_rmse_cm": 4.492}
    return {
        "metric": bench.METRIC, "value": 2520.0488668773014, "unit": "Mpix/s", "n_gpus": 1, "steps": 20, "warmup": 5,
        "ms_per_step": 0.12190239802002907, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f32", "data": "synthetic (room scene; ray-cast RGB-D frame)",
        "config": {"workload": bench.WORKLOAD, "width": 640, "height": 480, "gaussians": 200000, "pairs": 163361,
                   "records": 32808, "max_tile_pairs": 475, "l2": "flushed between timed steps (256 MB write)",
                   "parallelism": "replicas x1", "launch_schedule": tuned},
        "tracking_iters_per_s": 8203.284071866216,
        "e2e": {"value": 2579.5703629783193, "unit": "Mpix/s", "h2d_bytes_per_step": 6144000, "d2h_bytes_per_step": 64,
                "frame": "y" * 80, "copied_upload": {"value": 2334.687170493374, "unit": "Mpix/s", "frame": "z" * 60}},
        "gpu_launches": 160, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 9},
        "roofline": {"kernel": "k_track_tile", "bound": "alu", "achieved": 12.731476341062123, "peak": 80.54784,
                     "unit": "TFLOP/s", "frac": 0.15806105217796187, "traffic": 11020000, "traffic_from": "p" * 200},
        "kernels_us": _kernels(), "kernels_us_note": "n" * 225,
        "pairs_per_step": {k: 17531293 for k in ("fwd_evals", "fwd_contrib", "bwd_evals", "bwd_contrib")},
        "useful_pair_evals_per_s": 1.8e11, "roofline_kernels": leg["roofline_kernels"],
        "isotropic": {"anisotropic": {"us_per_iter": 129.27}, "isotropic": {"us_per_iter": 125.08}, "workload": "w" * 100},
        "batched": {"batched_bf16": leg, "batched_fp32": leg, "plain_fp32": leg, "speedup_vs_tuned_plain": 1.6745390795427046},
        "mapping": {"chunks": {str(k): {"ms_per_window": 2.5 + k, "mpix_per_s": 2000.0} for k in (1, 2, 4, 8)}},
        "sequence": {"workload": "s" * 90, "tracking_fixed_map": seq, "slam_from_empty_map": seq,
                     "slam_from_empty_map_isotropic": seq},
        "cpu_baseline": {"value": 1.1469287975787124, "unit": "Mpix/s", "cores": 16, "kind": "oracle",
                         "sample": "57 full tracking iterations of the 640x480 / 200k workload in 15.3 s",
                         "accuracy_vs_oracle": {"tracking_frame": acc, "mapping_keyframe_1": acc,
                                                "sequence_drift": {"trans_diff_mm_per_frame": [0.0025] * 200}}}}


def test_the_printed_line_is_short_and_whole():
    rec = _record()
    line = json.dumps(bench.headline(rec))
    assert len(json.dumps(rec)) > 8000 and len(line) < 2500 and "\n" not in line
    got = json.loads(line)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "gpu_launches", "clocks"):
        assert got[k] == rec[k]
    assert got["e2e"]["value"] == rec["e2e"]["value"] and got["e2e"]["h2d_bytes_per_step"] == 6144000
    assert got["config"]["workload"] == bench.WORKLOAD and got["cpu_baseline"]["value"] == rec["cpu_baseline"]["value"]
    assert got["legs"]["mapping_window_ms"] == 3.5


def test_legs_left_out_stay_out():
    rec = _record()
    for k in ("isotropic", "batched", "mapping", "sequence", "cpu_baseline"):
        del rec[k]
    rec["roofline"] = None
    assert "legs" not in bench.headline(rec) and "cpu_baseline" not in bench.headline(rec)
