"""The benchmark's printed line holds the benchmark's keys and fits a log's tail of 3000 characters; the
20 KB of the whole measurement, of which a tail holds no line, stay out of it."""
import json

import bench


def test_printed_line_fits_a_log_tail():
    kernels = {f"kernel_number_{i}": {"ms_per_step": 0.7381055951118469, "achieved": 684.9205362322091, "peak": 1938.6,
                                      "unit": "TFLOP/s", "peak_source": "measured bf16_tflops"} for i in range(40)}
    leg = {"workload": "w" * 300, "pairs_per_s": 43219.512345, "ms_per_step": 1.5, "kernels": kernels}
    full = {"metric": bench.METRIC, "value": 24748.0335748474, "unit": "pairs/s", "n_gpus": 1, "steps": 10, "warmup": 3,
            "ms_per_step": 2.5860640525817873, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "bf16", "data": "synthetic", "config": bench.arm_config(64, 8, "bf16"),
            "roofline": {"kernel": "tc_dec3_final", "bound": "tensor", "achieved": 684.8, "peak": 1938.6,
                         "unit": "TFLOP/s", "frac": 0.3532, "traffic": None},
            "rooflines": kernels, "kernel_time_share": {k: 0.1 for k in kernels},
            "cpu_baseline": {"value": 1.0117296577577972, "unit": "pairs/s", "cores": 16, "kind": "oracle",
                             "cpu_model": "c" * 40, "nproc": 16, "sample": "s" * 160},
            "e2e": {"value": 18542.194153453096, "unit": "pairs/s", "h2d_bytes_per_step": 59904000,
                    "d2h_bytes_per_step": 119232000, "api": "a" * 80},
            "gpu_launches": 100, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"],
                                            "samples": 8, "power_w_max": 909.95, "note": "n" * 90},
            "fp32_peaks": {}, "delta_epe_px": 0.0001441827283503727, "wta_flip_fraction": 0.0,
            "forms": {f: {"pairs_per_s": 24748.0335748474, "rooflines": kernels} for f in ("fp32", "bf16", "fp8")},
            "uneven_batch": leg, "table1_net": leg, "train_step": leg,
            "coarse_variants": {name: leg for name, _ in bench.COARSE_VARIANTS}}
    text = json.dumps(bench.headline(full))
    assert len(text) <= 2500
    got = json.loads(text)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "cpu_baseline"):
        assert got[k] == full[k]
    assert got["pairs_per_s"]["form_fp8"] == 24748.0 and got["pairs_per_s"]["train_step"] == 43219.5
    for leg in ("uneven_batch", "table1_net", "train_step"):  # legs that were left out
        full[leg] = None
    del full["coarse_variants"]
    full["cpu_baseline"] = full["roofline"] = None
    assert set(bench.headline(full)["pairs_per_s"]) == {"form_fp32", "form_bf16", "form_fp8"}
