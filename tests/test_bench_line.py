"""The line bench.py prints: it has what its readers need and stays short whatever the blocks hold."""
import json

import bench


def _layer(name):
    return {"layer": name, "us": 1234.56, "density": 0.2995, "kernel": "tcgen05 channel-major", "gated_tflops": 1234.5,
            "gbs": 1234.5, "roof_us": 123.45, "roof_frac": 0.322, "bound": "hbm", "flop_reduction": 2.107,
            "executed_over_gated": 2.107, "blocks_skipped": "0/409600", "us_density1": 1234.56,
            "speedup_vs_density1": 0.991}


def _record(layers, blocks):
    return {"metric": bench.METRIC, "value": 2235126.9, "unit": bench.UNIT, "n_gpus": 1, "steps": 200, "warmup": 10,
            "ms_per_step": 0.11453, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "bf16",
            "data": "synthetic",
            "config": {k: "x" * 60 for k in ("workload", "calibration", "l2", "parallelism", "e2e")},
            "clocks": {"sm_mhz": 1965.0, "sm_max_mhz": 1965.0, "reasons": [], "samples": 11},
            "e2e": {"value": 169646.3, "unit": "images/s", "h2d_bytes_per_step": 62914560, "d2h_bytes_per_step": 66846720},
            "gpu_launches": 800, "speedup_vs_density1": 0.989,
            "roofline": {"bound": "hbm", "achieved": 2104.7, "peak": 6542.4, "unit": "GB/s", "frac": 0.3217, "traffic": None,
                         "algorithmic_bytes": 69279744, "kernel": "tcgen05 tap-stacked (c64@32)",
                         "peak_source": "of measured", "us_per_launch": 32.92},
            "cpu_baseline": {"value": 450.774, "unit": "images/s", "cores": 16, "kind": "oracle", "sample": "y" * 110},
            "layers": layers, "blocks": blocks}


def test_the_line_is_short_and_whole():
    blocks = [{"workload": "imagenet_resnet18_gated_3x3_layers", "batch": 64, "groups": b["groups"], "rho": b["rho"],
               "dtype": b["dtype"],
               "densities": {str(d): {"us_all_layers": 1234.56, "layers": [_layer("c")] * 7} for d in b["densities"]}}
              for b in bench.EXTRA_BLOCKS]
    blocks.append({**{k: 0.123456 for k in bench.NETWORK_KEYS}, "workload": "cg_resnet18_forward",
                   "ms_per_operator": {f"layer{i}": 0.1234 for i in range(30)}, "kernels": {str(i): "k" * 20 for i in range(21)}})
    out = _record([_layer(n) for n in ("c64@32", "c128@16", "c256@8", "c512@4")], blocks)
    line = bench.headline(out)
    assert "\n" not in line and len(line) < 3000
    got = json.loads(line)
    assert {k: v for k, v in got.items() if k not in ("layers", "blocks")} == \
        {k: v for k, v in out.items() if k not in ("layers", "blocks")}
    assert [x["us"] for x in got["layers"]] == [1234.56] * 4 and len(got["blocks"]) == len(blocks)
    assert got["blocks"][0]["us_all_layers"] == {str(d): 1234.56 for d in bench.EXTRA_BLOCKS[0]["densities"]}
    assert len(out["blocks"][0]["densities"]["0.1"]["layers"]) == 7      # (the record itself keeps everything)
