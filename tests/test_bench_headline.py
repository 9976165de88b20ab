"""The bench's result line: one short JSON line after the marked detail line."""
import json

import bench


def test_result_is_one_short_json_line(capsys):
    """A reader who has only the last 3000 bytes of the output finds the result whole."""
    per_view = [{"view": v, "n_hist_bounded": {str(k): 0.123456 for k in range(8)}} for v in range(40)]
    line = {"metric": "rays/s " + "x" * 80, "value": 12345678.901234, "unit": "rays/s", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 23.456789, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f16",
            "data": "synthetic (seeded room scene, fitted networks)",
            "config": {"workload": "w" * 120, "rays_per_step": 307200, "views": 10, "samples_per_step": 5.79e6,
                       "grid": "256^3 f32 + uint8", "alg1": {}, "fallback_frac_per_view": [0.1234] * 10,
                       "networks": "SDF 8x256 PE6 skip4 + colour 4x256 PE4", "parallelism": "replicas x1, rays independent"},
            "e2e": {"value": 1.2e7, "unit": "rays/s", "h2d_bytes_per_step": 7372800, "d2h_bytes_per_step": 3686400},
            "gpu_launches": 200, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 60},
            "psnr_gate": {"pixels": 300000, "psnr_tsdf_gpu": 30.123456, "meets_oracle_minus_0p1dB": True},
            "quality": {"per_view": per_view}, "comparator": {"per_view": per_view}, "cpu_baseline": None}
    bench.report(line)
    out = capsys.readouterr().out
    rows = out.splitlines()
    assert rows[0].startswith("detail: ") and json.loads(rows[0][len("detail: "):]) == line
    parsed = [json.loads(r) for r in rows if r.startswith("{")]
    assert len(parsed) == 1 and rows[-1].startswith("{") and len(rows[-1]) < 2800
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "e2e", "gpu_launches", "clocks"):
        assert parsed[0][k] == line[k], k
    assert parsed[0]["config"]["rays_per_step"] == 307200 and "fallback_frac_per_view" not in parsed[0]["config"]
