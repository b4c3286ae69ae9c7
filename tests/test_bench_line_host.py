"""The line that bench.py prints: short enough to be read whole, the contract's numbers in full."""
import json

import bench

MODES = ["fp32", "fp32_da", "fp32_da_multi", "fp64", "fp32_cached", "fp32_da_cached", "fp32_da_multi_cached", "fp64_cached"]


def _mode():
    return {"proposals_per_s": 7123456.123456789, "ms_per_step": 0.14375123456789, "acceptance": 0.20812345678901234,
            "eff": {"docc": 1.0 / 3.0}, "error_bars_binning": {str(k): [1.0 / 3.0] * 8 for k in range(60)}}


def test_printed_line_is_short_and_keeps_the_numbers():
    sweep = {"workload": "five_orbital_sweep_beta50_1024_chains", "metric": "Metropolis proposals/s (all chains)",
             "measure_every": 50, "speedup_fp32_over_fp64": 2.9 / 3.0, **{m: _mode() for m in MODES},
             "speedup_at_equal_error": {f"{a}_over_{b}": {"docc": 1.0 / 3.0, "order": 2.0 / 3.0} for a in MODES[:6] for b in MODES[:2]},
             "throughput_8192_chains": {m: _mode() for m in MODES[:6]} | {"chains": 8192},
             "other_betas": {b: {"beta": 10.0, **{m: _mode() for m in MODES[:3]}} for b in ("beta_10", "beta_100")}}
    line = {"value": 31167819.40549416, "ms_per_step": 0.13141759924590588, "vs_baseline": None, "data": "synthetic",
            "e2e": {"value": 20380866.951263875, "h2d_bytes_per_step": 5052944}, "config": {"beta": 50.0},
            "roofline": {"frac": 0.0011416109114340569, "traffic": None, "nan": float("nan")}, "sweep": sweep}
    assert len(json.dumps(line)) > 30000
    out = bench.printed_line(line)
    text = json.dumps(out)
    assert len(text) < 8192 - 5000  # the other keys of a full run take 4,700
    assert out["value"] == line["value"] and out["e2e"] == line["e2e"] and out["ms_per_step"] == line["ms_per_step"]
    assert out["sweep"]["fp32"]["proposals_per_s"] == 7123460.0 and out["roofline"]["frac"] == 0.00114161
    assert out["sweep"]["beta_100"]["fp32"] == 7123460.0
    assert bench.printed_line({**line, "sweep": None})["sweep"] is None
