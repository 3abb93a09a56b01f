"""What bench.py prints: one line on stdout, short enough for what keeps only the end of a program's output, tables on stderr."""
import json

import velora_inputs as vi


def test_the_line_is_short_and_the_tables_go_to_stderr(capsys):
    import bench
    row = {"kernel": "weight_grad factored P = dY^T Z, dW = P v", "shape": "8192x11008x4096", "Dsub": 64, "us": 59.123456789, "bytes": 272629760,
           "GB/s": 4611.123456789, "frac_measured": 0.7123456789, "us_graph": 57.123456789, "frac_graph": 0.73123456789}
    line = {"metric": bench.METRIC, "value": 1654321.987654321, "unit": bench.UNIT, "clocks": {"sm_mhz": 1605, "sm_max_mhz": 1965, "reasons": []},
            "config": bench.workload_config(vi.CONFIGS[bench.CONFIG_DEFAULT]),
            "roofline": {"kernel": "velora_linear_forward", "achieved": 1436.123456789, "frac": 0.8765432109876, "timing_floor_us": {"per_call": 6.5},
                         "compress": [row] * 6, "reconstruct": [row] * 6, "weight_grad_factored": [dict(row, shape="8192x%dx4096" % i) for i in range(6)]},
            "kernels": [row] * 60, "e2e": {"value": 334691.6303170865, "unit": bench.UNIT}}
    bench.emit(line)
    got = capsys.readouterr()
    assert got.out.count("\n") == 1 and len(got.out) < 3000
    out = json.loads(got.out)
    assert abs(out["value"] / line["value"] - 1) < 1e-5 and out["e2e"]["value"] == 334692.0 and out["config"] == line["config"]
    assert out["roofline"]["weight_grad_factored_us"]["8192x5x4096/64"] == 57.1235 and "kernels" not in out
    tables = [json.loads(l) for l in got.err.splitlines()]
    assert sum(t["table"] == "kernels" for t in tables) == 60 and {"compress", "reconstruct", "weight_grad_factored", "timing_floor_us"} <= {t["table"] for t in tables}
