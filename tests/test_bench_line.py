"""The benchmark's result is one line of JSON that is short enough to be read from the end of the output."""
import json

import bench


def test_the_result_line_stays_short_and_keeps_what_is_asked_for():
    keep = {"metric": "m", "value": 1.23456789012, "unit": "u", "ms_per_step": 2.0 / 3.0, "config": {"workload": "w" * 300},
            "e2e": {"value": 1.0, "h2d_bytes_per_step": 12345678901}, "gpu_launches": 40, "clocks": {"sm_mhz": 1860.0}}
    long = {str(i): {"ms": 1.0 / (i + 3), "gbs": 6000.0 / (i + 7), "note": "n" * 60} for i in range(40)}
    line = bench.result_line(dict(keep, by_mask=long, normclip_step=long, diag_step=long, graph_window=None))
    assert len(line) <= bench.MAX_LINE and "\n" not in line
    got = json.loads(line)
    assert all(k in got for k in keep) and got["value"] == 1.23457 and got["e2e"]["h2d_bytes_per_step"] == 12345678901
    full = bench.result_line(dict(keep, by_mask={"0": {"ms": 25.5}}))
    assert json.loads(full)["by_mask"] == {"0": {"ms": 25.5}}
