"""The bench's line stays short: the rows go into it with their times alone."""
import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))


def test_rows_keep_their_times():
    import bench
    detail = {"kernels": {f"kernel_{k}": {"launches": 20, "total_ms": 1.0, "avg_ms": 0.05} for k in range(20)},
              "roofline": {"bound": "tensor", "note": "x" * 500}}
    rows = {f"row{k}": {"workload": "n=1000 m=500500", "ms_per_call": 0.4 + k, "ms_per_call_cuda_graph": 0.3, **detail}
            for k in range(5)}
    rows.update({f"sweep{k}": {"workload": "n=5000", "n": 5000, "step": "one call",
                               "forms": {f: {"ms_per_step": 4.5, **detail} for f in ("split_bf16", "fp32", "loworder_fp32")}}
                 for k in range(5)})
    assert len(json.dumps(rows)) > 16384
    short = bench.short_rows(rows)
    assert len(json.dumps(short)) < 4096
    assert short["row2"] == {"workload": "n=1000 m=500500", "ms_per_call": 2.4, "ms_per_call_cuda_graph": 0.3}
    assert short["sweep1"]["forms"]["fp32"] == {"ms_per_step": 4.5}
