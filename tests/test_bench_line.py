"""The bench's one line: the headline's numbers as measured, the rest short enough for a reader that keeps the last
20 000 bytes of the output."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

KINDS = ["dgemm", "chol_leaf", "hbm_pass", "gemv", "jacobi_leaf", "sgemm", "dfgemm", "tcgemm", "ozgemm", "ozprep",
         "tcprep"]


def test_line_is_short_and_keeps_the_headline():
    import bench
    third = 1.0 / 3.0
    kinds = {k: {"ms": 100 * third, "launches": 1234, "flops": 1e15 * third, "bytes": 1e12 * third} for k in KINDS}
    table = bench.kernel_table(kinds, third, 7, {"hbm_gbs": 6767.7, "bf16_sustained": 1718.9})
    line = {"metric": bench.METRIC, "value": third, "ms_per_step": 1000 * third, "kernels": table,
            "e2e": {"value": third, "h2d_bytes_per_step": 2147483648}}
    for arm in range(5):                       # the arms beside the headline, with every kind of kernel in each
        line["arm%d" % arm] = {"s_per_solve": third, "kernels": bench.brief(table), "accuracy": [third] * 10}
    text = json.dumps(bench.rounded(line))
    back = json.loads(text)
    assert back["value"] == third and back["ms_per_step"] == 1000 * third and back["e2e"] == line["e2e"]
    assert set(back["arm0"]["kernels"]) == set(KINDS)
    for k in KINDS:
        assert abs(back["kernels"][k]["ms_per_step"] - table[k]["ms_per_step"]) <= 5e-6 * table[k]["ms_per_step"]
    # beside the tables the full line has about 6 KB of accuracies, notes and the methods' results
    assert len(text) <= 12000
