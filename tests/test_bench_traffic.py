"""The DRAM traffic that bench.py reports beside its roofline (no GPU): the figure is
that of the committed ncu summary, and only for the captured workload and layout."""
import os
import re

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
KEY = ("batch128", 1, 0, 32, 0, 200)


def test_reported_traffic_is_the_captured_one():
    text = open(os.path.join(ROOT, "profiles", "dram_traffic_batch128_n500-2000.md")).read()
    rows = re.findall(r"\| timed step \| \S+ \S+ \S+ \S+ \| ([\d.]+) GB \| ([\d.]+) GB \|", text)
    assert len(rows) == 2                     # the step's two launches
    total = sum(float(x) for r in rows for x in r)
    assert abs(bench.FUSED_TRAFFIC[KEY] / 1e9 - total) < 2.5e-3       # four figures rounded to 0.001 GB
    assert float(re.search(r"Traffic per step: ([\d.]+) GB", text).group(1)) == round(total, 2)


def test_no_other_layout_has_a_figure():
    assert list(bench.FUSED_TRAFFIC) == [KEY]


def test_the_line_reads_this_table():
    src = open(os.path.join(ROOT, "bench.py")).read()
    assert src.count("FUSED_TRAFFIC.get(") == 1 and "NCU_TRAFFIC.get(" not in src
