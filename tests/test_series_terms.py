"""The term counts of the FP64 series: every threshold keeps the first term left out below the
target, by the bound that the table's comment states."""
import math
import os
import re

from paper_2202_10647_gb300 import build


def test_flow_thresholds():
    src = open(os.path.join(build.CSRC, "ion_device.cuh")).read()
    table = re.search(r"kThrFlow\[.*?\] = \{(.*?)\};", src, re.S).group(1)
    rows = [[float(x.rstrip("f")) for x in re.findall(r"[\d.e+-]+f", row)]
            for row in re.findall(r"\{(.*?)\}", table, re.S)]
    assert len(rows) == 5 and all(len(r) == 18 for r in rows)
    for w, row in enumerate(rows, start=2):
        assert row == sorted(row) and row[-1] > 1.0  # 2 W dt goes up to 1
        for i, x in enumerate(row):
            k = i + 1
            paths = sum(math.comb(k, j) for j in range(min(w - 1, k) + 1))
            assert (x / 2) ** k * paths / math.factorial(k) <= 2e-17 * (1 + 1e-4)
