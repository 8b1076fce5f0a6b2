"""The benchmark's ground points of records are the sums of their float pairs."""
import numpy as np

import bench
from paper_2405_04229_gb300 import binding as B


def test_ground_sums_both_parts():
    r = np.zeros(2, B.RECORD_DTYPE)
    r["x"], r["x_lo"], r["y"], r["y_lo"] = [1000.0, -5.0], [37.25, 0.5], [2000.0, 8.0], [-12.5, 0.25]
    x, y = bench.ground(r)
    assert x.tolist() == [1037.25, -4.5] and y.tolist() == [1987.5, 8.25]
