"""The end-to-end record of bench.py carries the host link's own rate beside that of the pass that reads
through it (host logic, no GPU)."""
import math
import os

import bench


def test_link_rates_are_medians_of_the_same_bytes():
    r = bench.link_rates(8_000_000_000, [40.0, 39.0, 200.0], [38.0, 37.0, 36.0])
    assert math.isclose(r["pass1_host_read_gbs"], 200.0)
    assert math.isclose(r["link_copy_gbs"], 8000.0 / 37.0)
    assert math.isclose(r["pass1_frac_of_link"], 37.0 / 40.0)


def test_the_record_holds_them():
    src = open(os.path.join(os.path.dirname(os.path.abspath(bench.__file__)), "bench.py")).read()
    assert "**link_rates(" in src
