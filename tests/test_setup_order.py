"""What the V-cycle can do without is allocated after everything that setup needs, so that it never is the reason for a
setup that runs out of memory.  Read from the source: memory that runs out at one allocation cannot be arranged here.
"""
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_the_mapped_columns_come_last():
    src = open(os.path.join(ROOT, "paper_2010_11130_gb300", "csrc", "air_api.cu")).read()
    end = src[src.index("int air_setup_end("):]
    end = end[:end.index("\n}\n")]
    assert end.count("air_build_fold(") == 1
    rest = end[end.index("air_build_fold("):]
    assert not any(f in rest for f in ("dalloc", "dmalloc", "air_build_sell", "air_gs_build", "air_tune_lanes"))
