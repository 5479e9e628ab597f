"""bench.py prints its line from runs too short for a clock sample too."""
import bench


def test_clock_of_a_run_without_samples():
    assert bench.clock_mhz(None) == 2070.0
    assert bench.clock_mhz({"sm_mhz": None, "sm_max_mhz": 2000.0}) == 2000.0
    assert bench.clock_mhz({"sm_mhz": 1900.0, "sm_max_mhz": 2000.0}) == 1900.0


def test_only_the_helper_reads_the_summary():
    with open(bench.__file__) as f:
        src = f.read()
    assert "clk[" not in src
