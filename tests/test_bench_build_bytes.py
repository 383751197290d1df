"""The benchmark's bytes of a build on CPU: only bucket lines that its kernels read count."""

import pytest

import bench


@pytest.mark.parametrize("ranked,small,want", [(1, 0, 0.42), (0, 0, 1.42), (0, 1, 0.0)])
def test_line_reads_of_a_build(ranked, small, want):
    n = 1000
    st = {"insert_probes": 1420, "last_build_ranked": ranked, "last_build_small": small}
    assert bench.build_line_reads(st, n) == pytest.approx(want)


def test_a_two_phase_build_stays_below_the_copy_rate():
    """2^28 keys at load factor 0.9 (1.1025 visits a key in 5.05 ms of build) read and write no more
    than the device can move; every visit as a line read gave more than the measured copy rate."""
    n, ms, peak = 1 << 28, 5.05, 6799.6
    st = {"insert_probes": int(1.1025 * n), "last_build_ranked": 1}
    lines = bench.build_line_reads(st, n)
    assert bench.bytes_per_key("insert", lines, 0.9) * n / (ms / 1e3) / 1e9 < peak
    assert bench.bytes_per_key("insert", 1.1025, 0.9) * n / (ms / 1e3) / 1e9 > peak
