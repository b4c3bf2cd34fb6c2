"""The digit products that the bench line counts for the folded direct sum: slots
of the kernel's tiles, against a count target line by target line, and the
committed line, whose rate cannot exceed the card's."""
import json
import os

import pytest

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("n,nrhs,lines", [(1024, 8, 4), (512, 5, 4), (64, 1, 32), (97, 2, 16), (129, 3, 8)])
def test_slots_of_the_tiles(n, nrhs, lines):
    slots = 0
    for lo in range(0, n, lines):
        tile = range(lo, min(lo + lines, n))
        slots += 1 + max(abs(i - j) for i in tile for j in (0, n - 1))     # distances 0 .. the farthest source line
    chunks = (n + 127) // 128
    assert bench.conv_digit_flops(n, nrhs) == 2.0 * 128 * 1024 * 128 * slots * chunks * chunks


def test_committed_line_counts_these():
    with open(os.path.join(ROOT, "profiles", "bench_n1024_line.json")) as fh:
        roof = json.load(fh)["roofline"]
    flops = roof["digit_mac_tflops"] * 1e12 * roof["launch_seconds"]
    assert abs(flops / bench.conv_digit_flops(1024, 8) - 1.0) <= 1e-9
    assert roof["digit_mac_occupancy"] <= 1.0
