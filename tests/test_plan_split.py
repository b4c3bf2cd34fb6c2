"""Which problems of a batch are planned with every thread, one after the other,
and which side by side: large problems never on one thread each (four of
n = 512, one of n = 1024 among small ones), many small ones never in turn."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1307_2666_gb300", "csrc")


def cost(active, threads, k):
    """Modelled time with the first k in turn, in DOFs of one thread."""
    start, every = 48.0 * threads, 0.7 * threads
    t = sum(start + a / every for a in active[:k])
    return t + (start + max(active[k], sum(active[k:]) / every) if k < len(active) else 0.0)


def test_plans_by_size(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = tmp_path / "plan_split"
    subprocess.run([gxx, "-O1", "-std=c++17", "-fopenmp", "-I", CSRC, os.path.join(ROOT, "tests", "plan_split_harness.cpp"),
                    os.path.join(CSRC, "geometry.cpp"), "-o", str(exe)], check=True)
    sq = lambda *n: [v * v for v in n]
    cases = [(16, sq(512, 512, 512, 512)), (16, sq(1024, 64, 64, 64)), (16, sq(*[1024] * 4)), (8, sq(*[512] * 4)),
             (16, sq(*[64] * 100)), (16, sq(*[256] * 16)), (16, [200] * 24), (16, sq(1024)), (16, []), (1, sq(64, 64)),
             (4, sq(*[48] * 200)), (16, [0, 0, 0])]
    rng = np.random.default_rng(1)
    for _ in range(200):
        n = int(rng.integers(1, 40))
        cases.append((int(rng.integers(2, 80)), sorted((int(v) for v in 10.0 ** rng.uniform(0, 6.2, n)), reverse=True)))
    text = "".join(f"{t} {len(a)} {' '.join(map(str, a))}\n" for t, a in cases)
    got = list(map(int, subprocess.run([str(exe)], input=text, check=True, capture_output=True, text=True).stdout.split()))
    assert len(got) == len(cases)
    assert got[0] == 4 and got[1] >= 1 and got[2] == 4 and got[3] == 4      # every thread for the large ones
    assert got[4] == got[5] == got[6] == got[10] == 0                       # side by side
    assert got[7:10] == [1, 0, 2]
    for (threads, a), k in zip(cases, got):
        assert 0 <= k <= len(a) and k != len(a) - 1 or len(a) <= 1
        if threads > 1 and len(a) > 1:
            assert cost(a, threads, k) <= min(cost(a, threads, 0), cost(a, threads, len(a))) * (1 + 1e-12)
