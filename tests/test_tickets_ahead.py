"""Tour tickets that a warp fetches ahead (host-side check of the kernel's own rule): a
short call still gives every walk a tour, whoever asks first, and a long one reaches the
most that a warp may hold."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2002_03000_gb300", "csrc")


def _ahead(tmp_path, cases):
    exe = str(tmp_path / "tickets")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-I", CSRC,
                    os.path.join(ROOT, "tests", "host", "tickets.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], input="".join("%d %d %d\n" % c for c in cases), capture_output=True, text=True,
                         check=True, timeout=60).stdout
    return [int(v) for v in out.split()]


def test_short_calls_leave_every_walk_a_tour(tmp_path):
    cases = [(k * walks, walks, most) for walks in (1, 2, 12, 48, 64, 65, 4096) for k in range(1, 25) for most in (2, 8)]
    for (left, walks, most), ahead in zip(cases, _ahead(tmp_path, cases)):
        assert 0 <= ahead <= most
        # every walk alone in its warp, all asking at once
        assert walks * (1 + ahead) <= max(walks, left // 2), (left, walks, most, ahead)
        if left >= 2 * walks * (most + 1):
            assert ahead == most


def test_edges(tmp_path):
    cases = [(0, 12, 8), (-5, 12, 8), (11, 12, 8), (48, 12, 8), (215, 12, 8), (216, 12, 8),
             (1 << 40, 1, 8), (10, 1, 8), (17, 1, 8), (18, 1, 8)]
    assert _ahead(tmp_path, cases) == [0, 0, 0, 1, 7, 8, 8, 4, 7, 8]
