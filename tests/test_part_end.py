"""The end of a shared tour's parts (host-side check of the order that the kernel uses).

The parts of a tour that grow on several walks end in any order; the last of them squares
the tour's sums into Q_n up to the deepest length that any of them reached.  The kernel's
own function (csrc/perm_parts.h) is compiled for the host and run through every order of
the accesses of up to three parts: exactly one part is the last, and it knows the depth."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2002_03000_gb300", "csrc")


def test_the_last_part_knows_the_deepest_length(tmp_path):
    exe = str(tmp_path / "part_end")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-I", CSRC,
                    os.path.join(ROOT, "tests", "host", "part_end.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
    assert r.stdout.startswith("ok ")
