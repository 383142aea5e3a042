"""CPU check of the selection's cuts on the bits of the doubles (csrc/select_cuts.cuh), compiled for the host
from the same source with undefined behaviour trapped: every combination of zeros, denormals, ordinary and
extreme values, infinities and NaN as thresholds and as values gives what the comparisons give."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def test_cuts_are_the_comparisons(tmp_path):
    exe = str(tmp_path / "cuts")
    subprocess.run(["g++", "-O1", "-std=c++17", "-fsanitize=undefined", "-fsanitize-undefined-trap-on-error",
                    os.path.join(HERE, "select_cuts_harness.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stdout)
    assert int(r.stdout) == 23 ** 4
