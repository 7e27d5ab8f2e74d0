"""The float pairs' host harness (test_dfloat.py) once more with a tracker that
keeps a NaN: a difference that is not a number, wherever it comes among the
samples, counts as beyond every bound."""
import shutil
import subprocess

import pytest

import test_dfloat

LOSES = "if (!(r <= worst)) worst = r; }"
KEEPS = "if (worst == worst && !(r <= worst)) worst = r; }"


def run(tmp_path, source):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    (tmp_path / "h.cpp").write_text(source)
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-I", test_dfloat.CSRC, str(tmp_path / "h.cpp"), "-o",
                    str(tmp_path / "h")], check=True)
    out = subprocess.run([str(tmp_path / "h")], check=True, capture_output=True, text=True).stdout
    return {k: float(v) for k, v in (line.split() for line in out.splitlines())}


def test_every_sample_is_a_number_within_its_bound(tmp_path):
    assert test_dfloat.HARNESS.count(LOSES) == 1
    got = run(tmp_path, test_dfloat.HARNESS.replace(LOSES, KEEPS))
    assert len(got) == 6 and all(v <= 1.0 for v in got.values()), got


def test_the_tracker_keeps_a_nan(tmp_path):
    planted = test_dfloat.HARNESS.replace(LOSES, KEEPS).replace("  // split and back", "  see(NAN, 1);\n  // split and back")
    got = run(tmp_path, planted)
    assert not got["split"] <= 1.0 and all(v <= 1.0 for k, v in got.items() if k != "split"), got
