"""The constants of the fixed-point FP64 step (host code of csrc/) under
UndefinedBehaviorSanitizer, for every lattice speed and relaxation time that a
context can be created with.  CPU only; skipped when g++ cannot build
sanitized binaries."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_constants_are_exact_and_defined_behaviour(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    exe = str(tmp_path / "fixed_ubsan")
    cmd = [gxx, "-O1", "-g", "-std=c++20", "-fsanitize=undefined,float-cast-overflow", "-fno-sanitize-recover=undefined",
           "-ffp-contract=off", "-I", os.path.join(ROOT, "paper_0912_2913_gb300", "csrc"), "-o", exe,
           os.path.join(ROOT, "tests", "sanitize", "fixed_driver.cpp")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0 and "sanitize" in r.stderr:
        pytest.skip("sanitized build unavailable")
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
    assert "runtime error" not in r.stderr, r.stderr
