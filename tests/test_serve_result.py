"""The host's reading of a serving slot against a thread that publishes as the
device does (serve_result_driver.cpp)."""
import os
import shutil
import subprocess

import pytest

from tests.helpers import ROOT


def run(tmp_path, *flags, args=()):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    exe = tmp_path / "serve_result"
    cmd = ["g++", "-O2", "-std=c++17", "-pthread", *flags, "-I", os.path.join(ROOT, "paper_1511_06103_gb300", "csrc"),
           os.path.join(ROOT, "tests", "serve_result_driver.cpp"), "-o", str(exe)]
    b = subprocess.run(cmd, capture_output=True, text=True)
    assert b.returncode == 0, b.stderr
    return subprocess.run([str(exe), *args], capture_output=True, text=True, timeout=120)


def test_timed_out_slot_is_never_finished(tmp_path):
    r = run(tmp_path)
    assert r.returncode == 0, r.stdout + r.stderr


def test_no_data_race(tmp_path):
    """Under ThreadSanitizer: what follows done is read behind an acquire."""
    probe = tmp_path / "probe.cpp"
    probe.write_text("int main() { return 0; }")
    exe = tmp_path / "probe"
    b = subprocess.run(["g++", "-fsanitize=thread", str(probe), "-o", str(exe)], capture_output=True, text=True)
    if b.returncode != 0 or subprocess.run([str(exe)]).returncode != 0:
        pytest.skip("no ThreadSanitizer runtime here")
    r = run(tmp_path, "-g", "-fsanitize=thread", args=("short",))
    assert r.returncode == 0 and "WARNING: ThreadSanitizer" not in r.stderr, r.stdout + r.stderr
