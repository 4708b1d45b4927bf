"""Kernel attributes and occupancy are looked up for each device, once, under
a lock; no source keeps them in a flag of the whole process."""
import glob
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2402_05283_gb300", "csrc")


def test_values_are_kept_by_device(tmp_path):
    cc = shutil.which("g++")
    if not cc:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "per_device")
    r = subprocess.run([cc, "-std=c++17", "-O2", "-Wall", "-Werror", "-pthread", "-I", CSRC,
                        os.path.join(ROOT, "tests", "per_device_client.cpp"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok"


def test_no_process_wide_flags():
    """A function-local static of a launcher holds per-device facts only."""
    plain = []
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        for i, line in enumerate(open(f), 1):
            if re.match(r"\s+static\s+(const\s+)?(bool|int|cudaError_t|Ready)\b[^(]*[=;{]", line):
                plain.append(f"{os.path.basename(f)}:{i}: {line.strip()}")
    assert not plain, plain
