"""The scheduler's internal functions, through a small host program linked with the
library (no GPU needed)."""
import os
import shutil
import subprocess

import pytest

from conftest import ROOT

PKG = os.path.join(ROOT, "paper_2406_19013_gb300")


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_2406_19013_gb300 import build
    lib = build.build()
    exe = str(tmp_path_factory.mktemp("probe") / "sched_probe")
    cuda = os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"))
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(PKG, "csrc"),
                    "-I", os.path.join(cuda, "include"), os.path.join(ROOT, "tests", "sched_probe.cpp"),
                    lib, "-Wl,-rpath," + PKG, "-o", exe], check=True)

    def run(query, *sizes):
        args = [a for n in sizes for a in (query, str(n))]
        out = subprocess.run([exe, *args], check=True, capture_output=True, text=True).stdout
        return [[int(v) for v in line.split()] for line in out.splitlines()]

    return run


def test_tuning_compares_covers_on_a_full_gpu(probe):
    sizes = (1, 2, 16, 17, 32, 48, 64, 65, 96, 128, 192, 256)
    for n_in, channels, *ctas in probe("tune", *sizes):
        # whole units for every SM, whatever the cover
        assert channels % 152 == 0
        assert ctas == [152, 152, 152], (n_in, channels)
