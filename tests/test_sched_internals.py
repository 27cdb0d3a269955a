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


def test_tmem_kernel_split_models_its_unpack(probe):
    # a chunk costs more the more rows it decodes: 2 for each of 64, 128 and 192
    # staged inputs, at the 2.4 cycles a row that chunk_cost states
    got = probe("tm", 16, 64, 65, 128, 129, 192)
    assert [row[1] for row in got] == [128, 128, 256, 256, 384, 384]
    costs = [row[3] for row in got]
    assert costs[0] == costs[1] < costs[2] == costs[3] < costs[4] == costs[5]
    assert abs((costs[2] - costs[0]) - 128 * 2.4) < 1
    assert abs((costs[4] - costs[2]) - 128 * 2.4) < 1


def test_unit_counts_do_not_overflow(probe):
    # the allocation-free call takes any channel count, with units of 8 channels
    sizes = (1, 7, 8, 9, 1000, 2**31 - 9, 2**31 - 8, 2**31 - 7, 2**31 - 1)
    for n_chan, n_units, last in probe("channels", *sizes):
        assert n_units == -(-n_chan // 8)
        assert 0 <= last < n_chan <= last + 8
