"""Host logic of what is kept per device (PerDevice in csrc/cue_internal.h): function attributes and
cluster sizes belong to the device that was current, so each device finds its own, once; a number
past the table is found anew on each call."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1405_3331_gb300", "csrc")

SRC = r"""
#include <cstdio>
#include "cue_internal.h"
int main()
{
    static cue::PerDevice p;
    int calls = 0, bad = 0;
    auto at = [&](int dev, int value) { return p.on(dev, [&] { ++calls; return value; }); };
    bad += at(0, 16) != 16 || at(0, 8) != 16 || calls != 1;      // once on the first device
    bad += at(1, 0) != 0 || calls != 2;                          // the second finds its own, 0 (refused) too
    bad += at(1, 16) != 0 || at(0, 8) != 16 || calls != 2;
    bad += at(63, 5) != 5 || at(63, 6) != 5 || calls != 3;
    bad += at(64, 7) != 7 || at(64, 8) != 8 || at(-1, 9) != 9 || calls != 6;
    std::printf("%s\n", bad ? "bad" : "ok");
    return bad;
}
"""


def test_each_device_finds_its_own_number_once(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "per_device.cu", tmp_path / "per_device"
    src.write_text(SRC)
    subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a", "-I", os.path.join(ROOT, "include"),
                    "-I", CSRC, str(src), "-o", str(exe)], check=True, capture_output=True, text=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr


@pytest.mark.parametrize("name", ["k_tiles.cu", "k_graph.cu"])
def test_allowances_are_set_through_it(name):
    """Every allowance these files set is set under a PerDevice, none behind a flag of the process."""
    text = open(os.path.join(CSRC, name)).read()
    assert "cudaFuncSetAttribute" in text and "static PerDevice" in text
    assert "static bool ready" not in text and "static int size" not in text
