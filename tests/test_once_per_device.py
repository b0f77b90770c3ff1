"""Set-up that holds for one device is done once on each (csrc/once.h), compiled
with the host compiler: a second GPU to see it on is not needed."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2210_15763_gb300", "csrc")

PROGRAM = r"""
#include "once.h"
#include <cstdio>
#include <thread>
#include <vector>
int main() {
    bbl::OncePerDevice once;
    for (int dev : {0, 3, 63})
        if (!once.need(dev)) return 1;
    once.done(3);
    if (once.need(3) || !once.need(0) || !once.need(63) || !once.need(2)) return 2;
    std::vector<std::thread> t;
    for (int dev = 0; dev < 64; ++dev) t.emplace_back([&once, dev] { if (once.need(dev)) once.done(dev); });
    for (auto& x : t) x.join();
    for (int dev = 0; dev < 64; ++dev)
        if (once.need(dev)) return 3;
    once.done(64);
    once.done(-1);
    if (!once.need(64) || !once.need(-1)) return 4;
    return 0;
}
"""


def test_each_device_is_set_up_once(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    (tmp_path / "once.cpp").write_text(PROGRAM)
    exe = str(tmp_path / "once")
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(tmp_path / "once.cpp"), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0


def test_no_set_up_flag_per_process():
    """Function attributes belong to a device: no kernel's are guarded by a flag of the process."""
    for f in sorted(os.listdir(CSRC)):
        if f.endswith(".cu"):
            text = open(os.path.join(CSRC, f)).read()
            assert "static bool attr" not in text, f
