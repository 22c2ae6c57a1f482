"""Host-side parts of csrc/launch.h that need no GPU."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "launch.h"
#include <thread>
int main() {
    fdg::OncePerDevice a, b;
    if (a.done(0) || a.done(63)) return 1;
    a.set(0);
    if (!a.done(0) || a.done(1) || b.done(0)) return 2;             // another device, another kernel: still to do
    a.set(63); a.set(64); a.set(-1);
    if (!a.done(63) || a.done(64) || a.done(-1) || a.done(1)) return 3;
    std::thread t([&] { for (int i = 0; i < 64; i += 2) b.set(i); });
    for (int i = 1; i < 64; i += 2) b.set(i);
    t.join();
    for (int i = 0; i < 64; ++i) if (!b.done(i)) return 4;          // no thread undoes another's
    return 0;
}
"""


def test_kernel_attributes_are_set_once_per_device(tmp_path):
    """A kernel's shared-memory limit is set for one device: every device of the process has to have it set."""
    inc = "/usr/local/cuda/include"
    if not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("no CUDA headers")
    src = tmp_path / "once.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "once"
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-pthread", "-I", inc, "-I", os.path.join(ROOT, "paper_2509_05679_b200", "csrc"), str(src), "-o", str(exe)])
    assert subprocess.call([str(exe)]) == 0
