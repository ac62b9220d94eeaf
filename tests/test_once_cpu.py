"""A kernel's shared-memory limit is raised once on each device (csrc/slr_once.h)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdio>
#include "slr_once.h"
int main() {
    slr::OncePerDevice once;
    int a = 0, b = 0, calls = 0;
    bool up = true;
    auto on = [&](const void* key, int dev) {
        return once.run(key, dev, [&]() { ++calls; return up; });
    };
    auto say = [&](bool ok) { std::printf("%d%d ", ok, calls); };
    say(on(&a, 0)); say(on(&a, 0));            // once
    say(on(&a, 1)); say(on(&a, 1));            // again on another device
    say(on(&b, 1));                            // another kernel
    up = false; say(on(&b, 0));                // a refusal is reported and not remembered
    up = true; say(on(&b, 0)); say(on(&a, 0));
}
"""


def test_once_for_each_kernel_and_device(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_1505_04340_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert out == ["11", "11", "12", "12", "13", "04", "15", "15"]
