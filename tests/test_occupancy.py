"""What the library remembers of a kernel's launch limits (csrc/occupancy.h) is
kept per device, and nothing is remembered of a preparation or a query that
failed.  The class is host code: compiled here with a stand-in for two devices."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_05447_gb300", "csrc")

PROGRAM = r"""
#include "occupancy.h"
#include <cstdio>
#include <cstdlib>
#include <set>

static std::set<std::pair<int, const void *>> allowed;   // kernels allowed their shared memory, per device
static int prepared = 0, asked = 0;
static bool refuse = false, lost = false;

static int ask(gpe::Occupancy &o, int dev, const void *k, size_t smem)
{
    return o.blocks(dev, k, smem,
        [&] { ++prepared; if (!refuse) allowed.insert({dev, k}); return !refuse; },
        [&] { ++asked; return lost ? 0 : (smem > 48 * 1024 && !allowed.count({dev, k}) ? 0 : (dev == 0 ? 6 : 3)); });
}
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); std::exit(1); } } while (0)

int main()
{
    gpe::Occupancy o;
    int a, b;
    CHECK(ask(o, 0, &a, 100000) == 6 && prepared == 1 && asked == 1);
    CHECK(ask(o, 0, &a, 100000) == 6 && prepared == 1 && asked == 1);   // remembered
    CHECK(ask(o, 0, &a, 50000) == 6 && prepared == 1 && asked == 2);    // another size
    CHECK(ask(o, 1, &a, 100000) == 3 && prepared == 2);                 // the other device: prepared there, its own answer
    CHECK(allowed.count({1, &a}) == 1);
    CHECK(ask(o, 0, &a, 100000) == 6);
    refuse = true;                                                      // a failure is not remembered
    CHECK(ask(o, 0, &b, 100000) == 1);
    refuse = false;
    CHECK(ask(o, 0, &b, 100000) == 6);
    lost = true;
    CHECK(ask(o, 1, &b, 100000) == 1);
    lost = false;
    CHECK(ask(o, 1, &b, 100000) == 3);
    for (size_t n = 1; n <= 1000; ++n) CHECK(ask(o, 0, &a, n) == 6);    // more sizes than are remembered
    return 0;
}
"""


def test_limits_are_kept_per_device(tmp_path):
    cxx = shutil.which("g++") or pytest.skip("no C++ compiler")
    src, exe = tmp_path / "occupancy.cpp", tmp_path / "occupancy"
    src.write_text(PROGRAM)
    r = subprocess.run([cxx, "-std=c++17", "-Wall", "-Werror", "-I" + CSRC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
