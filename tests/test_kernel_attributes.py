"""The opt-in for more than 48 KB of dynamic shared memory is made per handle
(csrc/nls_attr.h): a function attribute belongs to one device, so what one
handle has opted in says nothing about another's device."""
import glob
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2403_16341_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include <map>
#include <set>

#include "nls_attr.h"

int current = 0, calls = 0, refuse = 0;
std::map<int, std::set<const void *>> device; // what each device has opted in
int set(const void *f, int)
{
    ++calls;
    if (refuse) return refuse;
    device[current].insert(f);
    return 0;
}
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main()
{
    const char k0 = 0, k1 = 0;
    nls::SmemOptIns a, b; // handles on device 0 and 1
    const int big = 100 * 1024;
    current = 0;
    CHECK(a.ensure(&k0, big, set) == 0 && a.ensure(&k0, big, set) == 0 && calls == 1);
    CHECK(a.ensure(&k1, 48 * 1024, set) == 0 && calls == 1); // no opt-in needed
    current = 1;
    CHECK(b.ensure(&k0, big, set) == 0);
    CHECK(device[0].count(&k0) && device[1].count(&k0));
    refuse = 7; // an error is passed on, and the next launch tries again
    CHECK(b.ensure(&k1, big, set) == 7 && b.ensure(&k1, big, set) == 7);
    refuse = 0;
    CHECK(b.ensure(&k1, big, set) == 0 && device[1].count(&k1));
    return 0;
}
"""


def test_each_handle_opts_in_on_its_device(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    (tmp_path / "t.cpp").write_text(HARNESS)
    subprocess.run([cxx, "-std=c++17", "-Wall", "-Werror", "-I", CSRC, "-o", str(tmp_path / "t"), str(tmp_path / "t.cpp")],
                   check=True)
    r = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_no_attribute_is_set_once_per_process():
    # a function-local static runs once, on whichever device is current then
    for f in glob.glob(os.path.join(CSRC, "*")):
        assert not re.search(r"static\s+[^;{}]*=\s*cudaFuncSetAttribute", open(f).read()), f
