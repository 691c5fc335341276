"""Whether a caller's device array may be written in place: it has to lie in one allocation (the library's
own test, in_one_allocation, on a fake of the driver's address ranges).  No GPU needed."""
import ctypes
import os
import shutil
import subprocess

import pytest

from paper_1301_3423_gb300 import builder


@pytest.fixture(scope="module")
def holds(tmp_path_factory):
    d = tmp_path_factory.mktemp("range")
    # allocations [1000, 1800), [1800, 2000) and [5000, 5800)
    (d / "range.cpp").write_text('''#include "rlb_ctx.h"
static bool fake(uintptr_t p, uintptr_t* base, size_t* size) {
  const uintptr_t at[3][2] = {{1000, 800}, {1800, 200}, {5000, 800}};
  for (auto& a : at)
    if (p >= a[0] && p < a[0] + a[1]) return *base = a[0], *size = a[1], true;
  return false;
}
extern "C" int holds(long p, long bytes) { return rlb::in_one_allocation(fake, (uintptr_t)p, (size_t)bytes); }
''')
    cuda = os.path.dirname(os.path.dirname(builder._nvcc()))
    cmd = [shutil.which("g++") or "g++", "-std=c++17", "-shared", "-fPIC", "-o", str(d / "range.so"), str(d / "range.cpp")]
    for inc in (builder.CSRC, builder.INCLUDE, os.path.join(cuda, "include")):
        cmd += ["-I", inc]
    subprocess.check_call(cmd)
    return ctypes.CDLL(str(d / "range.so")).holds


@pytest.mark.parametrize("p,size,want", [
    (1000, 800, True), (1008, 792, True), (1792, 8, True),  # whole, to the end, the last element
    (1000, 808, False),   # one element too many: its end lies in the next allocation
    (1000, 1000, False),  # both ends in allocations of the device, and no gap between them
    (1000, 4800, False),  # both ends in allocations, unmapped addresses between
    (1800, 208, False), (2000, 8, False), (4992, 16, False)])
def test_array_lies_in_one_allocation(holds, p, size, want):
    assert bool(holds(p, size)) == want
