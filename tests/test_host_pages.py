"""Pages of a download's destination made before the copy (csrc/host_pages.h): fresh memory gets its pages, no byte
of it or of its neighbours changes, and memory that cannot be written is left for the copy to refuse, where a touch
of each page would end the process."""
import os
import shutil
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = """
#include "host_pages.h"
extern "C" void populate(void *p, size_t n) { ccz4::populate_pages(p, n); }
"""
CHILD = """
import ctypes, mmap, sys
lib = ctypes.CDLL(sys.argv[1])
lib.populate.argtypes = [ctypes.c_void_p, ctypes.c_size_t]
libc = ctypes.CDLL(None, use_errno=True)
libc.mmap.restype = ctypes.c_void_p
libc.mmap.argtypes = [ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_long]
libc.mincore.argtypes = [ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p]
page, n = mmap.PAGESIZE, 32
def fresh(prot):
    return libc.mmap(None, n * page, prot, mmap.MAP_PRIVATE | mmap.MAP_ANONYMOUS, -1, 0)
def present(p):
    v = (ctypes.c_ubyte * n)()
    assert libc.mincore(p, n * page, v) == 0
    return [x & 1 for x in v]
p = fresh(mmap.PROT_READ | mmap.PROT_WRITE)
lib.populate(p + 3 * page + 100, 5 * page)          # pages 3 to 8
here = present(p)
assert here == [0] * n or here[3:9] == [1] * 6, here  # (a kernel without the request leaves them)
ctypes.memset(p, 0x5A, n * page)
lib.populate(p, n * page)
lib.populate(p + 8, 1)
assert ctypes.string_at(p, n * page) == b"\\x5a" * (n * page)
lib.populate(fresh(mmap.PROT_READ), n * page)       # read-only
lib.populate(fresh(0), n * page)
lib.populate(None, page)
lib.populate(p, 0)
print("done")
"""


def test_pages_are_made_and_nothing_else_happens(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src, out = str(tmp_path / "pages.cpp"), str(tmp_path / "libpages.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([cxx, "-O2", "-fPIC", "-shared", "-I" + os.path.join(ROOT, "paper_2406_11626_gb300", "csrc"), src,
                    "-o", out], check=True)
    r = subprocess.run([sys.executable, "-c", CHILD, out], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout == "done\n", (r.returncode, r.stdout, r.stderr)
