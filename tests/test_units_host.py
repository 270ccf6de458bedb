"""How a simulator pass numbers its work units (ko_units.cuh, compiled for the
host): the parts of every list entry are numbered once each, and no more units
than the list holds that the pass writes its abandoned ones to."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include "ko_units.cuh"
// Units of a list pass; -1 if they are not every part of every entry once, each entry `left` kernels deep.
extern "C" long long list_units(long long items, int levels, int left, long long threads, long long room, int fine)
{
    const kounits::Numbering u = kounits::number_list(items, levels, threads, room, fine != 0);
    const int m = levels + 1;
    unsigned long long seen = 0, prev = ~0ull;
    for (unsigned long long i = 0; i < u.units; i++) {
        const kounits::Unit e = kounits::unit_at(u, i);
        if (e.item != prev) {
            if (prev == ~0ull ? e.item != 0 : e.item != prev + 1) return -1;
            if (seen != 0 && prev != ~0ull) return -1;
            prev = e.item;
        }
        const kounits::Unit c = kounits::cut_unit(e.item, 0, m - left, m, e.x, e.part);
        if (!c.valid) continue;
        if (e.part != seen) return -1;
        const unsigned parts = kounits::parts(left, c.x - (m - left));
        seen = seen + 1 == parts ? 0 : seen + 1;
    }
    if (items && (prev != (unsigned long long)items - 1 || seen != 0)) return -1;
    return (long long)u.units;
}
extern "C" int singles(long long items, int levels, long long room, long long *units)
{
    kounits::Numbering u;
    const bool all = kounits::number_singles(items, levels, room, u);
    *units = (long long)u.units;
    return all;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("units_host")
    src, so = str(d / "units.cpp"), str(d / "libunits.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC",
                    "-I", os.path.join(ROOT, "paper_1511_07983_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(cuda, "include"), src, "-o", so], check=True)
    lib = ctypes.CDLL(so)
    i64 = ctypes.c_longlong
    lib.list_units.argtypes = [i64, ctypes.c_int, ctypes.c_int, i64, i64, ctypes.c_int]
    lib.list_units.restype = i64
    lib.singles.argtypes = [i64, ctypes.c_int, i64, ctypes.POINTER(i64)]
    return lib


@pytest.mark.parametrize("levels", range(7))
@pytest.mark.parametrize("items,threads,room", [(0, 1824, 1024), (1, 1, 1), (336, 1824, 1024), (840, 3648, 1024),
                                                (1024, 43776, 1024), (500, 100000, 2000), (7, 6000, 100000)])
def test_list_pass_numbers_each_part_once_within_its_list(lib, levels, items, threads, room):
    for fine in (0, 1):
        for left in {levels + 1, max(levels, 1)}:     # whole entries, and some cut before
            units = lib.list_units(items, levels, left, threads, room, fine)
            assert 0 <= units <= room and units >= items
    n = ctypes.c_longlong()
    lib.singles(items, levels, room, ctypes.byref(n))
    assert n.value <= room
