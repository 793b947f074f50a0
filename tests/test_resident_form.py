"""Which inputs the resident sort and merge take on a device (csrc/resident_form.cuh), on the host: a whole
B200, one with fewer SMs, one without large clusters or without cooperative launches."""
import ctypes as C
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2404_09679_b200", "csrc")
PROBE = r"""
#include "resident_form.cuh"
using namespace antdt;
extern "C" int holds(const int* lim, int64_t nnz) {
  ResidentLimits l{lim[0], {lim[1], lim[2], lim[3], lim[4]}};
  return resident_holds(l, nnz);
}
extern "C" void form(int64_t nnz, int* out) {
  const ResidentForm f = resident_form(nnz);
  out[0] = f.ctas; out[1] = f.chunk; out[2] = f.cluster;
}
"""
LARGEST = 148 * 512 * 24
CLUSTER = 16 * 4 * 512
SIZES = [1, 1024, 1025, 2049, 8 * 1024, 8 * 1024 + 1, CLUSTER, CLUSTER + 1, 148 * 512 * 4, 148 * 512 * 4 + 1, 148 * 512 * 8,
         148 * 512 * 16 + 1, LARGEST - 31, LARGEST]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("resident_form")
    src, so = str(d / "probe.cpp"), str(d / "probe.so")
    open(src, "w").write(PROBE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-fPIC", "-shared", "-I", CSRC, src, "-o", so], check=True)
    L = C.CDLL(so)
    L.holds.argtypes = [C.POINTER(C.c_int), C.c_int64]
    L.form.argtypes = [C.c_int64, C.POINTER(C.c_int)]
    return L


def _holds(lib, lim, n):
    return bool(lib.holds((C.c_int * 5)(*lim), n))


def _form(lib, n):
    out = (C.c_int * 3)()
    lib.form(n, out)
    return tuple(out)


def test_a_whole_device_takes_everything_up_to_the_limit(lib):
    whole = (16, 296, 296, 148, 148)
    for n in SIZES:
        ctas, chunk, cluster = _form(lib, n)
        assert _holds(lib, whole, n) and ctas * chunk >= n and chunk <= 512 * 24 and ctas <= (16 if cluster else 148)
    for n in (0, -1, LARGEST + 1, 1 << 40):
        assert not _holds(lib, whole, n)


@pytest.mark.parametrize("lim", [(16, 264, 264, 132, 132), (8, 296, 296, 148, 148), (0, 0, 0, 0, 0), (16, 0, 0, 0, 0),
                                 (0, 148, 148, 148, 147), (1, 40, 40, 20, 20)])
def test_a_smaller_device_takes_only_what_it_holds_at_once(lib, lim):
    for n in SIZES:
        ctas, chunk, cluster = _form(lib, n)
        items = (chunk + 511) // 512
        most = lim[0] if cluster else lim[1 + [i for i, k in enumerate((4, 8, 16, 24)) if items <= k][0]]
        assert _holds(lib, lim, n) == (ctas <= most)
