"""Index arithmetic shared by the kernels (csrc/index_math.cuh), compiled for the host: values that stale
memory can hold and sizes at the limit of what the entry points accept."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2404_09679_b200", "csrc")
PROBE = r"""
#include "index_math.cuh"
using namespace antdt;
extern "C" void key_workers(const uint32_t* key, int n, int key_bits, int worker_bits, uint32_t* out) {
  for (int i = 0; i < n; ++i) out[i] = key_worker(key[i], key_bits, worker_bits);
}
extern "C" int32_t run_index_of(int32_t first, int64_t o_begin) { return run_index(first, o_begin); }
// slots that the turns of a group cover (a turn inside the group by its first and last lane); -1: the turns do not end
extern "C" int64_t covered(uint32_t span, uint32_t skew) {
  const BagSpan s(span, skew);
  int64_t n = 0, turns = 0;
  for (uint32_t base = 0; base < s.total; base += kSpanTurn) {
    if (++turns > (1ll << 24) + 1) return -1;
    if (s.whole(base) && s.whole(base + kSpanTurn - 4)) { n += kSpanTurn; continue; }
    for (uint32_t x = base; x < base + kSpanTurn; ++x) n += s.holds(x);
  }
  return n;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("index_math")
    src, so = str(d / "probe.cpp"), str(d / "probe.so")
    open(src, "w").write(PROBE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-fsanitize=undefined", "-fno-sanitize-recover",
                    "-static-libubsan", "-fPIC", "-shared", "-I", CSRC, src, "-o", so], check=True)
    return C.CDLL(so)


@pytest.mark.parametrize("key_bits,worker_bits", [(1, 5), (17, 5), (27, 5), (31, 5), (24, 7), (25, 7)])
def test_worker_of_any_key_is_an_index_into_the_worker_tables(lib, key_bits, worker_bits):
    keys = np.concatenate([np.random.default_rng(0).integers(0, 1 << 32, size=1000, dtype=np.uint64),
                           [0, 1, (1 << 32) - 1, 1 << 31]]).astype(np.uint32)
    out = np.zeros_like(keys)
    lib.key_workers(C.c_void_p(keys.ctypes.data), keys.size, key_bits, worker_bits, C.c_void_p(out.ctypes.data))
    assert out.max() < 1 << worker_bits
    w = np.arange(min(1 << worker_bits, 1 << (32 - key_bits)), dtype=np.uint64)      # and it is the worker of a good key
    good = (w << np.uint64(key_bits) | np.uint64((1 << key_bits) - 1)).astype(np.uint32)
    out = np.zeros_like(good)
    lib.key_workers(C.c_void_p(good.ctypes.data), good.size, key_bits, worker_bits, C.c_void_p(out.ctypes.data))
    assert np.array_equal(out, w)


@pytest.mark.parametrize("o_begin", [0, 16, 64, 4096, (1 << 31) - 64])
def test_run_index_of_a_tile_is_never_outside_what_precedes_it(lib, o_begin):
    f = lambda first: lib.run_index_of(C.c_int32(first), C.c_int64(o_begin))  # noqa: E731
    for good in {0, o_begin // 2, o_begin}:
        assert f(good) == good
    for stale in (-1, -(1 << 31), -2, (1 << 31) - 1, o_begin + 1):
        assert 0 <= f(stale) <= o_begin


@pytest.mark.parametrize("skew", [0, 1, 2, 3])
def test_turns_of_a_group_of_bags_cover_its_slots_once(lib, skew):
    lib.covered.restype = C.c_int64
    for span in [0, 1, 2, 3, 4, 5, 124, 125, 127, 128, 129, 1000, (1 << 31) - 129, (1 << 31) - 128, (1 << 31) - 4,
                 (1 << 31) - 1]:
        assert lib.covered(C.c_uint32(span), C.c_uint32(skew)) == span
