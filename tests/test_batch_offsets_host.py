"""Batch offsets outside their contract stay inside the arrays (CPU).

The offsets of batched calls are device arrays that the library does not check.
The search for the instance that owns a position (csrc/ddm_ranges.h) is compiled
for the host here and run over offsets that do not start at 0, end below the
set's size, descend, or hold anything, through an accessor that counts accesses
outside the array; over proper offsets it is compared with numpy's search.
"""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_1309_3458_gb300 import build as B

SRC = r"""
#include "ddm_ranges.h"
struct Checked {
  const unsigned long long* p; uint32_t len; uint64_t* outside;
  unsigned long long operator[](unsigned long long i) const {
    if (i >= len) { ++*outside; return 0; }
    return p[i];
  }
};
// instance of every position, as the fill kernel finds it; returns the accesses
// outside off[0..count] and the instances outside [0, count)
extern "C" uint64_t fill(const unsigned long long* off, uint32_t count, uint32_t total, uint32_t span, uint32_t* inst) {
  uint64_t wrong = 0;
  Checked c{off, count + 1u, &wrong};
  for (uint32_t i0 = 0; i0 < total; i0 += span) {
    ddm::OwnerSearch s(count);
    for (int guard = 0; s.more(); ++guard) {
      if (guard > 40) return ~0ull;  // does not end
      uint32_t yes = 0;
      for (uint32_t l = 0; l < 32; ++l) yes |= (uint32_t)s.probe(c, l, i0) << l;
      s.take(yes);
    }
    const uint32_t end = total - i0 < span ? total : i0 + span;
    for (uint32_t l = 0; l < 32; ++l) {
      ddm::OwnerWalk<Checked> owner(c, count, s.lo);
      for (uint32_t i = i0 + l; i < end; i += 32) {
        inst[i] = owner.at(i);
        wrong += inst[i] >= count;
      }
    }
  }
  return wrong;
}
"""


@pytest.fixture(scope="module")
def fill(tmp_path_factory):
    d = tmp_path_factory.mktemp("ranges")
    (d / "r.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-std=c++17", "-I", B.CSRC, "-o", str(d / "r.so"),
                    str(d / "r.cpp")], check=True)
    f = ctypes.CDLL(str(d / "r.so")).fill
    f.restype = ctypes.c_uint64

    def run(off, total, span=1024):
        off = np.ascontiguousarray(off, dtype=np.uint64)
        inst = np.zeros(total, dtype=np.uint32)
        bad = f(off.ctypes.data_as(ctypes.c_void_p), ctypes.c_uint32(len(off) - 1), ctypes.c_uint32(total),
                ctypes.c_uint32(span), inst.ctypes.data_as(ctypes.c_void_p))
        return bad, inst
    return run


@pytest.mark.parametrize("count", [1, 2, 31, 32, 33, 1024, 1025, 5000])
def test_offsets_outside_the_contract(fill, count):
    rng = np.random.default_rng(count)
    total = 7001
    proper = np.concatenate([[0], np.sort(rng.integers(0, total + 1, count - 1)), [total]])
    short, late, high = proper.copy(), proper.copy(), proper.copy()
    short[-1 - count // 3:] = total // 2                      # ends below the total
    late[: 1 + count // 2] += total // 3                      # starts above 0
    high[-1] = np.iinfo(np.int64).max                         # ends far above it
    for off in (short, np.zeros(count + 1), late, high, proper[::-1],
                rng.integers(0, 2 * total, count + 1), np.full(count + 1, 2 ** 64 - 1, dtype=np.uint64)):
        assert fill(off, total)[0] == 0


@pytest.mark.parametrize("count,span", [(1, 1024), (2, 32), (33, 64), (1025, 1024), (5000, 1024)])
def test_owner_of_every_position(fill, count, span):
    rng = np.random.default_rng(count + span)
    total = 4099
    off = np.concatenate([[0], np.sort(rng.integers(0, total + 1, count - 1)), [total]])  # empty ones too
    bad, inst = fill(off, total, span)
    assert bad == 0
    assert np.array_equal(inst, np.searchsorted(off, np.arange(total), side="right") - 1)


