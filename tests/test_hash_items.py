"""The hashing pass's item arithmetic on the host: every 16-byte load of every item lies inside
the column's count array, and the items together cover the column's key range once.  Active
columns (declared and masked arrays, ranges that begin and end anywhere in four slots) and
inactive ones (a key outside the declared domain, no surviving key, a range wider than the
array), read after a column whose smallest key is another one."""
import ctypes as C
import itertools

import pytest

from host_probe import compile_probe

SOURCE = r"""
#include "internal.cuh"
using namespace cmpk;
// out: loads, loads outside the array, keys of the range covered, keys covered twice or outside it
extern "C" void probe(int64_t base, int64_t cap, int masked, int some, int64_t key_min, int64_t key_max,
                      int64_t stale_kmin, int64_t stale_range, int groups, int64_t step, unsigned char* seen,
                      int64_t* out) {
  AggCol a = {};
  a.base = base;
  a.cap = cap;
  a.mask = masked ? uint64_t(cap) - 1 : ~0ull;
  a.kind = kAggCount;
  uint64_t ws[2] = {0, 0};  // (encoded) largest and smallest surviving key
  if (some) ws[0] = enc_max(key_max), ws[1] = enc_min(key_min);
  int64_t kmin = stale_kmin, range = stale_range;  // of the column before
  agg_active(a, 0, reinterpret_cast<unsigned char*>(ws), &kmin, &range);
  const int64_t len = ((range + 3 + groups - 1) / groups + step - 1) / step * step;
  const uint64_t off0 = uint64_t(kmin) - uint64_t(a.base);
  const uint64_t slots = uint64_t((cap + 3) / 4 * 4);
  for (int group = 0; group < groups + 1; group++) {
    const HashSpan s = hash_span(a, kmin, range, len, group, groups);
    for (int64_t j = s.begin; j < s.end; j += 4) {  // one lane's load
      out[0]++;
      const uint64_t at = (off0 + uint64_t(j)) & a.mask;
      if (at % 4 != 0 || at > slots - 4) out[1]++;
      for (int64_t k = j; k < j + 4 && k < range; k++)
        if (k >= 0) {
          if (seen[k]++) out[3]++;
          else out[2]++;
        }
    }
  }
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    L = compile_probe(tmp_path_factory.mktemp("probe"), SOURCE)
    i64, i32 = C.c_int64, C.c_int
    L.probe.argtypes = [i64, i64, i32, i32, i64, i64, i64, i64, i32, i64, C.c_char_p, C.POINTER(i64)]

    def run(base, cap, masked, keys, stale, groups, step=64):
        out = (i64 * 4)()
        lo, hi = keys if keys else (0, 0)
        L.probe(base, cap, masked, 1 if keys else 0, lo, hi, stale, 1000, groups, step, C.create_string_buffer(cap + 128), out)
        return tuple(out)
    return run


STALE = [0, 7, -3, 1 << 33, (1 << 61) - 1, -(1 << 62)]


@pytest.mark.parametrize("base", [0, 5, -7, 1 << 40, -(1 << 50) + 3])
def test_inactive_columns_load_nothing(probe, base):
    cap = 900
    for stale, groups in itertools.product(STALE, [1, 2, 9]):
        for keys in (None, (-(1 << 63), (1 << 63) - 1), (base, base + cap)):
            assert probe(base, cap, 0, keys, stale, groups) == (0, 0, 0, 0), (keys, stale)
            assert probe(0, 1024, 1, None if not keys else (base, base + 1024), stale, groups) == (0, 0, 0, 0)


@pytest.mark.parametrize("hi", [131, 132, 133, 134, 135, 898, 899])
@pytest.mark.parametrize("lo", [0, 1, 2, 3, 4, 131])
def test_items_cover_an_active_column_inside_its_array(probe, lo, hi):
    for stale, groups, step in itertools.product(STALE[:4], [1, 2, 9], [4, 64, 2048]):
        for base in (0, 5, -7, 1 << 40):
            loads, outside, covered, wrong = probe(base, 900, 0, (base + lo, base + hi), stale, groups, step)
            assert outside == 0 and wrong == 0 and covered == hi - lo + 1
        for first in (lo, 1024 * 77 + lo, lo - (1 << 50)):  # masked: the range may wrap around the array
            loads, outside, covered, wrong = probe(0, 1024, 1, (first, first + hi - lo), stale, groups, step)
            assert outside == 0 and wrong == 0 and covered == hi - lo + 1
