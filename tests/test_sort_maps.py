"""Key arithmetic of the batch sort (csrc/sort_maps.h), compiled for the host: no GPU needed."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1707_05354_gb300", "csrc")

# The rounds over a crowded bucket as the device takes them, on one thread: the elements of the turn's keys are done
# when at most `cap` of them are left, else the turn is narrowed to the longest prefix of sub-bins that fits.  Prints the
# number of rounds, or "endless" / "out of order".
ROUNDS = r"""
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "sort_maps.h"
using namespace gpulsm;
int main(int argc, char** argv) {
  const uint32_t n = strtoul(argv[1], 0, 0), cap = strtoul(argv[2], 0, 0), lo = strtoul(argv[3], 0, 0),
                 hi = strtoul(argv[4], 0, 0);
  std::vector<uint32_t> x(n);
  uint64_t s = 88172645463325252ull;
  for (auto& k : x) {
    s ^= s << 13; s ^= s >> 7; s ^= s << 17;
    k = lo + uint32_t((s >> 20) % (uint64_t(hi) - lo + 1));
  }
  KeyTurn turn;
  uint32_t done = 0, rounds = 0;
  uint64_t next_key = 0;
  while (done < n) {
    if (++rounds > 64 * (n / cap + 2)) return puts("endless"), 0;
    uint32_t c = 0, mn = ~0u, mx = 0;
    for (uint32_t k : x)
      if (k >= turn.a && k <= turn.b) ++c, mn = std::min(mn, k), mx = std::max(mx, k);
    if (c == 0) { turn.next(); continue; }
    if (mn < next_key) return puts("out of order"), 0;
    if (mn != mx && c > cap) {
      const SubMap map = SubMap::of(mn, float(mx - mn) + 1.0f);
      std::vector<uint32_t> cnt(kSubBins, 0);
      for (uint32_t k : x)
        if (k >= turn.a && k <= turn.b) ++cnt[map.sub(k)];
      uint32_t fit = 0, run = 0;
      for (uint32_t i = 0; i < kSubBins && (run += cnt[i]) <= cap; ++i) fit = i + 1;
      turn.narrow(mn, map, fit);
      continue;
    }
    done += c;
    next_key = uint64_t(mx) + 1;
    turn.next();
  }
  printf("%u\n", rounds);
}
"""


def run(tmp_path, source, *args):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = tmp_path / "t"
    (tmp_path / "t.cpp").write_text(source)
    subprocess.run([cxx, "-std=c++17", "-O2", "-I" + CSRC, str(tmp_path / "t.cpp"), "-o", str(exe)], check=True)
    return [subprocess.run([str(exe)] + [str(v) for v in a], capture_output=True, text=True, check=True, timeout=60).stdout.strip()
            for a in args]


def test_rounds_end_for_any_keys(tmp_path):
    """No key is outside the turns: neither 0 and 2^32 - 1 nor keys that another range was published for."""
    cases = [(n, cap, lo, hi) for n, cap in ((6000, 5120), (20000, 5120), (3000, 100))
             for lo, hi in ((0, 0xFFFFFFFF), (0, 0), (0, 1), (0xFFFFFFFF, 0xFFFFFFFF), (0xFFFFFFFE, 0xFFFFFFFF),
                            (5, 4100), (5, 4101), (1 << 31, (1 << 31) + 70000), (0, 0xFFFFFFFE), (1, 0xFFFFFFFF))]
    out = run(tmp_path, ROUNDS, *cases)
    for c, o in zip(cases, out):
        assert o.isdigit() and int(o) <= 8 * (c[0] // c[1] + 2) + min(c[0], 4 * (c[3] - c[2] + 1)), (c, o)


# Of 1000 batches of n keys spread evenly from lo to hi, those with more than `few` keys beyond the range that the map of
# 512 samples covers.
COVER = r"""
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "sort_maps.h"
using namespace gpulsm;
int main(int argc, char** argv) {
  const uint32_t n = strtoul(argv[1], 0, 0), lo = strtoul(argv[2], 0, 0), hi = strtoul(argv[3], 0, 0),
                 few = strtoul(argv[4], 0, 0);
  uint64_t s = 88172645463325252ull;
  std::vector<uint32_t> x(n);
  int bad = 0;
  for (int t = 0; t < 1000; ++t) {
    for (auto& k : x) {
      s ^= s << 13; s ^= s >> 7; s ^= s << 17;
      k = lo + uint32_t((s >> 20) % (uint64_t(hi) - lo + 1));
    }
    uint32_t mn = ~0u, mx = 0;
    for (uint64_t e = 0; e < 512; ++e) {
      mn = std::min(mn, x[e * n / 512]);
      mx = std::max(mx, x[e * n / 512]);
    }
    const KeyMap m = KeyMap::spanning(mn, mx, 256, 0, nullptr);
    uint32_t below = 0, above = 0;
    for (uint32_t k : x) {
      below += k < m.lo;
      above += k > m.lo && mul_hi(k - m.lo, m.mul) >= m.parts;
    }
    bad += below > few || above > few;
  }
  printf("%d\n", bad);
}
"""


def test_sampled_range_covers_even_keys(tmp_path):
    """More than the 48 keys that a sub-bin may hold are beyond the range in about two of e^10 = 22000 batches; three of
    1000 would be there with a probability of 10^-4."""
    cases = [(30000, 1 << 29, 5 << 29, 48), (1 << 17, 0, 1 << 31, 48), (30000, 1 << 20, 1 << 25, 48)]
    for c, o in zip(cases, run(tmp_path, COVER, *cases)):
        assert int(o) <= 2, (c, o)


# The largest part of the batched form's map over keys spread evenly from lo to hi, in percent of an even share, or what
# is wrong with the parts' bounds.
PARTS = r"""
#include <cstdio>
#include <cstdlib>
#include "sort_maps.h"
using namespace gpulsm;
int main(int argc, char** argv) {
  const uint32_t lo = strtoul(argv[1], 0, 0), hi = strtoul(argv[2], 0, 0), bits = strtoul(argv[3], 0, 0), n = 1u << bits;
  const PartMap m = PartMap::spanning(lo, hi, bits);
  uint64_t most = 0;
  for (uint32_t p = 0; p < n; ++p) {
    const uint64_t a = p ? m.lower(p) : 0, z = p + 1 < n ? m.lower(p + 1) : 1ull << 32;
    if (a < 0xFFFFFFFFull && z > a && (m.part(uint32_t(a)) != p || m.part(uint32_t(z - 1)) != p)) {
      if (z != 0xFFFFFFFFull) return puts("bounds"), 0;
    }
    const uint64_t x = a < lo ? lo : a, y = z > uint64_t(hi) + 1 ? uint64_t(hi) + 1 : z;
    if (y > x && y - x > most) most = y - x;
  }
  printf("%.1f\n", 100.0 * double(most) * n / (double(hi) - lo + 1));
}
"""


@pytest.mark.parametrize("bits", [1, 2, 3, 8])
def test_parts_are_even(tmp_path, bits):
    """A part is at most 5 % above its share: the range is widened by 1/50 at both ends (4 %), the factor rounded down by
    1/256 at most (0.4 %), and a bound to a whole key (of 780 at least)."""
    cases = [(lo, hi, bits) for lo, hi in ((0, 0xFFFFFFFE), (0, 1 << 31), (0, 3200000000), (1 << 30, 3 << 30),
                                           (0, 0xC0000000), (12345, 0x70000000), (0, 1 << 25), (77, 200000))]
    for c, o in zip(cases, run(tmp_path, PARTS, *cases)):
        assert float(o) <= 105.0, (c, o)
