"""The size rules of the coset-arithmetic product (csrc/pair_rules.h), compiled for the host."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1804_05028_gb300", "csrc")


def run(tmp_path, body):
    """What a program made of the rules and `body` prints."""
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text('#include "pair_rules.h"\n#include <cstdio>\n#include <initializer_list>\nusing namespace pair_rules;\n' + body)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout


# the last step of expand_kernel's loop: every thread's first position at or past the end, in the
# 32 bits the kernel counts in
LAST_STEP = """
static bool ends(uint64_t slots, uint32_t sms) {
  const uint32_t n = (uint32_t)slots, stride = expand_blocks(slots, sms) * kExpandThreads;
  for (uint32_t t = 0; t < stride && t < n; t++) {
    const uint32_t last = t + (n - 1 - t) / stride * stride;
    if ((uint32_t)(last + stride) < n) return false;   // wrapped to the front
  }
  return true;
}
"""


@pytest.mark.parametrize("sms", [1, 132, 152, 4096, 100000])
def test_expansion_ends(tmp_path, sms):
    out = run(tmp_path, LAST_STEP + """
int main() {
  const uint64_t n[] = {1, 255, 256, 257, 1u << 22, kMaxSlots - 1, kMaxSlots};
  for (uint64_t v : n) printf("%%d", ends(v, %d));
}
""" % sms)
    assert out == "1111111"


def test_row_enumeration_ends(tmp_path):
    """enum_rows' warps look at 1024 slots from any start inside a class."""
    out = run(tmp_path, """
int main() {
  const uint32_t end = (uint32_t)kMaxSlots;
  for (uint32_t p0 = end - 1024; p0 < end; p0++)
    for (uint32_t q = 0; q < 1024; q++)
      if ((uint32_t)(p0 + q) < p0) { printf("wraps"); return 0; }
  printf("ends");
}
""")
    assert out == "ends"


def test_emulation_sees_the_wrap(tmp_path):
    """Slots within one stride of 2^32 are what the bound keeps out."""
    out = run(tmp_path, LAST_STEP + 'int main() { printf("%d", ends(0xFFFFFF00ull, 152)); }')
    assert out == "0"


def test_routes(tmp_path):
    """Which way a product goes: s(earch), d(irect) or e(xpanded)."""
    out = run(tmp_path, """
static void q(int64_t rows, int64_t dim, double terms, uint64_t slots, bool c128 = false, bool tab = false) {
  putchar("sde"[route(rows, dim, terms, slots, c128, tab)]);
}
int main() {
  q(15, 15, 5, 20); q(15, 1 << 20, 10, 1 << 20);                         // less than half a warp
  q(16, 16, 5, 20); q(810, 810, 8.5, 1100); q(810, 810, 8.5, 1100, true);   // small sectors
  q(810, 810, 8.5, 1100, false, true); q(153, 153, 17, 300, false, true);   // one block, complex fp32
  q(168, 168, 6.6, 300, true); q(66, 66, 13, 130, true); q(300, 300, 6, 600, true);   // complex fp64
  q(153, 153, 17, 300); q(16384, 16384, 10, 16385);
  q(250000, 10000000, 10, 10000000); q(250001, 10000000, 10, 10000000);      // a term per four slots
  const int64_t big = 1ll << 27;
  q(16, big, 40, big); q(16, big + 8, 40, big); q(big / 8, big + 8, 40, big); q(big / 8 + 1, big + 8, 40, big);
}
""")
    assert out == "ss" + "dde" + "se" + "dee" + "ee" + "de" + "dsse"


def test_memory(tmp_path):
    """A plan only beside the vectors of a Lanczos run; the pool's bound."""
    out = run(tmp_path, """
int main() {
  const uint64_t D = 861602748, n = 920000000, GB = 1000000000;
  for (uint64_t f : {264 * GB, 48 * GB, 41 * GB, 38 * GB}) printf("%d%d ", fits(f, D, n, true).pair, fits(f, D, n, true).rows);
  const uint64_t E = 4200000000ull;      // 284 GB less 95 GB of basis and index
  printf("%d %d%d ", fits(189 * GB, E, E, true).pair, always_fits(1000, 2000), always_fits(D, n));
  printf("%d", pool_keep(n, true) <= 16 * n + (17u << 20) && pool_keep(n, false) <= 32 * n + (17u << 20));
}
""")
    assert out == "11 10 10 00 0 10 1"
