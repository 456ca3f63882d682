"""The ray caster's division by the voxel size (rounded reciprocal, remainder,
correction) at the quotients where its rounding is in doubt.  For 24-bit
mantissas a and b the value before the last rounding is off by less than
2.5 ulp(q) / b, so only a quotient that close to a midpoint m / 2^s of two
floats (m odd, 25 bits) could round the other way: |a 2^s - b m| <= 5.  Those are
found through the inverse of b modulo 2^s, for every b, and compared with IEEE
division on the CPU with the same float32 operations."""
import subprocess

SOURCE = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
// inverse of an odd b modulo 2^64 (Newton; each step doubles the correct bits)
static uint64_t inverse(uint64_t b) { uint64_t x = b; for (int i = 0; i < 6; ++i) x *= 2 - b * x; return x; }
int main() {
  long bad = 0, checked = 0;
  for (uint32_t bi = 1u << 23; bi < 1u << 24; ++bi) {
    const float b = static_cast<float>(bi), y = 1.0f / b;
    const int z = __builtin_ctz(bi);
    const uint64_t inv = inverse(bi >> z);
    for (int s = 24; s <= 25; ++s) {  // quotients in [1, 2), and in (1/2, 1)
      const uint64_t step = uint64_t{1} << (s - z);
      for (int c = -5; c <= 5; ++c) {  // a 2^s = b m + c
        if (c & ((1 << z) - 1)) continue;
        const uint64_t first = (static_cast<uint64_t>(static_cast<int64_t>(-c) >> z) * inv) & (step - 1);
        for (uint64_t m = first; m < uint64_t{1} << 25; m += step) {
          if (m < uint64_t{1} << 24) continue;
          const uint64_t a2s = static_cast<uint64_t>(bi) * m + static_cast<int64_t>(c);
          const uint64_t ai = a2s >> s;
          if ((ai << s) != a2s || ai < 1u << 23 || ai >= 1u << 24) continue;
          const float a = static_cast<float>(ai), q = a * y;
          bad += fmaf(fmaf(-q, b, a), y, q) != a / b;
          ++checked;
        }
      }
    }
  }
  std::printf("%ld of %ld\n", bad, checked);
  return bad != 0;
}
"""


def test_quotients_next_to_midpoints(tmp_path):
    src, exe = tmp_path / "d.cpp", tmp_path / "d"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout.split()[2]) > 10_000_000
