"""The ray caster's three-instruction division by the voxel size (Markstein:
a rounded reciprocal, one remainder, one correction) against IEEE division:
floor(x / b + 1/2) for random and edge values of x over the voxel sizes that
take it, on the CPU with the same float32 operations (fmaf)."""
import subprocess

SOURCE = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
static uint64_t s = 88172645463325252ull;
static uint32_t rnd() { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return (uint32_t)(s >> 16); }
static float bits(uint32_t u) { float f; std::memcpy(&f, &u, 4); return f; }
// a sample's coordinate: in range (between -1e9 and 1e9) or not
static bool cell(float q, float* out) { float g = std::floor(q + 0.5f); *out = g; return g > -1.0e9f && g < 1.0e9f; }
int main() {
  long bad = 0, checked = 0;
  const float sizes[] = {0.006f, 0.008f, 0.01f, 0.05f, 1.0f, 0.1f, 1.0f / 3, 3.0f, 0x1p-60f, 0x1p60f, 0x1.fffffep-8f, 0x1.fffffep-60f, 0x1.000002p3f};
  for (int k = 0; k < 413; ++k) {
    float b = k < 13 ? sizes[k] : bits(((67 + rnd() % 121) << 23) | (rnd() & 0x7FFFFF));  // 2^-60 .. 2^60
    if (!(b >= 0x1p-60f && b <= 0x1p60f)) continue;
    const float y = 1.0f / b;
    for (int j = 0; j < 20000; ++j) {
      float x;
      if (j % 4 == 0) x = bits(rnd());                                            // any bit pattern
      else if (j % 4 == 1) x = (float)((int)(rnd() % 4001) - 2000) * b;           // near lattice points
      else if (j % 4 == 2) x = ((float)((int)(rnd() % 4001) - 2000) + 0.5f) * b;  // near cell faces
      else x = ((float)rnd() / 4294967296.0f - 0.5f) * 4096.0f * b;
      const float q = x * y;
      const float z = fmaf(fmaf(-q, b, x), y, q);
      float g0, g1;
      const bool in0 = cell(x / b, &g0), in1 = cell(z, &g1);
      bad += in0 != in1 || (in0 && g0 != g1);
      ++checked;
    }
  }
  std::printf("%ld of %ld\n", bad, checked);
  return bad != 0;
}
"""


def test_division_by_the_voxel_size(tmp_path):
    src, exe = tmp_path / "d.cpp", tmp_path / "d"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout.split()[2]) > 7_000_000
