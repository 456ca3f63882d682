"""Each kernel's resident blocks are its own: two kernels of one signature, one
of which fits fewer blocks on an SM, asked for in either order."""
import os
import shutil
import subprocess

import pytest

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(shutil.which("nvcc") is None, reason="nvcc not available")]

SOURCE = r"""
#include <cstdio>
#include "ash_kernels.cuh"
// 256 threads and KB of static shared memory
template <int KB>
__global__ void __launch_bounds__(256) probe_kernel(int* out) {
  __shared__ int s[KB * 256];
  s[threadIdx.x] = out[threadIdx.x];
  __syncthreads();
  out[threadIdx.x] = s[255 - threadIdx.x];
}
template <int KB>
bool right(int block) {
  int api = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&api, probe_kernel<KB>, block, 0) != cudaSuccess) return false;
  const int got = ash::resident_blocks<probe_kernel<KB>>(block);
  std::printf("%d KB, %d threads: %d, occupancy API %d\n", KB, block, got, api);
  return got == api;
}
int main(int argc, char**) {
  bool ok = true;
  for (int again = 0; again < 2; ++again)
    for (int block : {256, 128})
      ok = (argc > 1 ? right<40>(block) && right<1>(block) : right<1>(block) && right<40>(block)) && ok;
  ash::Launch L;
  L.block = 256;
  L.sms = 2;
  const int held = 2 * ash::resident_blocks<probe_kernel<40>>(256);
  ok = ok && ash::resident_grid<probe_kernel<40>>(1000, L) == held && ash::resident_grid<probe_kernel<40>>(1, L) == 1;
  L.one_wave = false;
  ok = ok && ash::resident_grid<probe_kernel<40>>(1000, L) == 1000;
  return ok ? 0 : 1;
}
"""


@pytest.mark.parametrize("args", [[], ["reversed"]])
def test_each_kernel_has_its_own(tmp_path, args):
    from paper_2110_00511_gb300 import build
    lib = build.build()
    src, exe = tmp_path / "r.cu", tmp_path / "r"
    src.write_text(SOURCE)
    subprocess.run(["nvcc", *build.ARCH, *build.FLAGS, "-o", str(exe), str(src), lib,
                    "-Xlinker", "-rpath," + os.path.dirname(lib)], check=True)
    r = subprocess.run([str(exe), *args], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
