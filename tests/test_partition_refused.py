"""A ranged call whose partition the device refuses: nothing of the partition
may be used.  The refusal here is that of a machine without a visible GPU (the
opt-in to shared memory and every launch return an error, on the host), for a
map put together by hand with an allocator of host memory."""
import os
import shutil
import subprocess

import pytest


SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include "ash_internal.h"
static int allocs = 0, frees = 0;
static void* take(size_t bytes, int, ash_stream, void*) { ++allocs; return std::malloc(bytes); }
static void give(void* p, int, ash_stream, void*) { ++frees; std::free(p); }
template <int D>
void check(ash::DimKernels k) {
  ash_map m;
  m.key_dim = D;
  m.device = 0;
  m.K = k;
  m.alloc.alloc = take;
  m.alloc.free = give;
  ash_default_tuning(&m.tuning);
  for (int again = 0; again < 2; ++again) {  // a refusal must not be remembered as a success
    ash::host::PartBufs pb;
    const bool done = ash::host::partition_call(&m, nullptr, 10000, again ? 8 : 3, nullptr, &pb);
    if (done || pb.mem || allocs != frees || allocs == 0) {
      std::printf("%d dimensions, call %d: done %d, %d allocations, %d freed\n", D, again, done, allocs, frees);
      std::exit(1);
    }
  }
}
int main() {
  check<1>(ash::dim_kernels_1());
  check<4>(ash::dim_kernels_4());
  check<5>(ash::dim_kernels_5());
  check<8>(ash::dim_kernels_8());
  std::puts("ok");
}
"""


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="nvcc not available")
def test_refused_partition_is_not_used(tmp_path):
    from paper_2110_00511_gb300 import build
    lib = build.build()
    src, exe = tmp_path / "p.cu", tmp_path / "p"
    src.write_text(SOURCE)
    subprocess.run(["nvcc", *build.ARCH, *build.FLAGS, "-o", str(exe), str(src), lib,
                    "-Xlinker", "-rpath," + os.path.dirname(lib)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, env={**os.environ, "CUDA_VISIBLE_DEVICES": ""})
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
