"""A batch whose launches are refused: the maps no longer count on invariants
that the part that did run may have broken.  The refusal is that of a machine
without a visible GPU, for maps put together by hand."""
import os
import shutil
import subprocess

import pytest

SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include "ash_batch.cu"
static void* take(size_t bytes, int, ash_stream, void*) { return std::malloc(bytes); }
static void give(void* p, int, ash_stream, void*) { std::free(p); }
static ash_map* map() {
  ash_map* m = new ash_map();
  m->device = 0;
  m->key_dim = 3;
  m->S = 4;
  m->capacity = 1000;
  m->n_slots = 2000;
  m->n_buckets = 500;
  ash_default_tuning(&m->tuning);
  return m;
}
int main() {
  ash_batch b;
  b.grid = 8;
  b.alloc.alloc = take;
  b.alloc.free = give;
  for (auto& s : b.slot) s.h = static_cast<ash::BatchTable*>(std::calloc(1, sizeof(ash::BatchTable)));
  ash_map *filled = map(), *emptied = map(), *searched = map();
  int32_t key[3] = {0, 0, 0}, idx[1];
  uint8_t mask[1];
  ash_batch_op ops[3] = {};
  const int32_t kinds[3] = {ASH_OP_ACTIVATE, ASH_OP_ERASE, ASH_OP_FIND};
  ash_map* maps[3] = {filled, emptied, searched};
  for (int i = 0; i < 3; ++i) {
    ops[i].map = maps[i];
    ops[i].op = kinds[i];
    ops[i].keys = key;
    ops[i].n = 1;
    ops[i].buf_indices = idx;
    ops[i].masks = mask;
  }
  const ash_status s = ash_batch_run(&b, ops, 3, nullptr);
  const bool right = s != ASH_OK && !filled->pref_placed && !emptied->heap_identity && searched->pref_placed &&
                     searched->heap_identity && filled->heap_identity;
  std::printf("%s: status %d, %d %d %d %d\n", right ? "ok" : "wrong", s, filled->pref_placed, emptied->heap_identity,
              searched->pref_placed, searched->heap_identity);
  return right ? 0 : 1;
}
"""


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="nvcc not available")
def test_refused_launch_keeps_no_invariant(tmp_path):
    from paper_2110_00511_gb300 import build
    lib = build.build()
    src, exe = tmp_path / "b.cu", tmp_path / "b"
    src.write_text(SOURCE)
    flags = [f for f in build.FLAGS if f not in ("-O3", "-lineinfo")]
    subprocess.run(["nvcc", *build.ARCH, *flags, "-O0", "-Xptxas", "-O0", "-o", str(exe), str(src), lib,
                    "-Xlinker", "-rpath," + os.path.dirname(lib)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, env={**os.environ, "CUDA_VISIBLE_DEVICES": ""})
    assert r.returncode == 0, r.stdout + r.stderr
