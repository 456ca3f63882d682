"""Registers of kernels that keep many loads in flight, as the compiler prints
them: no more than let as many blocks reside as the kernels were measured with.
Key dimensions and bucket sizes away from the default are where a change goes
unseen."""
import os
import re
import shutil
import subprocess

import pytest

# kernel: most registers
LIMITS = {
    # finds: several keys per thread and wide buckets
    "find_kernel<3, 4, 1>": 32, "find_kernel<3, 8, 1>": 40, "find_kernel<3, 16, 1>": 64,
    "find_kernel<3, 4, 2>": 64, "find_kernel<3, 8, 2>": 64, "find_kernel<3, 16, 2>": 64,
    "find_kernel<3, 4, 4>": 80, "find_kernel<3, 8, 4>": 100, "find_kernel<3, 16, 4>": 80,
    "find_kernel<8, 4, 1>": 64, "find_kernel<8, 16, 2>": 96, "find_kernel<8, 16, 4>": 128,
    # preferred-slot claims: six blocks for 4 slots and up to four dimensions, elsewhere as many as fit
    "claim_pref_kernel<3, 4, 1>": 40, "claim_pref_kernel<4, 4, 1>": 40, "claim_pref_kernel<3, 8, 1>": 48,
    "claim_pref_kernel<3, 16, 1>": 64, "claim_pref_kernel<5, 4, 1>": 40, "claim_pref_kernel<8, 4, 1>": 48,
    "claim_pref_kernel<8, 8, 1>": 64,
    # commits: eight blocks
    "commit_kernel<3, 1, false, int const*, true>": 32, "commit_kernel<3, 2, false, int const*, true>": 32,
    "commit_kernel<8, 1, false, int const*, true>": 32, "commit_kernel<8, 2, false, int const*, true>": 32,
}


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="nvcc not available")
def test_registers(tmp_path):
    from paper_2110_00511_gb300 import build
    src = tmp_path / "r.cu"
    names = [f"(void*)ash::{k}" for k in LIMITS]
    src.write_text('#include "ash_kernels.cuh"\nvoid* kernels[] = {\n' + ",\n".join(names) + "};\n")
    r = subprocess.run(["nvcc", *build.ARCH, *build.FLAGS, "-Xptxas", "-v", "-c", "-o", os.devnull, str(src)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    text = subprocess.run(["c++filt"], input=r.stderr, capture_output=True, text=True, check=True).stdout
    used = {m[1].replace(", int const*", ""): int(m[2]) for m in
            re.finditer(r"entry function 'void ash::(\w+<.*?>)\(.*?Used (\d+) registers", text, re.S)}
    limits = {k.replace(", int const*", ""): most for k, most in LIMITS.items()}
    assert used.keys() >= limits.keys()
    over = {k: (used[k], most) for k, most in limits.items() if used[k] > most}
    assert not over, f"(used, most): {over}"
